"""The one-CTA tensor-core solver where its LSQR changes form: free sets that
grow past one, two, three and four 128-pixel tiles (f = 128, 256, 384, 512),
with Kp = 32 and 64, odd p, both costs.  The oracle replays the decisions
(ties within 1e-6 of scale); the image is held to max(1e-4, 8 cond(M_F) 2^-24),
the attainable accuracy of FP32 LSQR vectors."""
import numpy as np
import pytest

import synth
from oracle import imager as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import paper_1505_01348_gb300 as G
    G.load(build_if_missing=True)
    return G


# (seed, p, n_l, n_m, sources, N, radius, cost, kappa, free pixels reached at least)
CASES = [
    (901, 30, 26, 18, 6, 8000, 18.0, O.COST_PWLS, 0.3, 256),
    (902, 48, 26, 22, 8, 20000, 30.0, O.COST_PWLS, 0.5, 512),
    (903, 45, 25, 24, 8, 20000, 30.0, O.COST_LS, 0.5, 512),
    (904, 64, 30, 25, 8, 30000, 30.0, O.COST_PWLS, 0.3, 512),
]


@pytest.mark.parametrize("case", CASES, ids=[f"p{c[1]}_{'pwls' if c[7] else 'ls'}" for c in CASES])
def test_growing_free_set_follows_the_oracle(G, case):
    seed, p, nl, nm, nsrc, N, rad, cost, kappa, reach = case
    job = synth.custom(seed, p, nl, nm, nsrc, N, radius=rad, snr_db=0.0)
    prm = O.Params(cost=cost, kappa=kappa, eps_floor=1e-6, feas_tol=1e-5, lsqr_atol=1e-6, lsqr_btol=1e-6)
    im = G.Imager.from_job(job, cost=cost, kappa=kappa, eps_floor=1e-6, feas_tol=1e-5, precision=G.PREC_F16X3)
    sigma, info = im.solve()
    log = [(k, q) for k, q, _ in im.events()]
    sets = im.sets()
    im.close()
    assert info.converged == 1
    f = np.cumsum([1 if k == 0 else -1 for k, _ in log])
    assert f.max() > reach
    A = O.steering_matrix(job.ant_xyz, job.l, job.m, job.lam)
    bnd = O.bounds(A, None, job.R, job.N, prm)
    prob = O.cost_problem(A, None, job.R, bnd, cost)
    rep = O.active_set_follow(prob, bnd.eps, prm, log, tol=1e-6)
    assert not rep.violations, (rep.violations[:3], rep.max_margin)
    np.testing.assert_array_equal(sets, rep.result.sets)
    # M_F^H M_F of the columns s_j vect(c_j c_j^H): s_i s_j |c_i^H c_j|^2
    F = np.nonzero(sets == O.SET_F)[0]
    C = A[:, F] if cost == O.COST_LS else np.linalg.solve(O.cholesky_lower(job.R), A[:, F])
    s = np.ones(F.size) if cost == O.COST_LS else np.sum(np.abs(C) ** 2, axis=0) ** -2.0
    gram = np.abs(C.conj().T @ C) ** 2 * np.outer(s, s)
    cond = np.sqrt(np.linalg.cond(gram))
    err = np.linalg.norm(sigma - rep.result.sigma) / np.linalg.norm(rep.result.sigma)
    assert err <= max(1e-4, 8.0 * cond * 2.0 ** -24)


def test_clusters_of_ctas_do_not_change_the_image(G):
    """One job (a cluster shares its gradients) and many jobs at once (one CTA each)."""
    job = synth.custom(910, 40, 33, 21, 5, 2000, radius=20.0)
    for prec in (G.PREC_FP32, G.PREC_F16X3):
        ims = [G.Imager.from_job(job, kappa=3.0, max_outer=60, precision=prec) for _ in range(60)]
        one, _ = ims[0].solve()
        outs, _ = G.solve_batch(ims)
        for o in outs:
            np.testing.assert_array_equal(o, one)
        few, _ = G.solve_batch(ims[:9])
        for o in few:
            np.testing.assert_array_equal(o, one)
        for im in ims:
            im.close()


def test_growing_free_set_in_bf16x3(G):
    """The split tiles streamed from global memory with BF16 parts (three and
    four tiles).  Products keep about 16 bits: decisions are admitted within the
    operators' tolerance (1e-4 of scale), the image is held to
    max(1e-3, 8 cond(M_F) 2^-16)."""
    job = synth.custom(905, 48, 26, 22, 8, 20000, radius=30.0, snr_db=0.0)
    prm = O.Params(cost=O.COST_LS, kappa=0.5, eps_floor=1e-6, feas_tol=1e-4, lsqr_atol=1e-6, lsqr_btol=1e-6)
    im = G.Imager.from_job(job, cost=O.COST_LS, kappa=0.5, eps_floor=1e-6, feas_tol=1e-4, precision=G.PREC_BF16X3)
    sigma, info = im.solve()
    log = [(k, q) for k, q, _ in im.events()]
    sets = im.sets()
    im.close()
    assert info.converged == 1
    assert np.cumsum([1 if k == 0 else -1 for k, _ in log]).max() > 384
    A = O.steering_matrix(job.ant_xyz, job.l, job.m, job.lam)
    bnd = O.bounds(A, None, job.R, job.N, prm)
    rep = O.active_set_follow(O.cost_problem(A, None, job.R, bnd, O.COST_LS), bnd.eps, prm, log, tol=1e-4)
    assert not rep.violations, (rep.violations[:3], rep.max_margin)
    np.testing.assert_array_equal(sets, rep.result.sets)
    F = np.nonzero(sets == O.SET_F)[0]
    cond = np.sqrt(np.linalg.cond(np.abs(A[:, F].conj().T @ A[:, F]) ** 2))
    err = np.linalg.norm(sigma - rep.result.sigma) / np.linalg.norm(rep.result.sigma)
    assert err <= max(1e-3, 8.0 * cond * 2.0 ** -16)
