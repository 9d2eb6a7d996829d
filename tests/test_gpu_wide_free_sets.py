"""LSQR of the wide solver (64 < p <= 128) on long free lists: every CTA of the
cluster form takes several forward tasks and several adjoint items per phase,
phase after phase on the same barriers, for about a thousand passes; above 512
free pixels the kernels take over.  The oracle replays the decisions (ties
within 1e-6 of scale); the image is held to max(1e-4, 8 cond(M_F) 2^-24), the
attainable accuracy of FP32 LSQR vectors."""
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


def test_cluster_lsqr_on_a_growing_list_follows_the_oracle(G):
    # 572 free pixels: five tiles, nine 64-pixel stages
    job = synth.custom(923, 66, 26, 22, 8, 30000, radius=30.0, snr_db=0.0)
    prm = O.Params(cost=O.COST_LS, kappa=0.5, eps_floor=1e-6, feas_tol=1e-5, lsqr_atol=1e-6, lsqr_btol=1e-6)
    im = G.Imager.from_job(job, cost=O.COST_LS, kappa=0.5, eps_floor=1e-6, feas_tol=1e-5, precision=G.PREC_F16X3)
    sigma, info = im.solve()
    log = [(k, q) for k, q, _ in im.events()]
    sets = im.sets()
    im.close()
    assert info.converged == 1
    assert np.cumsum([1 if k == 0 else -1 for k, _ in log]).max() > 512
    A = O.steering_matrix(job.ant_xyz, job.l, job.m, job.lam)
    bnd = O.bounds(A, None, job.R, job.N, prm)
    rep = O.active_set_follow(O.cost_problem(A, None, job.R, bnd, O.COST_LS), bnd.eps, prm, log, tol=1e-6)
    assert not rep.violations, (rep.violations[:3], rep.max_margin)
    np.testing.assert_array_equal(sets, rep.result.sets)
    F = np.nonzero(sets == O.SET_F)[0]
    cond = np.sqrt(np.linalg.cond(np.abs(A[:, F].conj().T @ A[:, F]) ** 2))
    err = np.linalg.norm(sigma - rep.result.sigma) / np.linalg.norm(rep.result.sigma)
    assert err <= max(1e-4, 8.0 * cond * 2.0 ** -24)


# one kernel per subproblem in the cluster form, six per iteration otherwise
@pytest.mark.parametrize("p,prec", [(66, 1), (128, 2)])
def test_long_lists_leave_the_cluster(G, p, prec):
    job = synth.custom(940 + p, p, 40, 40, 12, 20000, radius=60.0, snr_db=0.0)

    def run(passes):
        im = G.Imager.from_job(job, precision=prec, kappa=0.1, lsqr_maxit=20, max_outer=passes)
        _, info = im.solve()
        im.close()
        return info

    a, b, c = run(900), run(960), run(1120)
    assert a.n_free < b.n_free <= 512 < c.n_free
    per_it = lambda x, y: (y.cyc_aux[0] - x.cyc_aux[0]) / (y.lsqr_iters - x.lsqr_iters)
    assert per_it(a, b) < 3.0               # kernels of a pass over its 20 iterations
    assert per_it(b, c) > 3.0               # most of these passes have more than 512


@pytest.mark.parametrize("p,cost", [(72, O.COST_PWLS), (120, O.COST_LS)])
def test_host_loop_runs_the_same_forms(G, p, cost, monkeypatch):
    """The solve's graph and the host-driven loop give the same bits on lists
    to both sides of 512 pixels."""
    job = synth.custom(950 + p, p, 30, 30, 10, 20000, radius=50.0, snr_db=0.0)
    out = []
    for graph in ("1", "0"):
        monkeypatch.setenv("IMG_SOLVE_GRAPH", graph)
        im = G.Imager.from_job(job, precision=1, cost=cost, kappa=0.1, lsqr_maxit=20, max_outer=1200)
        out.append(im.solve())
        im.close()
    assert out[0][1].n_free > 512
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1].lsqr_iters == out[1][1].lsqr_iters
