"""The panelled Cholesky factor and inverse at the edges of its panels (16
columns), tiles (16 x 8) and CTA item groups, against the FP64 oracle.

The MVDR denominators ||L^-1 a||^2 see every entry of L^-1.  On FP32
operators their tolerance is the operators' 1e-5 (relative L2)."""
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


def _mvdr_error(mv, job):
    A = O.steering_matrix(job.ant_xyz, job.l, job.m, job.lam)
    ref = 1.0 / O.mvdr_h(A, job.R)
    return float(np.linalg.norm(mv - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("p", [2, 3, 15, 16, 17, 24, 31, 32, 33, 64, 65, 129, 255, 384])
def test_inverse_factor_at_panel_edges(G, p):
    job = synth.custom(700 + p, p, 11, 9, 3, 8 * p + 50, radius=6.0)
    im = G.Imager.from_job(job)
    assert _mvdr_error(im.mvdr_bound(), job) <= 1e-5
    im.close()


def test_batch_of_unequal_sizes(G):
    """One launch sized for the largest job leaves the smaller ones right."""
    jobs = [synth.custom(720 + p, p, 9, 7, 2, 8 * p + 50, radius=6.0) for p in (50, 2, 17, 64, 16, 33)]
    ims = [G.Imager.from_job(j) for j in jobs]
    G.prepare_batch(ims)
    for im, job in zip(ims, jobs):
        assert _mvdr_error(im.mvdr_bound(), job) <= 1e-5
        im.close()


@pytest.mark.parametrize("p,k", [(2, 1), (16, 15), (17, 16), (40, 15), (40, 16), (40, 39), (100, 47)])
def test_bad_pivot_is_reported(G, p, k):
    """A negative pivot in column k: the call fails, and the context takes the next covariance."""
    job = synth.custom(740 + p, p, 5, 4, 1, 8 * p + 50, radius=4.0)
    im = G.Imager.from_job(job)
    R = np.eye(p, dtype=np.complex128)
    R[k, 0] = R[0, k] = 1.5
    im.set_covariance(R, job.N)
    with pytest.raises(G.ImgError) as e:
        im.mvdr_bound()
    assert e.value.code == G.IMG_ENOTPD
    im.set_covariance(job.R, job.N)
    assert _mvdr_error(im.mvdr_bound(), job) <= 1e-5
    im.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("p", [2, 5, 8])
def test_small_jobs_take_the_same_bits_from_either_form(G, p, prec):
    """Alone, a small job is factored by one CTA; in a batch with a larger job
    it goes through the panels and the larger job's pixel grid."""
    small = synth.custom(760 + p, p, 13, 17, 2, 8 * p + 50, radius=4.0)
    large = synth.custom(770, 40, 33, 20, 2, 400, radius=4.0)
    a = G.Imager.from_job(small, precision=prec)
    b, c = G.Imager.from_job(small, precision=prec), G.Imager.from_job(large, precision=prec)
    G.prepare_batch([b, c])
    np.testing.assert_array_equal(a.dirty(), b.dirty())
    np.testing.assert_array_equal(a.mvdr_bound(), b.mvdr_bound())
    np.testing.assert_array_equal(a.solve()[0], b.solve()[0])
    for im in (a, b, c):
        im.close()


@pytest.mark.parametrize("p", [16, 45, 64])
def test_server_factor_takes_the_same_bits(G, p):
    """The server's fused kernel factors in one CTA, img_solve over panels."""
    job = synth.custom(780 + p, p, 18, 15, 3, 8 * p + 50, radius=6.0)
    im = G.Imager.from_job(job, precision=1, kappa=3.0)
    alone, _ = im.solve()
    im.close()
    srv = G.Server()
    image, _, _ = srv.wait(srv.submit_job(job, precision=1, kappa=3.0))
    srv.close()
    np.testing.assert_array_equal(alone, image)
