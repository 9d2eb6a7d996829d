"""Waits that run out on the GPU, reported without a fault: the bounded waits
of the tensor-core kernels on barriers that nothing arrives at."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import paper_1505_01348_gb300 as G
    G.load(build_if_missing=True)
    return G


# thread 32 waits for the solver's tile copies, thread 0 writes the status
@pytest.mark.parametrize("thread", [0, 31, 32, 255])
def test_a_wait_of_one_thread_reaches_the_status(G, thread):
    from paper_1505_01348_gb300._lib import check_wait
    assert check_wait(1000, arrive=False, thread=thread) == G.IMG_ETIMEOUT
    assert check_wait(1000, arrive=True, thread=thread) == G.IMG_OK


# one context per place that waits: CUDA-core, one-CTA, streamed and work-item operators
@pytest.mark.parametrize("p,prec", [(20, 0), (40, 1), (72, 2), (288, 1)])
def test_the_next_call_that_waits_reports_an_operators_late_wait(G, p, prec):
    job = synth.custom(31, p, 12, 10, 2, 2 * p + 60, radius=5.0)
    im = G.Imager.from_job(job, precision=prec, max_outer=20)
    x = np.random.default_rng(p).random(job.Q)
    K, U = im.psi(x), np.eye(p, dtype=np.complex128)
    calls = {"psi": lambda: im.psi(x), "psi_adj": lambda: im.psi_adj(U), "dirty": im.dirty,
             "solve": lambda: im.solve(), "ls_image": lambda: im.ls_image(maxit=5),
             "prepare_batch": lambda: G.prepare_batch([im]), "solve_batch": lambda: G.solve_batch([im])}
    for name, call in calls.items():
        im.set_covariance(job.R, job.N)          # bounds and factor are recomputed
        assert im._lib.img_check_wait_ctx(im.h, 500, 1) == G.IMG_OK
        call()
        assert im._lib.img_check_wait_ctx(im.h, 500, 0) == G.IMG_OK
        with pytest.raises(G.ImgError) as e:
            call()
        assert e.value.code == G.IMG_ETIMEOUT, name
        call()                                   # reported once, and the context works on
    np.testing.assert_array_equal(im.psi(x), K)
    im.close()
