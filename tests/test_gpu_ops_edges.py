"""The forward Psi at the sizes where its stages have few tasks or its blocks
are ragged, and its outputs' alignment, against plain FP64 products.

Tolerances: the operators' (1e-5 relative; BF16x3 1e-4)."""
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


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# Kp = 32 and 64 (4 tasks a stage), 96 (6 and 8), 128, 160, 256, 352 (short last block)
@pytest.mark.parametrize("p", [2, 32, 33, 64, 65, 96, 97, 160, 225, 353])
@pytest.mark.parametrize("grid", [(9, 70), (70, 9), (33, 40)])
def test_forward_at_task_counts(G, p, grid):
    job = synth.custom(800 + p, p, grid[0], grid[1], 2, 2 * p + 50, radius=6.0)
    A = O.steering_matrix(job.ant_xyz, job.l, job.m, job.lam)
    x = np.random.default_rng(p).random(job.Q)
    ref = (A * x) @ A.conj().T
    for prec, tol in ((G.PREC_F16X3, 1e-5), (G.PREC_BF16X3, 1e-4)):
        im = G.Imager.from_job(job, precision=prec)
        assert _rel(im.psi(x), ref) <= tol
        # a call's scale does not outlive it
        assert _rel(im.psi(1e-6 * x), 1e-6 * ref) <= tol
        im.close()


def test_forward_into_an_8_byte_aligned_matrix(G):
    torch = pytest.importorskip("torch")
    p = 45
    job = synth.custom(850, p, 20, 30, 2, 500, radius=6.0)
    im = G.Imager.from_job(job, precision=G.PREC_F16X3)
    x = torch.rand(job.Q, dtype=torch.float64, device="cuda")
    buf = torch.zeros(2 * p * p + 1, dtype=torch.float64, device="cuda")
    K = torch.empty(p, p, dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    im.psi(x, K)
    im.psi(x, buf[1:])
    assert torch.equal(torch.view_as_real(K).reshape(-1), buf[1:])
    assert buf[0].item() == 0.0
    im.close()
