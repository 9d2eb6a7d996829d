"""The server's pooled contexts and the jobs' arithmetic: a job gets the image
it gets alone whatever arithmetic the context's last job of the shape had."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import paper_1505_01348_gb300 as G
    G.load(build_if_missing=True)
    return G


@pytest.mark.parametrize("p,n", [(96, 16), (40, 18)])
def test_arithmetics_in_turn_on_one_shape(G, p, n):
    job = synth.custom(990 + p, p, n, n - 1, 4, 3000, radius=10.0)
    kw = dict(kappa=3.0, max_outer=40)
    alone = {}
    for prec in (G.PREC_F16X3, G.PREC_BF16X3, G.PREC_FP32):
        im = G.Imager.from_job(job, precision=prec, **kw)
        alone[prec] = im.solve()[0]
        im.close()
    assert not np.array_equal(alone[G.PREC_F16X3], alone[G.PREC_BF16X3])
    srv = G.Server()
    for prec in (G.PREC_BF16X3, G.PREC_F16X3, G.PREC_FP32, G.PREC_BF16X3, G.PREC_F16X3):
        image, _, _ = srv.wait(srv.submit_job(job, precision=prec, **kw))
        np.testing.assert_array_equal(image, alone[prec])
    srv.close()
