"""Waits that run out on the GPU, reported without a fault: the bounded waits
of the tensor-core kernels on barriers that nothing arrives at."""
import pytest

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
