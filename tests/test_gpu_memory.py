"""Memory that the library keeps between calls can be had back."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1311_6696_gb300 import peps
    return torch, peps


def test_released_memory_is_free_again(env):
    """Once the kernels of a call are loaded, a call and a release leave the
    device's free memory where it was (to one 2 MB page of the runtime's own),
    and the call after that gives the same result."""
    torch, peps = env
    from paper_1311_6696_gb300 import synth
    A = synth.peps_gauss(4, 6, 2, 6, seed=3)

    def call():
        return peps.norm(A, 36, mode="var", precision="tf32x3")

    first = call()
    peps.release_memory()
    before = torch.cuda.mem_get_info()[0]
    assert call() == first
    assert before - torch.cuda.mem_get_info()[0] >= 32 << 20     # kept for the next call
    peps.release_memory()
    assert before - torch.cuda.mem_get_info()[0] <= 2 << 20
    assert call() == first
