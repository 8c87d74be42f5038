"""Kernels that serve two arrays by blockIdx.y keep their parameters out of local memory."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["rev_select", "scan"])
def test_no_local_memory(kernel):
    import paper_2603_21710_gb300 as fg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.zeros(1, device="cuda:0")
    fg.load()
    assert fg._lib.test_get(f"{kernel}_local_bytes") == 0
