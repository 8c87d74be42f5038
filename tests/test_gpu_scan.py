"""Prefix sums and compaction at the edges of the scan's tiles and of its two forms (above 8M entries the
tiles' sums are scanned first): the members of an HNSW layer are the ids of that level, ascending."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M,level", [(1, 2, 1), (37, 2, 1), (2047, 2, 2), (2048, 2, 2), (2049, 2, 2),
                                       (2048 * 256 + 3, 16, 3), (2048 * 4096, 16, 4), (2048 * 4096 + 2049, 16, 4)])
def test_layer_members(n, M, level):
    import paper_2603_21710_gb300 as fg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    levels, counts = fg.hnsw_levels(n, M, seed=11)
    want = torch.nonzero(levels >= level)[:, 0].to(torch.int32)
    assert counts[level] == want.numel()
    if want.numel() == 0:
        return
    X = torch.rand((n, 4), device="cuda")
    ly = fg.hnsw_layer(X, levels, level, want.numel(), M=8, ef=8)
    assert torch.equal(ly["members"], want)
