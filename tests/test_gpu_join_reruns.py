"""Update's re-runs when every vertex overflows the proposal buffer again.

Random lists propose far more than the smallest buffer holds, run after run, and the vertices joined at once fill it together:
the number of vertices left over stays the same for several runs although each merges a full buffer. The pass must
go on until all have fitted and keep the lists of a pass with room for everything.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _lists(X, k, rng):
    """k random neighbours of every vertex, sorted, with their exact squared distances (integer coordinates)."""
    N = len(X)
    ids = np.empty((N, k), np.int32)
    dist = np.empty((N, k), np.float32)
    for u in range(N):
        v = rng.permutation(N - 1)[:k]
        v[v >= u] += 1
        dv = ((X[v] - X[u]) ** 2).sum(1)
        o = np.lexsort((v, dv))
        ids[u], dist[u] = v[o], dv[o]
    return ids, dist


# the join's forms: byte rows, BF16 and FP16 operands, FP32 tile
@pytest.mark.parametrize("join_filter,lo,hi,d", [("tc", 0, 256, 16), ("tc", -9, 10, 32), ("tc", -600, 601, 4), ("fp32", -9, 10, 8)])
def test_a_pass_goes_on_while_all_vertices_overflow(join_filter, lo, hi, d):
    import paper_2603_21710_gb300 as fg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(d)
    N, k = 4000, 32
    X = rng.integers(lo, hi, (N, d)).astype(np.float32)
    ids, dist = _lists(X, k, rng)
    adj = torch.full((N, 1), -1, dtype=torch.int32, device=dev)
    inp = fg.MergeInput.from_flat(torch.from_numpy(X).to(dev), [N // 2, N - N // 2], adj, [0, 0])

    def run():
        g = {"ids": torch.from_numpy(ids).to(dev), "dist": torch.from_numpy(dist).to(dev),
             "flags": torch.ones((N, k), dtype=torch.uint8, device=dev)}
        return g, fg.refine_pass(inp, g, join_filter=join_filter)

    fg.load()
    try:
        fg._lib.test_set("prop_cap", 1 << 24)   # room for every proposal
        want, st = run()
        assert st["join_reruns"] == 0
        fg._lib.test_set("prop_cap", 1)         # raised to what one vertex can propose
        got, st = run()
    finally:
        fg._lib.test_set("prop_cap", 0)
    assert st["join_reruns"] >= 2
    for q in ("ids", "dist", "flags"):
        assert torch.equal(got[q], want[q]), q
