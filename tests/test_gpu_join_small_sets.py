"""The join's 64-row tile at the edges of its candidate sets.

List lengths around a quarter, a half and the whole of the 64 candidates it takes (and one past them, the 128-row
tile's): refinement passes must keep the lists of the FP32 tile bit for bit with every operand.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("operand", ["f16", "bf16", "fp8"])
@pytest.mark.parametrize("metric", ["l2", "ip", "cos"])
@pytest.mark.parametrize("k,d", [(1, 4), (3, 36), (15, 36), (16, 128), (17, 20), (31, 36), (32, 132), (33, 36), (63, 12), (65, 36)])
def test_small_sets_keep_the_fp32_lists(k, d, metric, operand):
    import paper_2603_21710_gb300 as fg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(100 * k + d)
    n, half = 900, 500
    X = rng.standard_normal((12, d))[rng.integers(0, 12, n)] + 0.5 * rng.standard_normal((n, d))
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    if operand == "bf16":
        X = X.to(torch.bfloat16).float()
    graphs = [fg.build_pg(x, M=10, ef=24, metric=metric) for x in (X[:half], X[half:])]
    inp = fg.MergeInput([X[:half], X[half:]], [a for a, _ in graphs], [e for _, e in graphs], metric=metric)
    lists = {q: t for q, t in fg.cross_query(inp, k).items() if q != "stats"}
    for _ in range(2):
        got = {}
        for f in ("fp32", "fp8" if operand == "fp8" else "tc"):
            got[f] = {q: t.clone() for q, t in lists.items()}
            st = fg.refine_pass(inp, got[f], join_filter=f)
            assert f == "fp32" or st["join_class"][3] == 0, st["join_class"]
        ref, new = got.values()
        for q in ("ids", "dist", "flags"):
            assert torch.equal(new[q], ref[q]), q
        lists = ref
