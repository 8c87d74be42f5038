"""The join's tensor-core operands over dimensions, magnitudes and metrics.

Rows are padded to whole MMA steps, FP32 rows become FP16 under a power-of-two factor per row, and an
E4M3 tile that is too coarse for the lists gives way to them: a refinement pass must keep the lists of the
FP32 tile bit for bit whatever the operand.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _data(kind, n, d, rng):
    X = rng.standard_normal((20, d))[rng.integers(0, 20, n)] + 0.3 * rng.standard_normal((n, d))
    if kind == "tiny":
        X *= 1e-9
    elif kind == "huge":
        X *= 1e8
    elif kind == "rows":      # magnitudes differ by row, some rows are zero, some coordinates far below the rest
        X *= np.exp2(rng.integers(-20, 20, (n, 1)))
        X[:, 0] *= 1e-7
        X[::97] = 0.0
    elif kind == "bf16":      # BF16 values: the BF16 operand is exact
        X = torch.from_numpy(X).to(torch.bfloat16).double().numpy()
    return X.astype(np.float32)


def _pass(inp, kn, join_filter):
    import paper_2603_21710_gb300 as fg
    g = {k: v.clone() for k, v in kn.items()}
    st = fg.refine_pass(inp, g, join_filter=join_filter)
    return g, st


@pytest.mark.parametrize("metric", ["l2", "ip", "cos"])
@pytest.mark.parametrize("d,kind", [(4, "plain"), (12, "rows"), (20, "tiny"), (36, "huge"), (96, "plain"), (100, "rows"),
                                    (128, "plain"), (128, "bf16"), (132, "rows"), (260, "plain"), (404, "huge")])
def test_operands_keep_the_fp32_lists(d, kind, metric):
    import paper_2603_21710_gb300 as fg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(d)
    n, k = 1500, 24
    X = torch.from_numpy(_data(kind, n, d, rng)).to(dev)
    sizes = [700, 500, 300]
    adj, ent, o = [], [], 0
    for s in sizes:
        a, e = fg.build_pg(X[o:o + s], M=12, ef=32, metric=metric)
        adj.append(a)
        ent.append(e)
        o += s
    inp = fg.MergeInput([X[:700], X[700:1200], X[1200:]], adj, ent, metric=metric)
    kn = {q: t for q, t in fg.cross_query(inp, k).items() if q != "stats"}
    ref, st = _pass(inp, kn, "fp32")
    assert st["join_class"][3] > 0
    for f in ("tc", "fp8"):
        got, st = _pass(inp, kn, f)
        assert st["join_class"][3] == 0 and sum(st["join_class"][:3]) > 0, st["join_class"]
        for q in ("ids", "dist", "flags"):
            assert torch.equal(got[q], ref[q]), (f, q)
