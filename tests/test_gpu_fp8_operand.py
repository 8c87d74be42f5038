"""Which operand Update's tensor-core tile reads when FP8 is asked for, and each form of the E4M3 tile.

The E4M3 tile is used where it is fine enough for the lists and gives way to the 16-bit one otherwise; the call says
which ran. With the test hook that keeps E4M3 in any case, every tile size over one and several K chunks must keep the
lists of the FP32 tile bit for bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def hooks():
    import paper_2603_21710_gb300 as fg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fg.load()
    yield fg._lib
    fg._lib.test_set("fp8_force", 0)


def _input(n, d, centres, spread, metric, rng, bf16=False):
    """Two shards of points around random centres (none: isotropic noise)."""
    import paper_2603_21710_gb300 as fg
    X = rng.standard_normal((n, d))
    if centres:
        X = rng.standard_normal((centres, d))[rng.integers(0, centres, n)] + spread * X
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    if bf16:
        X = X.to(torch.bfloat16).float()
    half = n // 2
    graphs = [fg.build_pg(x, M=12, ef=32, metric=metric) for x in (X[:half], X[half:])]
    return fg.MergeInput([X[:half], X[half:]], [a for a, _ in graphs], [e for _, e in graphs], metric=metric)


def _pass(inp, lists, join_filter, rev_cap=0):
    import paper_2603_21710_gb300 as fg
    g = {q: t.clone() for q, t in lists.items()}
    st = fg.refine_pass(inp, g, rev_cap=rev_cap, join_filter=join_filter)
    return g, st["join_class"], fg.last_join_operand()


# k, the share of new entries and the cap of the reverse lists: sets of at most 64, of 65 to 128, and above 128 candidates
# (the last of both kinds, so that the new ones are at most 128)
@pytest.mark.parametrize("k,new,cap,tile", [(14, 1.0, 0, 0), (50, 1.0, 0, 1), (120, 0.4, 55, 2)])
@pytest.mark.parametrize("metric", ["l2", "ip", "cos"])
@pytest.mark.parametrize("d", [36, 128, 260, 960])
def test_e4m3_tiles_keep_the_fp32_lists(hooks, d, metric, k, new, cap, tile):
    import paper_2603_21710_gb300 as fg
    rng = np.random.default_rng(d + k)
    inp = _input(1200, d, 4, 0.3, metric, rng)
    lists = {q: t for q, t in fg.cross_query(inp, k).items() if q != "stats"}
    lists["flags"] = torch.from_numpy((rng.random((1200, k)) < new).astype(np.uint8)).cuda()
    ref, cls, operand = _pass(inp, lists, "fp32", cap)
    assert operand == "none" and cls[3] > 0
    hooks.test_set("fp8_force", 1)
    got, cls, operand = _pass(inp, lists, "fp8", cap)
    assert operand == "e4m3" and cls[tile] > 0 and cls[3] == 0, (operand, cls)
    for q in ("ids", "dist", "flags"):
        assert torch.equal(got[q], ref[q]), q


def test_e4m3_is_kept_where_it_is_fine_enough(hooks):
    import paper_2603_21710_gb300 as fg
    inp = _input(1200, 256, 0, 0.0, "l2", np.random.default_rng(1))   # isotropic: neighbours about as far as the norms
    lists = {q: t for q, t in fg.cross_query(inp, 24).items() if q != "stats"}
    ref, _, _ = _pass(inp, lists, "fp32")
    got, cls, operand = _pass(inp, lists, "fp8")
    assert operand == "e4m3" and cls[3] == 0
    for q in ("ids", "dist", "flags"):
        assert torch.equal(got[q], ref[q]), q


@pytest.mark.parametrize("bf16,other", [(False, "fp16"), (True, "bf16")])
def test_a_coarse_e4m3_gives_way_and_keeps_no_memory(hooks, bf16, other):
    import paper_2603_21710_gb300 as fg
    inp = _input(6000, 960, 1, 0.05, "l2", np.random.default_rng(2), bf16)   # neighbours far nearer than the norms
    lists = {q: t for q, t in fg.cross_query(inp, 12).items() if q != "stats"}
    ref, _, _ = _pass(inp, lists, "fp32")
    high = {}
    for f in ("tc", "fp8"):
        torch.cuda.synchronize()
        hooks.test_set("pool_high_bytes", 0)
        got, cls, operand = _pass(inp, lists, f)
        high[f] = hooks.test_get("pool_high_bytes")
        assert operand == other and cls[3] == 0, (f, operand, cls)
        for q in ("ids", "dist", "flags"):
            assert torch.equal(got[q], ref[q]), (f, q)
    assert 0 < high["fp8"] <= high["tc"] + 4096, high
