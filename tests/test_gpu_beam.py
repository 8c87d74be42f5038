"""The beam search at the edges of its pool sizes and row widths.

Integer coordinates with many equal distances make every FP32 sum exact and every tie decided by
id, so the search must equal the oracle's bit for bit at any pool size; float rows of up to 128
coordinates must give the canonical FP32 distance, restated here in numpy.
"""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L2, IP = 0, 1


def _dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _graph(rng, n, R):
    g = np.full((n, R), -1, np.int32)
    for v in range(n):
        deg = int(rng.integers(R // 2, R + 1))
        g[v, :deg] = rng.choice(n, deg, replace=False)
    return g


def _search(X, g, Q, beam, topk, metric, dtype=None):
    import paper_2603_21710_gb300 as fg
    dev = _dev()
    t = [torch.from_numpy(a).to(dev) for a in (X, g, Q)]
    if dtype is not None:
        t[0], t[2] = t[0].to(dtype), t[2].to(dtype)
    ids, dist = fg.search(t[0], t[1], 3, t[2], topk=topk, beam=beam, metric={L2: "l2", IP: "ip"}[metric])
    return ids.cpu().numpy(), dist.cpu().numpy()


@pytest.mark.parametrize("beam", [1, 2, 31, 32, 33, 63, 64, 65, 96, 127, 128])
def test_search_pool_sizes_with_ties(beam):
    rng = np.random.default_rng(beam)
    X = rng.integers(0, 4, (700, 16)).astype(np.float32)
    Q = rng.integers(0, 4, (65, 16)).astype(np.float32)
    g = _graph(rng, 700, 40)
    ids, dist = _search(X, g, Q, beam, beam, L2)
    oi, od, _ = O.search(X, g, 3, Q, beam, beam, L2)
    assert np.array_equal(ids, oi)
    assert np.array_equal(dist, od)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("metric", [L2, IP])
@pytest.mark.parametrize("d", [4, 28, 32, 36, 64, 100, 124, 128, 132, 256, 260, 960])
def test_search_row_widths(d, metric, dtype):
    rng = np.random.default_rng(d)
    X = rng.integers(0, 8, (300, d)).astype(np.float32)
    Q = rng.integers(0, 8, (33, d)).astype(np.float32)
    g = _graph(rng, 300, 33)
    ids, dist = _search(X, g, Q, 48, 48, metric, torch.bfloat16 if dtype == "bf16" else None)
    oi, od, _ = O.search(X, g, 3, Q, 48, 48, metric)
    assert np.array_equal(ids, oi)
    assert np.array_equal(dist, od)


@pytest.mark.parametrize("metric", [L2, IP])
@pytest.mark.parametrize("d", [8, 32, 60, 68, 96, 128])
def test_float_rows_give_the_canonical_distance(d, metric):
    rng = np.random.default_rng(100 + d)
    X = rng.standard_normal((200, d)).astype(np.float32)
    Q = rng.standard_normal((20, d)).astype(np.float32)
    g = _graph(rng, 200, 24)
    ids, dist = _search(X, g, Q, 64, 64, metric)
    a, b = Q[:, None, :], X[ids]
    t = (a - b) * (a - b) if metric == L2 else a * b   # one rounding each, as a fused multiply-add with 0
    c = t.reshape(20, 64, d // 4, 4)
    p = np.zeros((20, 64, 32), np.float32)             # lane partials, one float4 chunk per lane
    p[:, :, :d // 4] = (c[..., 0] + c[..., 1]) + (c[..., 2] + c[..., 3])
    for o in (16, 8, 4, 2, 1):
        p = p[:, :, :o] + p[:, :, o:2 * o]
    s = p[:, :, 0]
    assert np.array_equal(dist, s if metric == L2 else np.float32(1) - s)


@pytest.mark.parametrize("nq", [1, 304, 305, 608, 609, 1216, 1217])
@pytest.mark.parametrize("d,dtype", [(20, "f32"), (132, "f32"), (768, "bf16"), (772, "bf16")])
def test_few_and_many_queries_agree(d, dtype, nq):
    """A query's result does not depend on how many come with it (a block per query, or a warp), cosine and
    layered searches included."""
    import paper_2603_21710_gb300 as fg
    dev = _dev()
    g = torch.Generator(device=dev).manual_seed(d)
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    X = torch.randn((3000, d), generator=g, device=dev).to(t)
    Q = torch.randn((1300, d), generator=g, device=dev).to(t)
    X[17] = 0   # a row without a norm
    adj, entry = fg.build_pg(X, M=12, ef=24, metric="cos")
    ly = fg.build_layers(X, M=8, ef=16, seed=3, metric="cos")
    a = fg.search(X, adj, entry, Q, topk=10, beam=40, metric="cos")
    b = fg.search(X, adj, entry, Q[:nq], topk=10, beam=40, metric="cos")
    c = fg.search_hnsw(X, adj, ly["layers"], ly["entry"], Q, topk=10, beam=40, metric="cos")
    e = fg.search_hnsw(X, adj, ly["layers"], ly["entry"], Q[:nq], topk=10, beam=40, metric="cos")
    for x, y in zip(a + c, b + e):
        assert torch.equal(x[:nq], y)
