"""Neighbour selection where a list ends early, under every metric and row storage.

A list is its entries before the first empty one (the oracle's rule): whatever stands behind it must neither be
kept nor read as a vertex. Small integer coordinates make squared L2 and inner product exact, so those must equal the
oracle bit for bit; under cosine a list with a hole must give what the list cut there gives.
"""
import functools

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# N (at most 2,048: four warps per vertex), d, k, R, coordinate range, dtype: bytes (two windows), bytes beyond 64, rows staged,
# rows in place, wide FP32 and BF16 rows
FORMS = [(2100, 16, 64, 32, 0, 256, "f32"), (2100, 32, 33, 33, 0, 256, "f32"), (2100, 16, 100, 40, 0, 256, "f32"),
         (2100, 36, 48, 24, -9, 9, "f32"), (2100, 128, 100, 64, -9, 9, "f32"), (2100, 132, 40, 24, -9, 9, "f32"),
         (2100, 132, 40, 24, -9, 9, "bf16"), (2100, 260, 70, 32, -9, 9, "bf16"), (300, 16, 64, 32, 0, 256, "f32"),
         (301, 36, 70, 32, -9, 9, "f32"), (300, 132, 70, 20, -9, 9, "f32"), (301, 260, 33, 16, -9, 9, "bf16")]


@functools.lru_cache(maxsize=None)
def _problem(N, d, k, lo, hi, metric):
    """Vectors and random sorted lists with holes, exact distances (cosine: rounded) and some protected vertices."""
    rng = np.random.default_rng(N + d + k)
    X = rng.integers(lo, hi, (N, d)).astype(np.float32)
    nrm = np.sqrt((X.astype(np.float64) ** 2).sum(1))
    ids = np.full((N, k), -1, np.int32)
    dist = np.full((N, k), np.inf, np.float32)
    for u in range(N):
        v = rng.permutation(N - 1)[:k]
        v[v >= u] += 1
        if metric == "l2":
            dv = ((X[v] - X[u]) ** 2).sum(1)
        else:
            dv = X[v].astype(np.float64) @ X[u].astype(np.float64)
            dv = 1.0 - (dv if metric == "ip" else dv / np.maximum(nrm[v] * nrm[u], 1e-30))
        dv = dv.astype(np.float32)
        o = np.lexsort((v, dv))
        ids[u, :len(v)], dist[u, :len(v)] = v[o], dv[o]
    cut = rng.integers(0, k + 1, N)
    cut[::5] = k                      # whole lists
    cut[1::5] = min(k - 1, 40)        # past a window of 32
    T = rng.integers(1, 5, N).astype(np.int32)
    return X, ids, dist, T, cut


def _prune(X, ids, dist, T, R, metric, dtype, alpha, rule):
    import paper_2603_21710_gb300 as fg
    dev = torch.device("cuda:0")
    N = len(X)
    sizes, adj = [N // 2, N - N // 2], torch.full((N, 1), -1, dtype=torch.int32, device=dev)
    x = torch.from_numpy(X).to(dev)
    inp = fg.MergeInput.from_flat(x.to(torch.bfloat16) if dtype == "bf16" else x, sizes, adj, [0, 0], metric=metric)
    kn = {"ids": torch.from_numpy(ids).to(dev), "dist": torch.from_numpy(dist).to(dev)}
    return [t.cpu().numpy() for t in fg.prune(inp, kn, torch.from_numpy(T).to(dev), R, alpha, rule=rule)]


@pytest.mark.parametrize("rule,alpha", [("arng", 1.0), ("arng", 1.3), ("mrng", 1.0)])
@pytest.mark.parametrize("metric", ["l2", "ip", "cos"])
@pytest.mark.parametrize("N,d,k,R,lo,hi,dtype", FORMS)
def test_a_list_ends_at_its_first_empty_entry(N, d, k, R, lo, hi, dtype, metric, rule, alpha):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X, full, fdist, T, cut = _problem(N, d, k, lo, hi, metric)
    holes, ended, edist = full.copy(), full.copy(), fdist.copy()
    for u in range(N):
        holes[u, cut[u]:cut[u] + 1] = -1           # valid ids go on behind the hole
        ended[u, cut[u]:] = -1
        edist[u, cut[u]:] = np.inf
    got = _prune(X, holes, fdist, T, R, metric, dtype, alpha, rule)
    want = _prune(X, ended, edist, T, R, metric, dtype, alpha, rule)
    if metric != "cos":
        P = O.Problem(X, [N // 2, N - N // 2], np.full((N, 1), -1, np.int32), np.zeros(2, np.int32), {"l2": 0, "ip": 1}[metric])
        g = O.KNNG(N, k)
        g.ids[:], g.dist[:] = ended, edist
        oi, od, oc, _ = O.prune(P, g, T, R, alpha, rule=rule)
        for a, b in zip(want, (oi, od, oc)):
            assert np.array_equal(a, b)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    assert ((got[0] >= 0).sum(1) == got[2]).all()


@pytest.mark.parametrize("metric", ["l2", "cos"])
@pytest.mark.parametrize("N,d,k,R,lo,hi,dtype", FORMS)
def test_an_id_past_the_vertices_is_reported(N, d, k, R, lo, hi, dtype, metric):
    import paper_2603_21710_gb300 as fg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X, full, fdist, T, _ = _problem(N, d, k, lo, hi, metric)
    for at in (0, min(k - 1, 33)):
        ids = full.copy()
        ids[N // 3, at] = N
        with pytest.raises(fg.FgimError, match="out of range"):
            _prune(X, ids, fdist, T, R, metric, dtype, 1.2, "arng")
