"""Neighbour selection at the edges of its windows, row storages and list lengths.

Integer coordinates make every distance exact, so the kept lists must equal the oracle's bit for bit
whichever form a list takes: bytes (integers in [0, 255], d % 16 == 0, k <= 64), rows staged in shared
memory, rows read in place, wide rows, and four warps per vertex (few lists).
"""
import functools

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@functools.lru_cache(maxsize=None)
def _problem(N, d, k, lo, hi):
    """Vectors and random sorted lists of length 0 .. k with exact distances."""
    rng = np.random.default_rng(N + d + k)
    X = rng.integers(lo, hi, (N, d)).astype(np.float32)
    ids = np.full((N, k), -1, np.int32)
    dist = np.full((N, k), np.inf, np.float32)
    for u in range(N):
        n = k if u % 3 else int(rng.integers(0, k + 1))
        v = rng.permutation(N - 1)[:n]
        v[v >= u] += 1
        dv = ((X[v] - X[u]) ** 2).sum(1)
        o = np.lexsort((v, dv))
        ids[u, :n], dist[u, :n] = v[o], dv[o]
    T = rng.integers(1, 4, N).astype(np.int32)   # a third of the vertices are protected
    return X, ids, dist, T


@pytest.mark.parametrize("rule,alpha", [("arng", 1.0), ("arng", 1.3), ("mrng", 1.0), ("tmng", 1.0)])
@pytest.mark.parametrize("N,d,k,R,lo,hi", [
    (2100, 16, 1, 1, 0, 256), (2100, 16, 33, 32, 0, 256), (2100, 32, 64, 20, 0, 256), (2100, 128, 64, 32, 100, 110),
    (2100, 16, 64, 128, 0, 256), (2100, 48, 65, 40, 0, 256), (2100, 16, 128, 24, 0, 256),   # bytes, and beyond 64
    (2100, 4, 16, 32, -9, 9), (2100, 36, 48, 32, -9, 9), (2100, 128, 31, 8, -9, 9),         # rows staged
    (2100, 100, 49, 32, -9, 9), (2100, 128, 128, 64, -9, 9),                                # rows in place
    (2100, 132, 40, 24, -9, 9), (300, 260, 70, 32, -9, 9),                                  # wide rows
    (300, 16, 64, 32, 0, 256), (301, 36, 128, 32, -9, 9), (40, 128, 33, 16, -9, 9)])        # four warps per vertex
def test_selection_equals_oracle(N, d, k, R, lo, hi, rule, alpha):
    import paper_2603_21710_gb300 as fg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X, ids, dist, T = _problem(N, d, min(k, N - 1), lo, hi)
    sizes, adj = [N // 2, N - N // 2], np.full((N, 1), -1, np.int32)
    tau = 2.0 if rule == "tmng" else 0.0
    P = O.Problem(X, sizes, adj, np.zeros(2, np.int32), 0)
    g = O.KNNG(N, ids.shape[1])
    g.ids[:], g.dist[:] = ids, dist
    oi, od, oc, _ = O.prune(P, g, T, R, alpha, rule=rule, tau=tau)
    dev = torch.device("cuda:0")
    inp = fg.MergeInput.from_flat(torch.from_numpy(X).to(dev), sizes, torch.from_numpy(adj).to(dev), [0, 0])
    kn = {"ids": torch.from_numpy(ids).to(dev), "dist": torch.from_numpy(dist).to(dev)}
    ei, ed, ec = fg.prune(inp, kn, torch.from_numpy(T).to(dev), R, alpha, rule=rule, tau=tau)
    assert np.array_equal(ec.cpu().numpy(), oc)
    assert np.array_equal(ei.cpu().numpy(), oi)
    assert np.array_equal(ed.cpu().numpy(), od)
