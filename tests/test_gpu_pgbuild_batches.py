"""The graph builder around the edges of its mean (rows read in groups, byte rows summed in parts) and of its batches.

The medoid is that of the sequential FP64 sums, so the entry equals the host builder's for any data; on integer
data the graph does too, bit for bit, whatever order the batch's reverse edges are grouped in.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,d", [("bytes", 16), ("bytes", 112), ("integers", 20), ("integers", 132), ("floats", 36)])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 513, 1030, 2600])
def test_mean_and_reverse_edges(kind, d, n):
    import paper_2603_21710_gb300 as fg
    from synth import pgbuild
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(1000 * d + n)
    if kind == "floats":
        X = (rng.standard_normal((n, d)) * np.exp(4.0 * rng.standard_normal((n, 1)))).astype(np.float32)
    else:
        X = rng.integers(0, 6, (n, d)).astype(np.float32) - (2.0 if kind == "integers" else 0.0)
    adj, entry = fg.build_pg(torch.from_numpy(X).cuda(), M=8, ef=16)
    ref, ref_entry = pgbuild.build_pg(X, 8, 16, 0)
    assert entry == ref_entry
    if kind != "floats":
        assert np.array_equal(adj.cpu().numpy(), ref)


@pytest.mark.parametrize("scale", [1e-38, 1e-42, 1e30])
def test_mean_of_zeros_and_subnormals(scale):
    """Rows with zeros of either sign, subnormal and very large coordinates: the medoid is the host builder's."""
    import paper_2603_21710_gb300 as fg
    from synth import pgbuild
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(5)
    X = rng.standard_normal((333, 36)).astype(np.float32)
    X[::3, ::2] = (X[::3, ::2].astype(np.float64) * scale).astype(np.float32)
    X[::7, ::5] = 0.0
    X[1::7, ::5] = -0.0
    _, entry = fg.build_pg(torch.from_numpy(X).cuda(), M=8, ef=16)
    assert entry == pgbuild.build_pg(X, 8, 16, 0)[1]
