"""The graph builder where one vertex receives more reverse edges in a batch than a merged list holds.

Identical points (every distance ties) and a row that is the nearest to every other under the inner product make
such hubs; on integer data the graph equals the host builder's bit for bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M", [(300, 12), (700, 12), (2600, 128)])
@pytest.mark.parametrize("kind", ["identical", "big_row"])
def test_hubs_equal_the_host_builder(kind, n, M):
    import paper_2603_21710_gb300 as fg
    from synth import pgbuild
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(n)
    if kind == "identical":
        X, metric = np.full((n, 20), 7.0, np.float32), 0
    else:
        X, metric = rng.integers(0, 4, (n, 20)).astype(np.float32), 1
        X[n // 2] = 200.0
    adj, entry = fg.build_pg(torch.from_numpy(X).cuda(), M=M, ef=48, metric=metric)
    ha, he = pgbuild.build_pg(X, M, 48, metric)
    assert entry == he
    assert np.array_equal(adj.cpu().numpy(), ha)
