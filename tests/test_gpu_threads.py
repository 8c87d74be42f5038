"""Calls of several host threads, each on its own stream, give what the same calls give alone.

The problems differ in dimension, storage, k and pool, so that the threads launch the same kernels with different amounts
of shared memory at the same time.
"""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# n, d, storage, k, join filter, search pool
PROBLEMS = [(3000, 32, torch.float32, 16, "tc", 64), (3500, 132, torch.float32, 40, "fp32", 128),
            (4000, 100, torch.bfloat16, 60, "tc", 24), (3000, 260, torch.float32, 8, "fp8", 48),
            (2500, 132, torch.bfloat16, 90, "tc", 100), (3000, 2048, torch.float32, 24, "tc", 128)]


def _problem(i, n, d, dtype):
    import paper_2603_21710_gb300 as fg
    g = torch.Generator(device="cuda:0")
    g.manual_seed(i)
    c = torch.randn(30, d, generator=g, device="cuda:0")
    X = c[torch.randint(0, 30, (n,), generator=g, device="cuda:0")] + 0.4 * torch.randn(n, d, generator=g, device="cuda:0")
    X = X.to(dtype)
    parts = [X[:n // 2].contiguous(), X[n // 2:].contiguous()]
    graphs = [fg.build_pg(x, M=12, ef=32) for x in parts]
    return fg.MergeInput(parts, [a for a, _ in graphs], [e for _, e in graphs]), X


def _calls(inp, X, k, join_filter, beam):
    import paper_2603_21710_gb300 as fg
    out = fg.merge(inp, k=k, R=16, alpha=1.2, join_filter=join_filter)
    ids, _ = fg.search(X, out["ids"], out["entry"], X[:900].contiguous(), topk=8, beam=beam)
    layers = fg.build_layers(X, M=8, ef=32, seed=1)
    adj, entry = fg.build_pg(X[:1500].contiguous(), M=12, ef=32)
    return [out["ids"], out["dist"], ids, adj] + [ly["adj"] for ly in layers["layers"]]


def test_threads_do_not_disturb_each_other():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    work = []
    for i, (n, d, dtype, k, join_filter, beam) in enumerate(PROBLEMS):
        inp, X = _problem(i, n, d, dtype)
        work.append(((inp, X, k, join_filter, beam), [t.clone() for t in _calls(inp, X, k, join_filter, beam)]))
    torch.cuda.synchronize()
    failed = []

    def run(i):
        args, want = work[i]
        stream = torch.cuda.Stream()
        try:
            with torch.cuda.stream(stream):
                for _ in range(12):
                    got = _calls(*args)
                    stream.synchronize()
                    if len(got) != len(want) or not all(torch.equal(a, b) for a, b in zip(got, want)):
                        failed.append((i, "results differ"))
        except Exception as ex:
            failed.append((i, repr(ex)))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
