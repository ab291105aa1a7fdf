"""Calls that share the library's workspace pool: several host threads, each on a stream of
its own, with sizes that grow and shrink; every result must be the one of the same call made
alone (the kernels' summation orders do not depend on the buffer), bit for bit."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [1, 4])
def test_concurrent_calls(gpu_bmg, threads):
    g = torch.Generator(device="cuda").manual_seed(5)
    cases = []
    for n, k in [(70, 3), (642, 128), (10242, 33), (2562, 64), (10242, 128)]:
        ld = (k + 1) // 2 * 2
        X = torch.randn((n, ld), dtype=torch.float64, device="cuda", generator=g)
        Y = torch.randn((k, k), dtype=torch.float64, device="cuda", generator=g)
        cases.append((X, Y, k))

    def run(X, Y, k):
        G = torch.empty((k, k), dtype=torch.float64, device="cuda")
        U, th, V = torch.zeros_like(X), torch.empty(k, dtype=torch.float64, device="cuda"), torch.empty_like(G)
        gpu_bmg.gram_tc(X, X, k, G)
        gpu_bmg.expand(None, X, Y, k, U)
        gpu_bmg.dense_eig(G, torch.eye(k, dtype=torch.float64, device="cuda"), 0.0, k, th, V)
        return G, U, th

    ref = [run(*c) for c in cases]
    torch.cuda.synchronize()
    bad = []

    def worker(t):
        with torch.cuda.stream(torch.cuda.Stream()):
            for it in range(6):
                q = (t + it) % len(cases)
                out = run(*cases[q])
                torch.cuda.current_stream().synchronize()
                if not all(torch.equal(a, b) for a, b in zip(out, ref[q])):
                    bad.append((t, q))

    pool = [threading.Thread(target=worker, args=(t,)) for t in range(threads)]
    for t in pool:
        t.start()
    for t in pool:
        t.join()
    assert not bad
