"""Two contexts on two host threads, one stream each (what the end-to-end leg of the benchmark does): no call fails, and
every result is bit for bit what the same call gives alone. The pairs are chosen so that the two threads keep launching the
same kernels with different sizes of shared memory."""
import threading

import pytest
import torch

from paper_2609_21102_b200 import binding

pytestmark = pytest.mark.gpu
MUON = [list(binding.MUON_QUINTIC)] * 5
CLASSICAL = [list(binding.CLASSICAL_QUINTIC)] * 5


def _polar(b, m, n, k=16):
    g = torch.Generator(device="cuda").manual_seed(b + m + n)
    G = torch.randn((b, m, n), generator=g, device="cuda").bfloat16()
    return lambda c: c.defl_polar_batched(G, k, 8, 1, MUON, seed=3, gamma=1.01, exploit_symmetry=True)


def _psd(n, K=8):
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((n, n), generator=g, device="cuda")
    X = x + x.T
    V = torch.linalg.qr(torch.randn((n, K), generator=g, device="cuda"))[0].contiguous()
    return lambda c: c.defl_psd_project(X, 4, V.clone(), CLASSICAL, gamma=1.1, seed=5)


@pytest.mark.parametrize("one,two", [(lambda: _polar(8, 1600, 1600, 32), lambda: _polar(8, 1600, 3200, 32)),
                                     (lambda: _polar(12, 768, 768), lambda: _polar(8, 1024, 4096)),
                                     (lambda: _psd(1000), lambda: _psd(1024)),
                                     (lambda: _psd(2048), lambda: _psd(4096)),
                                     (lambda: _polar(4, 256, 384), lambda: _psd(640))],
                         ids=["polar_1600", "polar_768_1024", "psd_sums_by_all", "psd_sums_by_one", "polar_psd"])
def test_two_contexts_on_two_threads(one, two):
    calls = [one(), two()]
    alone = []
    for call in calls:
        c = binding.Context(0)
        alone.append(call(c).clone())
        torch.cuda.synchronize()
        c.close()
    errors, results = [], [None, None]
    start = threading.Barrier(2)

    def work(i):
        try:
            torch.cuda.set_device(0)
            c = binding.Context(0)
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                outs = [calls[i](c) for _ in range(50)]
                torch.cuda.current_stream().synchronize()
                results[i] = [torch.equal(o, alone[i]) for o in outs]
            c.close()
        except Exception as e:
            errors.append(repr(e))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert all(results[0]) and all(results[1])
