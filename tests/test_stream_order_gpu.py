"""Short calls are set up while the kernel before them still runs: results must be
those of plain stream order.  A chain of dependent short calls, with torch
kernels, copies and tap updates between them, on the default and on a side
stream and replayed from a CUDA graph, equals the same chain synchronised
after every call, bit for bit.
"""
import numpy as np
import pytest

from paper_1511_03599_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ppf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_03599_gb300 import ppf as m
    m.lib()
    return m


@pytest.mark.parametrize("C,T,S", [(512, 8, 64), (256, 8, 4096), (1024, 4, 40), (4096, 8, 20), (256, 32, 300), (3072, 3, 500)])
def test_chain_of_dependent_calls(ppf, C, T, S):
    h = synth.design_taps(C, T)
    x0 = torch.view_as_complex(torch.from_numpy(synth.stream(C, S + T - 1, "cf32", 1.0, 77))).cuda()
    h2 = torch.from_numpy(h[::-1].copy()).cuda()
    steps = 40

    with ppf.Plan(C, T, h, "cf32", "c64") as plan:
        h1 = torch.from_numpy(h).cuda()

        def chain(sync):
            x = x0.clone()
            y = torch.empty((S, C), dtype=torch.complex64, device="cuda")
            gx = gh = None
            for i in range(steps):
                plan.update_taps(h1 if i % 3 else h2)
                plan(x, out=y)
                sync()
                x[:S * C].copy_(y.reshape(-1) * (1.0 / C ** 0.5))      # the next call reads what this one wrote
                sync()
                plan(x, out=y)
                plan(x, out=y)
                x[:S * C] += y.reshape(-1) * 1e-3
                sync()
            gx, gh = plan.backward(y, x)
            sync()
            return x, y, gx, gh

        want = [v.clone() for v in chain(torch.cuda.synchronize)]
        got = chain(lambda: None)
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            got2 = chain(lambda: None)
        side.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            got3 = chain(lambda: None)
        g.replay()
        torch.cuda.synchronize()
        plan.check_device()
    for run in (got, got2, got3):
        for a, b in zip(want, run):
            assert torch.equal(torch.view_as_real(a) if a.is_complex() else a, torch.view_as_real(b) if b.is_complex() else b)
    assert all(bool(torch.isfinite(torch.view_as_real(v) if v.is_complex() else v).all()) for v in want)
