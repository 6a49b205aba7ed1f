"""Calls of many streams, and of lengths just over a round of batches, on the row and
the long-tap kernel: whichever batches a call runs on, each stream gives the bits of
the stream alone, and every output is written.  A few spectra per stream against the
FP64 oracle (relative L2 <= 1e-5).
"""
import numpy as np
import pytest

import oracle
from paper_1511_03599_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIGMA = {"ci8": 16.0, "ci16": 2000.0, "cf32": 1.0}


@pytest.fixture(scope="module")
def ppf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_03599_gb300 import ppf as m
    m.lib()
    return m


@pytest.mark.parametrize("C,T,in_dtype", [(384, 4, "ci8"), (768, 16, "cf32"), (1024, 3, "ci16"), (1024, 24, "cf32"),
                                          (2048, 8, "ci8"), (3072, 1, "cf32"), (4096, 16, "ci8"), (64, 17, "cf32"),
                                          (128, 24, "ci8"), (256, 64, "ci16"), (512, 33, "ci8")])
@pytest.mark.parametrize("ns,S", [(160, 1), (200, 4), (640, 9), (1500, 2), (64, 41), (3, 2900)])
def test_each_stream_gives_its_own_bits(ppf, C, T, in_dtype, ns, S):
    n_in = C * (S + T - 1)
    if ns * n_in > 1 << 25:
        pytest.skip("too large for a small test")
    h = synth.design_taps(C, T)
    base = torch.from_numpy(synth.stream(C, S + T + 30, in_dtype, SIGMA[in_dtype], 9900 + C + T)).cuda()
    xs = torch.stack([base[(i % 31) * C:(i % 31) * C + n_in] for i in range(ns)])
    with ppf.Plan(C, T, h, in_dtype, "c64") as plan:
        out = torch.full((ns, S, C), float("nan"), dtype=torch.complex64, device="cuda")
        ys = plan.execute(xs, out=out, n_streams=ns)
        plan.check_device()
        assert bool(torch.isfinite(torch.view_as_real(ys)).all())
        for i in sorted({0, 1, ns // 2, ns - 1}):
            assert torch.equal(torch.view_as_real(ys[i]), torch.view_as_real(plan(xs[i].clone()))), i
        for i in range(31, min(ns, 300)):
            assert torch.equal(torch.view_as_real(ys[i]), torch.view_as_real(ys[i % 31])), i
        plan.check_device()
        got = ys[ns - 1].cpu().numpy()
    x = xs[ns - 1].cpu().numpy()
    idx = np.unique(np.linspace(0, S - 1, 12).astype(np.int64))
    assert oracle.rel_l2_max_per_spectrum(got[idx], oracle.pfb_spectra(x, h, C, T, idx)) <= 1e-5
