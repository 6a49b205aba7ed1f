"""Short calls at C <= 1024: the row kernel's small batches, the carry kernel's
form for short ranges and its form for long ones do the same arithmetic per
output, so a slice of a stream gives the same bits through each.  Sizes sit
around the edges of the rules (one output, one small batch per SM, a few
batches per CTA, 16 batches per CTA) with ragged ends and tap counts below
their bucket; relative L2 <= 1e-5 against the FP64 oracle.
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


@pytest.mark.parametrize("C,T,in_dtype", [(64, 8, "ci8"), (64, 3, "cf32"), (128, 16, "ci16"), (128, 1, "cf32"),
                                          (256, 8, "cf32"), (256, 13, "ci8"), (512, 8, "ci8"), (512, 16, "ci16"),
                                          (512, 5, "cf32"), (1024, 8, "ci8"), (1024, 2, "ci8")])
def test_every_form_gives_the_same_bits(ppf, C, T, in_dtype):
    h = synth.design_taps(C, T)
    with ppf.Plan(C, T, h, in_dtype, "c64") as plan:
        info = plan.info()
        B, grid = info["batch"], info["grid"]
        S = 17 * grid * B + 3                             # beyond the short ranges
        x = synth.stream(C, S + T - 1, in_dtype, SIGMA[in_dtype], 8000 + C + T)
        xd = torch.from_numpy(x).cuda()
        y = torch.view_as_real(plan(xd))
        small = 4096 // C * 152                           # about one small batch per SM
        for n in (1, B - 1, B + 1, small, small + 1, grid * B - 1, 2 * grid * B + 1, 16 * grid * B - 5):
            if n < 1 or n > S:
                continue
            s0 = (S - n) // 2
            part = torch.view_as_real(plan(xd[s0 * C:(s0 + n + T - 1) * C].clone()))
            assert torch.equal(part, y[s0:s0 + n]), n
        xs = xd[:3 * (B + 2 + T - 1) * C].reshape(3, -1, 2).contiguous()    # three streams of a few spectra
        ys = plan.execute(xs, n_streams=3)
        for i in range(3):
            assert torch.equal(ys[i], plan(xs[i].clone())), i
        plan.check_device()
        idx = np.unique(np.concatenate([np.arange(T), np.arange(S - T, S), np.linspace(0, S - 1, 40).astype(np.int64)]))
        n = 2 * B + 3
        short = plan(xd[:(n + T - 1) * C].clone()).cpu().numpy()
        got = torch.view_as_complex(y)[torch.from_numpy(idx).cuda()].cpu().numpy()
    assert oracle.rel_l2_max_per_spectrum(got, oracle.pfb_spectra(x, h, C, T, idx)) <= 1e-5
    assert oracle.rel_l2_max_per_spectrum(short, oracle.pfb(x[:(n + T - 1) * C], h, C, T)) <= 1e-5


@pytest.mark.parametrize("C,T", [(64, 5), (256, 8), (512, 3)])
def test_non_finite_sample_in_short_calls(ppf, C, T):
    """One inf sample of FP32 input reaches the T output spectra that read it and no other."""
    with ppf.Plan(C, T, synth.design_taps(C, T), "cf32", "c64") as plan:
        for S in (3 * T + 2, 3 * plan.info()["grid"] * plan.info()["batch"]):
            x = synth.stream(C, S + T - 1, "cf32", 1.0, 8100 + C)
            r = S // 2 + T
            x[r * C + C // 3, 0] = np.inf
            finite = torch.isfinite(torch.view_as_real(plan(torch.from_numpy(x).cuda()))).all(dim=-1).all(dim=-1)
            want = torch.ones(S, dtype=torch.bool)
            want[r - T + 1:r + 1] = False
            assert torch.equal(finite.cpu(), want)
