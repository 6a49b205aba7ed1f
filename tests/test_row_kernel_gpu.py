"""The row kernel (large channel counts) at the sizes where it can go wrong:
one output, ragged last batches, the edge between its small batches (calls
that give an SM at most one) and its whole ones, ranges of several batches,
tap counts below their bucket and, beyond 16 taps, around the blocks of its
loop.  Tolerance: relative L2 <= 1e-5 against the
FP64 oracle, as for every complex FP32 output; both batch sizes do the same
arithmetic per output, so their results are equal bit for bit.
"""
import numpy as np
import pytest

import oracle
from paper_1511_03599_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIGMA = {"ci8": 16.0, "ci16": 2000.0, "cf32": 1.0}
ROW = 128                                             # plan_info variant bit of the row kernel
SHAPES = [(384, 8, "ci8"), (384, 13, "cf32"), (768, 3, "ci16"), (768, 16, "ci16"), (1024, 8, "ci16"), (1024, 5, "cf32"),
          (1024, 16, "ci8"), (1536, 7, "ci16"), (1536, 1, "cf32"), (2048, 8, "ci8"), (2048, 3, "cf32"),
          (2048, 16, "cf32"), (3072, 8, "ci16"), (3072, 6, "cf32"), (4096, 8, "ci8"), (4096, 13, "ci8"),
          (4096, 2, "ci16"), (4096, 6, "cf32"),
          (384, 23, "ci8"), (384, 40, "cf32"), (768, 33, "ci16"), (1024, 20, "cf32"), (1024, 64, "ci8"), (1536, 17, "cf32"),
          (2048, 31, "ci16"), (3072, 19, "cf32"), (3072, 64, "ci8"), (4096, 17, "ci8"), (4096, 45, "cf32")]


@pytest.fixture(scope="module")
def ppf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_03599_gb300 import ppf as m
    m.lib()
    return m


@pytest.mark.parametrize("C,T,in_dtype", SHAPES)
def test_short_and_long_calls_agree(ppf, C, T, in_dtype):
    h = synth.design_taps(C, T)
    with ppf.Plan(C, T, h, in_dtype, "c64") as plan:
        info = plan.info()
        assert info["variant"] & ROW
        B = info["batch"]
        S = 2 * info["grid"] * B + B // 2 + 1             # ranges of two and three batches, a ragged end
        x = synth.stream(C, S + T - 1, in_dtype, SIGMA[in_dtype], 7000 + C + T)
        xd = torch.from_numpy(x).cuda()
        y = torch.view_as_real(plan(xd))
        sms = info["grid"]
        for n in (1, max(1, B - 1), B + 1, sms * max(1, B // 4) // 2, sms * max(1, B // 4) + 1, sms * B // 2 + 3):
            s0 = (S - n) // 2
            part = torch.view_as_real(plan(xd[s0 * C:(s0 + n + T - 1) * C].clone()))
            assert torch.equal(part, y[s0:s0 + n]), n
        plan.check_device()
        idx = np.unique(np.concatenate([np.arange(T), np.arange(S - T, S), np.linspace(0, S - 1, 40).astype(np.int64)]))
        got = torch.view_as_complex(y)[torch.from_numpy(idx).cuda()].cpu().numpy()
    assert oracle.rel_l2_max_per_spectrum(got, oracle.pfb_spectra(x, h, C, T, idx)) <= 1e-5


@pytest.mark.parametrize("C,T", [(384, 5), (1024, 6), (1024, 3), (3072, 8), (4096, 3), (2048, 13), (1024, 21), (3072, 32), (4096, 18)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_sample_reaches_only_its_spectra(ppf, C, T, bad):
    """One inf or NaN sample of FP32 input reaches the T output spectra that read it and
    no other, whether the call runs on small or on whole batches."""
    with ppf.Plan(C, T, synth.design_taps(C, T), "cf32", "c64") as plan:
        for S in (3 * T + 2, 3 * plan.info()["grid"] * plan.info()["batch"]):
            x = synth.stream(C, S + T - 1, "cf32", 1.0, 7100 + C)
            r = S // 2 + T
            x[r * C + C // 3, 0] = bad
            finite = torch.isfinite(torch.view_as_real(plan(torch.from_numpy(x).cuda()))).all(dim=-1).all(dim=-1)
            want = torch.ones(S, dtype=torch.bool)
            want[r - T + 1:r + 1] = False
            assert torch.equal(finite.cpu(), want[:S])


@pytest.mark.parametrize("C,in_dtype,out_dtype", [(1536, "ci8", "c16"), (4096, "ci8", "c16"), (1024, "cf32", "c16")])
def test_many_short_streams(ppf, C, in_dtype, out_dtype):
    """Streams shorter than a batch: small batches for a few, shares of whole batches that
    cross streams for many; equal to one launch per stream."""
    T, S = 8, 3
    h = synth.design_taps(C, T, scale=1.0 / np.sqrt(C))
    with ppf.Plan(C, T, h, in_dtype, out_dtype) as plan:
        for ns in (5, 700):
            x = torch.from_numpy(np.stack([synth.stream(C, S + T - 1, in_dtype, SIGMA[in_dtype], 7200 + i)
                                           for i in range(ns)])).cuda()
            y = plan.execute(x, n_streams=ns)
            for i in (0, ns // 2, ns - 1):
                assert torch.equal(y[i], plan(x[i].clone())), i
        plan.check_device()
