"""The long-tap kernel (T = 17..64, C = 64..512) at the sizes where it can go
wrong: tap counts around its blocks of 8 (one tap left over brings in no row),
one output, the edge between its batches of 16 (short calls) and of 32, ragged
ends, streams shorter than a batch.  Relative L2 <= 1e-5 against the FP64
oracle; both batch sizes do the same arithmetic per output, so their results
are equal bit for bit.
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


@pytest.mark.parametrize("C,T,in_dtype", [(64, 17, "ci8"), (64, 24, "cf32"), (128, 25, "ci16"), (128, 63, "cf32"),
                                          (256, 33, "cf32"), (256, 64, "ci8"), (512, 18, "ci16"), (512, 32, "ci8"),
                                          (512, 49, "cf32"), (512, 64, "ci16")])
def test_batches_of_16_and_32_agree(ppf, C, T, in_dtype):
    h = synth.design_taps(C, T)
    with ppf.Plan(C, T, h, in_dtype, "c64") as plan:
        info = plan.info()
        assert info["variant"] & 64 and info["batch"] == 32
        S = 2 * info["grid"] * 32 + 21
        x = synth.stream(C, S + T - 1, in_dtype, SIGMA[in_dtype], 9000 + C + T)
        xd = torch.from_numpy(x).cuda()
        y = torch.view_as_real(plan(xd))
        for n in (1, 15, 17, 33, 152 * 16, 152 * 16 + 1, info["grid"] * 32 - 7):
            s0 = max(0, (S - n) // 2)
            part = torch.view_as_real(plan(xd[s0 * C:(s0 + n + T - 1) * C].clone()))
            assert torch.equal(part, y[s0:s0 + n]), n
        for ns in (3, 400):                               # streams of 7 spectra, in few and in many CTAs
            xs = xd[:ns * (7 + T - 1) * C].reshape(ns, -1, 2).contiguous() if ns == 3 else \
                xd[:(7 + T - 1) * C].reshape(1, -1, 2).repeat(ns, 1, 1).contiguous()
            ys = plan.execute(xs, n_streams=ns)
            for i in (0, 1, ns - 1):
                assert torch.equal(ys[i], plan(xs[i].clone())), (ns, i)
        plan.check_device()
        idx = np.unique(np.concatenate([np.arange(T), np.arange(S - T, S), np.linspace(0, S - 1, 40).astype(np.int64)]))
        got = torch.view_as_complex(y)[torch.from_numpy(idx).cuda()].cpu().numpy()
    assert oracle.rel_l2_max_per_spectrum(got, oracle.pfb_spectra(x, h, C, T, idx)) <= 1e-5


@pytest.mark.parametrize("C,T", [(64, 25), (256, 32), (512, 41)])
def test_non_finite_sample_reaches_only_its_spectra(ppf, C, T):
    with ppf.Plan(C, T, synth.design_taps(C, T), "cf32", "c64") as plan:
        for S in (3 * T, 2 * plan.info()["grid"] * 32):
            x = synth.stream(C, S + T - 1, "cf32", 1.0, 9100 + C)
            r = S // 2 + T
            x[r * C + C // 3, 0] = np.nan
            finite = torch.isfinite(torch.view_as_real(plan(torch.from_numpy(x).cuda()))).all(dim=-1).all(dim=-1)
            want = torch.ones(S, dtype=torch.bool)
            want[r - T + 1:r + 1] = False
            assert torch.equal(finite.cpu(), want)


def test_timeout_is_reported_and_the_next_call_is_right(ppf):
    """The injected wait runs out: status reported, context usable, next result right."""
    C, T, S = 256, 40, 3000
    h = synth.design_taps(C, T)
    x = synth.stream(C, S + T - 1, "ci8", 16.0, 9200)
    xd = torch.from_numpy(x).cuda()
    with ppf.Plan(C, T, h, "ci8", "c64") as plan:
        plan.set_debug_flags(1)
        plan(xd)
        with pytest.raises(ppf.PPFError) as ei:
            plan.check_device()
        assert ei.value.status == 5
        plan.set_debug_flags(0)
        got = plan(xd).cpu().numpy()
        plan.check_device()
    assert oracle.rel_l2(got, oracle.pfb(x, h, C, T)) <= 1e-5
