"""A bounded device wait that runs out (a barrier that nothing completes, 2 ms): the
status is reported, no result that depends on it looks complete, the launch ends at
once, and the next call is right.  In the three-pass adjoint at C >= 64 the inverse
DFT gives up and the second pass must not use its rows; at C = 32, whose inverse DFT
waits for nothing, the second pass gives up itself.
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


@pytest.mark.parametrize("C,T,in_dtype,S", [(512, 32, "ci8", 20), (512, 32, "ci8", 900), (512, 16, "cf32", 5000),
                                            (1024, 8, "cf32", 300), (4096, 8, "ci8", 40), (3072, 3, "ci16", 150),
                                            (128, 17, "ci16", 2500), (32, 8, "cf32", 3000)])
def test_three_pass_adjoint_reports_a_timeout(ppf, C, T, in_dtype, S):
    rng = np.random.default_rng(C + T)
    h = synth.design_taps(C, T)
    x = synth.stream(C, S + T - 1, in_dtype, SIGMA[in_dtype], 9500 + C)
    xd = torch.from_numpy(x).cuda()
    G = torch.from_numpy((rng.standard_normal((S, C)) + 1j * rng.standard_normal((S, C))).astype(np.complex64)).cuda()
    with ppf.Plan(C, T, h, in_dtype, "c64") as plan:
        plan.set_debug_flags(1)
        for want_input, want_taps in ((True, True), (True, False), (False, True)):
            gx, gh = plan.backward(G, xd, want_input=want_input, want_taps=want_taps)
            with pytest.raises(ppf.PPFError) as ei:
                plan.check_device()
            assert ei.value.status == 5
            if want_input and C != 32:
                assert bool(torch.isnan(torch.view_as_real(gx)).all())
            if want_taps:
                assert bool(torch.isnan(gh).all())
        plan.set_debug_flags(0)
        gx, gh = plan.backward(G, xd)
        plan.check_device()
    Gn = G.cpu().numpy().astype(np.complex128)
    assert oracle.rel_l2(gx.cpu().numpy().reshape(-1), oracle.pfb_grad_input(Gn, h, C, T).reshape(-1)) <= 1e-5
    assert oracle.rel_l2(gh.cpu().numpy(), oracle.pfb_grad_taps(Gn, x, C, T)) <= 1e-4


def _milliseconds(fn):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    a.record()
    fn()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b)


@pytest.mark.parametrize("C,T,in_dtype,S,back", [(64, 40, "ci8", 800000, False), (512, 40, "cf32", 60000, False),
                                                 (32, 32, "cf32", 800000, True)])
def test_a_launch_that_gave_up_ends_at_once(ppf, C, T, in_dtype, S, back):
    """The time to leave does not grow with the batches left (the long-tap kernel and
    the three-pass adjoint's second pass, dozens of batches per CTA): the 2 ms wait
    and at most the batch at hand."""
    dtype = {"ci8": torch.int8, "cf32": torch.float32}[in_dtype]
    x = torch.ones((C * (S + T - 1), 2), dtype=dtype, device="cuda")
    with ppf.Plan(C, T, synth.design_taps(C, T), in_dtype, "c64") as plan:
        y = plan(x)
        call = (lambda: plan.backward(y, x)) if back else (lambda: plan.execute(x, out=y))
        call()
        plan.check_device()
        good = _milliseconds(call)
        plan.set_debug_flags(1)
        ms = _milliseconds(call)
        with pytest.raises(ppf.PPFError):
            plan.check_device()
        assert 1.5 <= ms <= good + 30.0


# variant bits: 1 raw rows through a TMA ring, 4 carry kernel, 16 cluster kernel, 64 long-tap
# kernel, 128 row kernel
@pytest.mark.parametrize("C,T,in_dtype,S,family,ring", [(32, 8, "ci8", 5000, 0, 1), (32, 16, "cf32", 300, 0, 1),
                                                        (4096, 8, "ci8", 3000, 128, 1), (3072, 8, "cf32", 3000, 128, 0),
                                                        (1024, 4, "cf32", 6000, 128, 0), (3072, 8, "cf32", 9, 128, 0),
                                                        (1024, 8, "ci8", 9000, 4, 1), (512, 8, "ci8", 30, 4, 1),
                                                        (512, 64, "ci16", 40, 64, 1)])
def test_forward_reports_a_timeout(ppf, C, T, in_dtype, S, family, ring):
    """The give-up path of each forward body, named by its kernel family: the generic
    kernel's ring, the row kernel with its ring, staged and direct, in whole and small
    batches, the carry kernel's one-barrier and short forms, the long-tap kernel's."""
    h = synth.design_taps(C, T)
    x = synth.stream(C, S + T - 1, in_dtype, SIGMA[in_dtype], 9550 + C)
    xd = torch.from_numpy(x).cuda()
    with ppf.Plan(C, T, h, in_dtype, "c64") as plan:
        v = plan.info()["variant"]
        assert v & (4 | 16 | 64 | 128) == family and v & 1 == ring
        plan.set_debug_flags(1)
        plan(xd)
        with pytest.raises(ppf.PPFError) as ei:
            plan.check_device()
        assert ei.value.status == 5
        plan.set_debug_flags(0)
        got = plan(xd).cpu().numpy()
        plan.check_device()
    idx = np.unique(np.linspace(0, S - 1, 40).astype(np.int64))
    assert oracle.rel_l2_max_per_spectrum(got[idx], oracle.pfb_spectra(x, h, C, T, idx)) <= 1e-5
