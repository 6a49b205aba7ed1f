"""The three-pass adjoint's second pass at the ends of a stream, where only some
taps meet a row of it: streams shorter than a tile of 16 raw rows, than the taps
and around both, one or many, against the FP64 oracle (relative L2 1e-5 for the
input gradient, 1e-4 for the tap gradient); and an inf or NaN sample of FP32 input
reaches the tap gradients of its channel that read it and no others.
"""
import numpy as np
import pytest

import oracle
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


SIZES = [(S, T) for T in (17, 24, 63, 64) for S in (1, 2, 9, 15, 16, 17, 33, 64, 65, 100)]


@pytest.mark.parametrize("C,in_dtype", [(64, "cf32"), (128, "ci8"), (32, "ci16"), (384, "cf32")])
def test_short_streams(ppf, C, in_dtype):
    rng = np.random.default_rng(C)
    for S, T in SIZES:
        ns = 3
        h = synth.design_taps(C, T)
        x = np.stack([synth.stream(C, S + T - 1, in_dtype, {"cf32": 1.0}.get(in_dtype, 16.0), 9600 + i) for i in range(ns)])
        G = (rng.standard_normal((ns, S, C)) + 1j * rng.standard_normal((ns, S, C))).astype(np.complex64)
        with ppf.Plan(C, T, h, in_dtype, "c64") as plan:
            gx, gh = plan.backward(torch.from_numpy(G).cuda(), torch.from_numpy(x).cuda())
            plan.check_device()
        Gn = G.astype(np.complex128)
        ref_x = np.stack([oracle.pfb_grad_input(Gn[i], h, C, T).reshape(-1) for i in range(ns)])
        ref_h = sum(oracle.pfb_grad_taps(Gn[i], x[i], C, T).reshape(-1) for i in range(ns))
        assert oracle.rel_l2(gx.cpu().numpy().reshape(ns, -1), ref_x) <= 1e-5, (S, T)
        assert oracle.rel_l2(gh.cpu().numpy(), ref_h) <= 1e-4, (S, T)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("C,T,S", [(64, 17, 5), (64, 40, 9), (128, 64, 70), (32, 33, 33)])
def test_non_finite_sample_at_the_ends(ppf, C, T, S, bad):
    rng = np.random.default_rng(S)
    G = (rng.standard_normal((S, C)) + 1j * rng.standard_normal((S, C))).astype(np.complex64)
    with ppf.Plan(C, T, synth.design_taps(C, T), "cf32", "c64") as plan:
        for r in (0, 1, T // 2, S + T - 3, S + T - 2):
            x = synth.stream(C, S + T - 1, "cf32", 1.0, 9700)
            c = C // 3
            x[r * C + c, 1] = bad
            gx, gh = plan.backward(torch.from_numpy(G).cuda(), torch.from_numpy(x).cuda())
            plan.check_device()
            finite = torch.isfinite(gh).reshape(T, C).cpu()
            want = torch.ones((T, C), dtype=torch.bool)
            for t in range(T):
                if 0 <= r - t < S:
                    want[t, c] = False
            assert torch.equal(finite, want), r
            assert bool(torch.isfinite(torch.view_as_real(gx)).all())


@pytest.mark.parametrize("C,T,S,ns", [(384, 4, 9, 300), (1024, 1, 3, 500), (512, 24, 5, 200), (32, 2, 7, 900)])
def test_many_short_streams(ppf, C, T, S, ns):
    """One inverse DFT over the rows of all streams: each stream's input gradient is, bit
    for bit, the one of the stream alone, and the tap gradient the sum over the streams."""
    rng = np.random.default_rng(C + ns)
    h = synth.design_taps(C, T)
    x = rng.integers(-50, 50, (ns, C * (S + T - 1), 2), dtype=np.int8)
    G = (rng.standard_normal((ns, S, C)) + 1j * rng.standard_normal((ns, S, C))).astype(np.complex64)
    xd, Gd = torch.from_numpy(x).cuda(), torch.from_numpy(G).cuda()
    with ppf.Plan(C, T, h, "ci8", "c64") as plan:
        gx, gh = plan.backward(Gd, xd)
        for i in (0, 1, ns // 2, ns - 1):
            alone, _ = plan.backward(Gd[i].clone(), xd[i].clone())
            assert torch.equal(torch.view_as_real(gx[i]), torch.view_as_real(alone)), i
        plan.check_device()
    ref = sum(oracle.pfb_grad_taps(G[i].astype(np.complex128), x[i], C, T) for i in range(ns))
    assert oracle.rel_l2(gh.cpu().numpy(), ref.reshape(-1)) <= 1e-4
