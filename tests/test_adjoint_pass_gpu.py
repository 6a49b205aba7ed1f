"""The adjoint's one-pass gradient kernel (both sums over g_y) at the sizes where
it can go wrong: tap counts around its blocks of 8 and tiles of 16 rows,
streams shorter than the filter, many streams, every block width (C = 32, 64
and multiples of 128), each sum asked for alone.  Tolerances as for the other
adjoint paths: relative L2 <= 1e-5 for grad_x, <= 1e-4 for grad_h, against the
FP64 oracle.
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


@pytest.mark.parametrize("C,T,S,ns,in_dtype", [(32, 1, 50, 1, "cf32"), (32, 9, 700, 3, "ci8"), (64, 17, 1, 4, "ci16"),
                                               (64, 64, 333, 2, "cf32"), (128, 24, 5000, 1, "ci8"), (384, 8, 40, 1, "cf32"),
                                               (512, 16, 17, 300, "ci8"), (512, 25, 90, 2, "cf32"), (768, 2, 31, 3, "ci16"),
                                               (1024, 7, 2000, 1, "cf32"), (2048, 40, 100, 1, "ci8"), (4096, 8, 64, 2, "cf32")])
def test_matches_oracle_and_single_sums(ppf, C, T, S, ns, in_dtype):
    rng = np.random.default_rng(C + T + S + ns)
    h = synth.design_taps(C, T) + 0.01 * rng.standard_normal(C * T).astype(np.float32)
    x = np.stack([synth.stream(C, S + T - 1, in_dtype, SIGMA[in_dtype], 9300 + i) for i in range(ns)])
    G = (rng.standard_normal((ns, S, C)) + 1j * rng.standard_normal((ns, S, C))).astype(np.complex64)
    xd, Gd = torch.from_numpy(x).cuda(), torch.from_numpy(G).cuda()
    with ppf.Plan(C, T, h, in_dtype, "c64") as plan:
        gx, gh = plan.backward(Gd, xd)
        again, _ = plan.backward(Gd, xd, want_taps=False)
        _, gh2 = plan.backward(Gd, xd, want_input=False)
        plan.check_device()
    assert torch.equal(torch.view_as_real(gx), torch.view_as_real(again)) and torch.equal(gh, gh2)
    few = range(ns) if ns <= 4 else (0, ns // 2, ns - 1)
    gx = gx.reshape(ns, -1).cpu().numpy()
    for i in few:
        assert oracle.rel_l2(gx[i], oracle.pfb_grad_input(G[i].astype(np.complex128), h, C, T)) <= 1e-5
    want = sum(oracle.pfb_grad_taps(G[i].astype(np.complex128), x[i], C, T) for i in range(ns))
    assert oracle.rel_l2(gh.cpu().numpy().astype(np.float64), want) <= 1e-4


@pytest.mark.parametrize("C,T,S", [(512, 20, 100), (1024, 8, 40)])
def test_non_finite_sample_reaches_only_its_taps(ppf, C, T, S):
    """x[r] enters grad_h[t] only where 0 <= r - t < S: an inf in the first (last) raw
    row reaches tap 0 (T-1) of its channel and no other element."""
    rng = np.random.default_rng(5)
    G = torch.from_numpy((rng.standard_normal((S, C)) + 1j * rng.standard_normal((S, C))).astype(np.complex64)).cuda()
    for row, tap in ((0, 0), (S + T - 2, T - 1)):
        x = synth.stream(C, S + T - 1, "cf32", 1.0, 9400)
        x[row * C + 5, 0] = np.inf
        with ppf.Plan(C, T, synth.design_taps(C, T), "cf32", "c64") as plan:
            _, gh = plan.backward(G, torch.from_numpy(x).cuda())
        bad = (~torch.isfinite(gh)).nonzero().reshape(-1).tolist()
        assert bad == [tap * C + 5]
