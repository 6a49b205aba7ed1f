"""ppf_execute_batched over streams that lie any 16-byte multiple apart, not only
whole numbers of rows: every kernel family, short and long calls, streams of
less than a batch.  Each stream equals the same stream transformed alone, bit
for bit (the same kernel or one with the same arithmetic); the space between
the streams (NaN for FP32 input) is neither used nor written.
"""
import pytest

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


@pytest.mark.parametrize("S,ns", [(7, 3), (41, 40), (70, 300), (1, 200)])
@pytest.mark.parametrize("C,T,in_dtype,gap", [(64, 17, "cf32", 2), (64, 64, "ci8", 40), (128, 25, "ci16", 4),
                                              (256, 40, "ci8", 8), (512, 32, "cf32", 514), (512, 63, "ci16", 100),
                                              (512, 32, "ci8", 1024), (512, 8, "ci8", 8), (128, 16, "cf32", 6),
                                              (4096, 8, "ci8", 24), (3072, 3, "cf32", 2), (384, 20, "ci16", 12),
                                              (2048, 8, "cf32", 10), (32, 5, "ci8", 8)])
def test_streams_any_16_bytes_apart(ppf, C, T, in_dtype, gap, S, ns):
    n_in, n_out = C * (S + T - 1), C * S
    if ns * n_in > 1 << 25:
        pytest.skip("too large for a small test")
    h = synth.design_taps(C, T)
    x = torch.from_numpy(synth.stream(C, S + T - 1 + 8, in_dtype, SIGMA[in_dtype], 9400 + C + T)).cuda()
    in_stride, out_stride = n_in + gap, n_out + 6
    fill = float("nan") if in_dtype == "cf32" else 77
    xs = torch.full((ns, in_stride, 2), fill, dtype=x.dtype, device="cuda")
    for i in range(ns):
        xs[i, :n_in] = x[(i % 8) * C:(i % 8) * C + n_in]
    ys = torch.full((ns, out_stride, 2), -3.0, dtype=torch.float32, device="cuda")
    with ppf.Plan(C, T, h, in_dtype, "c64") as plan:
        ppf.check(ppf.lib().ppf_execute_batched(plan.handle, xs.data_ptr(), in_stride, ys.data_ptr(), out_stride, S, ns,
                                                torch.cuda.current_stream().cuda_stream))
        plan.check_device()
        for i in sorted({0, 1, 2, ns // 2, ns - 1}):
            alone = torch.view_as_real(plan(xs[i, :n_in].clone())).reshape(n_out, 2)
            assert torch.equal(ys[i, :n_out], alone), i
    assert bool((ys[:, n_out:] == -3.0).all())
