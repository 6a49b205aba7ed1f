"""How a beam set is cut into tiles, and the bodies of its wide beams on tiles of any
size: every beam at C >= 1024 equals ppf_execute bit for bit, whatever the tiles (one
batch, a few, the plan's own), with ragged counts and tap counts below their bucket.
Equal beams that fill the SMs evenly stay whole; a beam alone is spread over at least
half of them (tile sizes go in powers of two).
"""
import numpy as np
import pytest

from paper_1511_03599_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mods():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_03599_gb300 import beams, ppf
    ppf.lib()
    return beams, ppf


def _set(beams, defs, seed=9800):
    h = [synth.design_taps(C, T) for C, T, _ in defs]
    xs = [torch.from_numpy(synth.stream(C, S + T - 1, "ci8", 16.0, seed + i)).cuda() for i, (C, T, S) in enumerate(defs)]
    ys = [torch.empty((S, C), dtype=torch.complex64, device="cuda") for C, _, S in defs]
    bs = beams.BeamSet([d[0] for d in defs], [d[1] for d in defs], [d[2] for d in defs], h)
    bs.bind(xs, ys)
    return bs, h, xs, ys


@pytest.mark.parametrize("tile_samples", [None, 1 << 13, 3 << 14, 5 << 15, 1 << 20])
def test_wide_beams_equal_execute_on_any_tiles(mods, tile_samples):
    beams, ppf = mods
    defs = [(1024, 3, 1), (1024, 8, 333), (1024, 4, 64), (1024, 9, 17), (1024, 16, 500), (2048, 8, 201), (2048, 13, 77),
            (4096, 16, 50), (4096, 5, 103), (512, 8, 700)]
    bs, h, xs, ys = _set(beams, defs)
    if tile_samples:
        bs.set_tiling(tile_samples)
    for y in ys:
        y.fill_(float("nan"))
    bs.execute()
    bs.check_device()
    for (C, T, _), hi, x, y in zip(defs, h, xs, ys):
        with ppf.Plan(C, T, hi, "ci8", "c64") as plan:
            want = plan(x)
        if C >= 1024:
            assert torch.equal(torch.view_as_real(y), torch.view_as_real(want)), (C, T)
        else:
            assert float((y - want).abs().norm() / want.abs().norm()) <= 2e-6
    bs.close()


def test_even_sets_stay_whole_and_single_beams_are_spread(mods):
    beams, _ = mods
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for C in (64, 1024):
        n = 4 * sms
        bs = beams.BeamSet([C] * n, [4] * n, [(1 << 16) // C] * n, [np.ones(C * 4, np.float32)] * n)
        assert bs.info()["tiles"] == n
        bs.close()
        bs = beams.BeamSet([C], [4], [(1 << 24) // C], [np.ones(C * 4, np.float32)])
        assert bs.info()["tiles"] >= sms // 2
        bs.close()
