"""Compile-time refusals of the device code: forms that would hang or corrupt must not
compile.  Only the compiler's front end runs (no GPU).
"""
import subprocess

import pytest

from paper_1511_03599_gb300 import _build


def _front_end(tmp_path, body):
    try:
        nvcc = _build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src = tmp_path / "check.cu"
    src.write_text('#include "ppf_fwd.cuh"\n' + body)
    return subprocess.run([nvcc] + _build._flags() + ["-cuda", str(src), "-o", str(tmp_path / "check.ii")],
                          capture_output=True, text=True, timeout=300)


KERNEL = """
__global__ void k(ppf::FwdArgs a, unsigned char* smem) {{
    ppf::carry_range<512, {tm}, ppf::IN_CI8, ppf::OUT_CF32, false, {grp}, true>(a, a.in, a.out, 0, 1, smem);
}}
"""


def test_one_barrier_carry_form_needs_the_whole_cta(tmp_path):
    """At C = 512 with few int8 taps the carry body synchronises with CTA-wide barriers: a
    half-CTA group, whose other half runs tiles of its own, must not run it."""
    bad = _front_end(tmp_path, KERNEL.format(tm=4, grp="ppf::HalfGroup<256>"))
    assert bad.returncode != 0 and "synchronises the whole CTA" in bad.stderr
    for tm, grp in ((4, "ppf::CtaGroup"), (8, "ppf::HalfGroup<256>")):
        good = _front_end(tmp_path, KERNEL.format(tm=tm, grp=grp))
        assert good.returncode == 0, good.stderr[-2000:]
