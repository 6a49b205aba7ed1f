"""The benchmark names the kernel that a plan's variant bits stand for."""
import importlib
import os
import sys
import types

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("variant,name", [(7, "pfb_fwd_carry_kernel"), (5, "pfb_fwd_carry_kernel"), (23, "pfb_fwd_cluster_kernel"),
                                          (67, "pfb_fwd_longtap_kernel"), (131, "pfb_fwd_row_kernel"),
                                          (130, "pfb_fwd_row_kernel"), (3, "pfb_fwd_kernel"), (1, "pfb_fwd_kernel")])
def test_kernel_name(variant, name):
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    bench = importlib.import_module("bench")
    w = types.SimpleNamespace(C=512, in_dtype="ci8", out_dtype="c64")
    assert bench.kernel_name(w, {"variant": variant, "tap_bucket": 8}) == f"{name}<512,8,ci8,c64>"
