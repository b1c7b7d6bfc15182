"""gpz_compress_f64 rejects every invalid argument before anything is enqueued,
whichever of its two forms the data would then take."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def gpz():
    from paper_2508_10305_gb300 import build
    build.build()
    from paper_2508_10305_gb300 import gpz as m
    return m


@pytest.mark.parametrize("change", [
    {"params": None}, {"seg_bits": 4}, {"seg_bits": -1}, {"mode": 2}, {"eb": 0.0}, {"eb": float("inf")},
    {"out": None}, {"out": (1 << 20) + 2}, {"perm": (1 << 28) + 2}, {"fields": (4096, 8196, 12288)},
    {"fields": None}, {"ws": None}, {"ws": (1 << 24) + 64},
], ids=str)
def test_f64_argument_errors_need_no_device(gpz, change):
    n = 1000
    p = gpz.make_params(3, change.get("eb", 1e-9), change.get("mode", gpz.EB_ABS), change.get("seg_bits", 3))
    fields = change.get("fields", (4096, 8192, 12288))
    status = gpz.lib.gpz_compress_f64(
        (C.c_void_p * 3)(*fields) if fields else None, n, C.byref(p) if "params" not in change else None,
        C.c_void_p(change.get("out", 1 << 20)), gpz.gpz_bound_size_wide(n, 3), None, None,
        C.c_void_p(change.get("perm", None)), C.c_void_p(change.get("ws", 1 << 24)),
        int(gpz.lib.gpz_compress_f64_workspace_size(n, 3)), None, None)
    assert status == gpz.ERR_INVALID_ARG
