"""The largest channel: a population plane of less than 4 GiB, since the kernels' offsets inside a
plane are unsigned 32-bit bytes (a larger plane, which fits this GPU's memory in FP64 and FP32, would
wrap onto itself and give wrong fields).  Checked on the host, before any allocation."""
import ctypes
import os

import pytest

import lbm_workloads as WL

SIZES = {"fp64": 8, "fp32": 4, "fp16": 2}


def create(precision, nx, ny):
    import paper_2210_07501_gb300 as pkg
    pkg.build()
    lib = pkg.load()
    w = WL.channel(nx, ny, 10.0, W=3.0)
    d, p = pkg.make_domain(w["domain"], precision), pkg.make_params(w["params"])
    h = ctypes.c_void_p()
    rc = lib.lbm_create(ctypes.byref(d), ctypes.byref(p), None, ctypes.byref(h))
    one = lib.lbm_batch_create(1, ctypes.byref(d), ctypes.byref(p), None, ctypes.byref(h))
    return rc, one, pkg


@pytest.mark.parametrize("precision", list(SIZES))
@pytest.mark.parametrize("nx", [64, 8192, 8129])
def test_plane_of_4_gib_is_refused(precision, nx):
    rc, one, pkg = create(precision, nx, (1 << 32) // SIZES[precision] // ((nx + 63) // 64 * 64))
    assert rc == one == pkg.LBM_EINVAL


@pytest.mark.skipif(os.path.exists("/dev/nvidiactl"), reason="would allocate the channel")
@pytest.mark.parametrize("precision", list(SIZES))
@pytest.mark.parametrize("nx", [64, 8192, 8129])
def test_one_row_less_is_not(precision, nx):
    rc, one, pkg = create(precision, nx, (1 << 32) // SIZES[precision] // ((nx + 63) // 64 * 64) - 1)
    assert rc == one == pkg.LBM_ECUDA      # accepted; there is no device to create it on
