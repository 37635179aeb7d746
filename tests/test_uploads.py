"""Data go to the device on the stream whose kernels read them.  A plain cudaMemcpy or cudaMemset runs
on the legacy default stream: a handle's non-blocking stream does not wait for it, and it may return
before pageable data (or a fill) has reached the device."""
import glob
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_copy_or_fill_on_the_default_stream():
    for path in glob.glob(os.path.join(ROOT, "paper_2210_07501_gb300", "csrc", "*.cu*")):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.findall(r"\bcudaMem(?:cpy|set)\w*\b(?<!Async)\s*\(", code), path


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("nx,ny", [(37, 9), (5, 20000)])
def test_created_state_is_the_default_state(precision, nx, ny):
    """The populations lbm_create leaves (from tables uploaded just before) are bit for bit those of
    lbm_init_fields with every default."""
    import lbm_workloads as WL
    from paper_2210_07501_gb300 import Lbm
    w = WL.channel(nx, ny, ny - 4.3, W=3.0, q_phi=9, q_T=5, sigma1=-3e-4, heat_periods=1)
    g = Lbm(w["domain"], w["params"], precision=precision)
    a = g.lbm_get_state()
    g.lbm_init_fields()
    b = g.lbm_get_state()
    g.close()
    for k in a:
        assert np.array_equal(a[k], b[k]), k
