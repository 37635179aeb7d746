"""A state put into a handle whose step gave up waiting for its copies (the test hook of
test_gpu_fault.py: bounded waits, no GPU fault) makes it usable again."""
import numpy as np
import pytest

import lbm_workloads as WL

pytestmark = pytest.mark.gpu


def test_set_state_clears_the_fault():
    from paper_2210_07501_gb300 import LBM_EDEVICE, Lbm, LbmError
    w = WL.channel(64, 32, 16, W=4.0)            # one strip, one segment: one CTA
    ref, g = (Lbm(w["domain"], w["params"], precision="fp64") for _ in range(2))
    ref.lbm_step(5)
    state = ref.lbm_get_state()
    g.lbm_test_stall_copies(True)
    g.lbm_step(1)
    with pytest.raises(LbmError) as e:
        g.lbm_fields()
    assert e.value.status == LBM_EDEVICE
    g.lbm_test_stall_copies(False)
    g.lbm_set_state(state)
    ref.lbm_set_state(state)
    g.lbm_step(20)
    ref.lbm_step(20)
    a, b = g.lbm_fields(), ref.lbm_fields()
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    g.close()
    ref.close()
