"""The two launch shapes of the step, 2-D tiles and row-marching strips, give the same bits: the
arithmetic of a node and its order are shared.  Sizes at the edges of the tiles (32 x 8 in FP32
arithmetic), of the strips (128 columns) and of the domain's minimum, every lattice pair."""
import numpy as np
import pytest

import lbm_workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("qf,qt", [(5, 5), (5, 9), (9, 5), (9, 9)])
@pytest.mark.parametrize("nx,ny", [(3, 3), (31, 7), (32, 8), (33, 9), (130, 17), (200, 41)])
def test_tiles_equal_marching_strips(precision, qf, qt, nx, ny):
    from paper_2210_07501_gb300 import Lbm
    w = WL.channel(nx, ny, 0.45 * ny, W=3.0, q_phi=qf, q_T=qt, sigma0=2e-3, sigma1=-3e-4, sigma2=5e-4, T_hot=1.2,
                   T_cold=0.9, dT=0.6, heat_periods=2, tau_flow=0.9, visc_ratio=1.7, tau_T=1.1, cond_ratio=0.6,
                   tau_phi=0.75, rho_top=1.3, Fx_ext=2e-7, Fy_ext=-1e-7)
    r = WL.random_fields(nx, ny, seed=nx + ny)
    y = np.arange(ny)[:, None] + 0.5
    phi = np.clip(0.5 + 0.5 * np.tanh(2 * (y - w["domain"]["b"]) / 3.0) + 0.2 * r["phi_pert"], 0.0, 1.0)
    got = []
    for rows in (0, 8):                 # 0: the rule's choice, tiles at these sizes; else the march
        g = Lbm(w["domain"], w["params"], precision=precision)
        g.lbm_init_fields(phi=phi, u=r["u"] * 0.05, v=r["v"] * 0.05, T=1.0 + r["T_pert"], dp=r["dp"] * 0.1)
        g.lbm_set_segment(rows)
        g.lbm_step(12)
        got.append({**g.lbm_fields(), **{"state " + k: v for k, v in g.lbm_get_state().items()}})
        g.close()
    for k in got[0]:
        assert np.array_equal(got[0][k], got[1][k]), k


def test_more_tile_rows_than_a_grid_has():
    """A channel of more than 65535 rows of tiles, the most a grid has: the rule takes the march."""
    from paper_2210_07501_gb300 import Lbm
    w = WL.channel(3, 524300, 524290.0, W=3.0, sigma1=-3e-4, heat_periods=1)
    got = []
    for rows in (0, 64):
        g = Lbm(w["domain"], w["params"], precision="fp32")
        g.lbm_set_segment(rows)
        if rows == 0:
            assert g.lbm_autotune(1) > 0
        g.lbm_step(3)
        got.append(g.lbm_fields())
        g.close()
    for k in got[0]:
        assert np.array_equal(got[0][k], got[1][k]), k


@pytest.mark.parametrize("precision,n", [("fp32", 32), ("fp32", 33), ("fp64", 1), ("fp64", 33), ("fp16", 32)])
def test_batches_of_any_number_equal_single_channels(precision, n):
    """Batches of up to 32 channels carry their arguments in the launch's parameters, larger ones read
    them from device memory; on tiles (the rule's choice at these sizes) and after tuning, every
    channel has the bits of a handle of its own."""
    from paper_2210_07501_gb300 import Lbm, LbmBatch
    rng = np.random.Generator(np.random.PCG64(n))
    ws = [WL.channel(int(rng.choice([33, 64, 130])), int(rng.choice([9, 16, 25])), 5.0, W=3.0,
                     sigma1=float(rng.uniform(-2e-4, 2e-4)), sigma2=-2e-3, visc_ratio=float(rng.uniform(0.5, 2.0)))
          for _ in range(n)]
    b = LbmBatch(ws, precision=precision)
    b.lbm_batch_set_check_interval(10)
    b.lbm_batch_step(10)
    b.lbm_batch_autotune(1)
    b.lbm_batch_step(20)
    for c, w in enumerate(ws):
        g = Lbm(w["domain"], w["params"], precision=precision)
        g.lbm_set_check_interval(10)
        g.lbm_step(30)
        a, r = b.lbm_batch_fields(c), g.lbm_fields()
        for k in a:
            assert np.array_equal(a[k], r[k]), (c, k)
        assert b.lbm_batch_diag(c)["residual"] == g.lbm_diag()["residual"]
        g.close()
    b.close()
