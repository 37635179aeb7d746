"""Batches on either launch shape, below and above the 32 channels whose arguments travel in the launch's
parameters, against single channels; and the march's own edges, on channels that the rule steps on
tiles."""
import numpy as np
import pytest

import lbm_workloads as WL
from paper_2210_07501_gb300 import LBM_SEGMENT_TILES

pytestmark = pytest.mark.gpu
FIELDS = ("phi", "u", "v", "T", "dp")


def start(w, seed, u_amp=0.05):
    nx, ny = w["domain"]["nx"], w["domain"]["ny"]
    r = WL.random_fields(nx, ny, seed=seed)
    y = np.arange(ny)[:, None] + 0.5
    phi = np.clip(0.5 + 0.5 * np.tanh(2 * (y - w["domain"]["b"]) / w["domain"]["W"]) + 0.2 * r["phi_pert"], 0.0, 1.0)
    return dict(phi=phi, u=r["u"] * u_amp, v=r["v"] * u_amp, T=1.0 + r["T_pert"], dp=r["dp"] * 0.1)


@pytest.mark.parametrize("rows,kind", [(8, "strips"), (32, "strips"), (LBM_SEGMENT_TILES, "tiles")])
@pytest.mark.parametrize("precision,n", [("fp32", 32), ("fp32", 33), ("fp64", 32), ("fp64", 33), ("fp16", 32), ("fp16", 33)])
def test_batch_of_either_shape_equals_single_channels(precision, n, rows, kind):
    """Two of the channels start on the profile that their body force drives, so they converge at the second
    check and drop out while the others go on: every channel has the bits of a handle of its own,
    at the step where it stopped."""
    from paper_2210_07501_gb300 import Lbm, LbmBatch
    rng = np.random.Generator(np.random.PCG64(n))
    ws = [WL.channel(int(rng.choice([33, 64, 130, 257])), int(rng.choice([9, 16, 25, 67])), 5.0, W=3.0,
                     sigma1=float(rng.uniform(-2e-4, 2e-4)), sigma2=-2e-3, visc_ratio=float(rng.uniform(0.5, 2.0)))
          for _ in range(n)]
    still = (1, n - 1)
    for c in still:
        ws[c] = WL.channel(130, 67, 33.0, W=3.0, sigma0=0.0, sigma1=0.0, sigma2=0.0, dT=0.0, tau_flow=0.8,
                           Fx_ext=8 * 0.1 * 0.02 / 67 ** 2)
    b = LbmBatch(ws, precision=precision)
    b.lbm_batch_set_check_interval(10)
    b.lbm_batch_set_segment(rows)
    shape = b.lbm_batch_launch_shape()
    assert shape["kind"] == kind and (kind == "tiles" or shape["rows"] == rows)
    y = (np.arange(67)[:, None] + 0.5) / 67 * np.ones((1, 130))
    drift = dict(u=4 * 0.02 * y * (1 - y))
    for c in still:
        b.lbm_batch_init_fields(c, **drift)
    steps, _ = b.lbm_batch_run_to_steady(5e-3, 60)
    assert [s for c, s in enumerate(steps) if c in still] == [20, 20]
    assert all(s == 60 for c, s in enumerate(steps) if c not in still)
    for c, w in enumerate(ws):
        g = Lbm(w["domain"], w["params"], precision=precision)
        g.lbm_set_check_interval(10)
        if c in still:
            g.lbm_init_fields(**drift)
        g.lbm_step(steps[c])
        a, r = b.lbm_batch_fields(c), g.lbm_fields()
        for k in FIELDS:
            assert np.array_equal(a[k], r[k]), (c, k)
        assert b.lbm_batch_diag(c)["residual"] == g.lbm_diag()["residual"]
        g.close()
    b.close()


def test_batch_shapes_of_the_rule():
    """Tiles while the channels together have up to 2^20 nodes in FP64, then strips; a batch steps on after
    its shape was changed, and the autotuner's answer names what it keeps."""
    from paper_2210_07501_gb300 import LbmBatch
    for n, kind in ((4, "tiles"), (5, "strips")):
        b = LbmBatch([WL.channel(512, 512, 256.0, W=4.0, sigma1=1e-4)] * n, precision="fp64")
        b.lbm_batch_set_check_interval(2)
        rule = b.lbm_batch_launch_shape()
        assert rule["kind"] == kind
        b.lbm_batch_step(2)
        rows = b.lbm_batch_autotune(1)
        won = b.lbm_batch_launch_shape()
        b.lbm_batch_set_segment(0)
        assert b.lbm_batch_launch_shape() == rule
        b.lbm_batch_set_segment(rows)
        assert b.lbm_batch_launch_shape() == won
        b.lbm_batch_step(2)
        assert b.lbm_batch_diag(0)["steps"] == 4
        b.lbm_batch_set_segment(LBM_SEGMENT_TILES - 1)     # one segment a strip
        assert b.lbm_batch_launch_shape() == {"kind": "strips", "cols": 0, "rows": 512}
        assert b.lbm_batch_size()["ctas"] == n * 512 // 128
        b.lbm_batch_step(2)
        b.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("nx,ny", [(33, 9), (37, 23), (130, 23), (257, 67)])
def test_tiles_and_strips_by_name(precision, nx, ny):
    """Each shape asked for by name and confirmed: the same bits."""
    from paper_2210_07501_gb300 import Lbm
    w = WL.channel(nx, ny, 0.45 * ny, W=3.0, q_phi=9, q_T=5, sigma0=2e-3, sigma1=-3e-4, sigma2=5e-4, T_hot=1.2,
                   T_cold=0.9, dT=0.6, heat_periods=2, tau_flow=0.9, visc_ratio=1.7, tau_T=1.1, cond_ratio=0.6,
                   tau_phi=0.75, rho_top=1.3, Fx_ext=2e-7)
    got = []
    for rows, kind in ((LBM_SEGMENT_TILES, "tiles"), (8, "strips"), (64, "strips")):
        g = Lbm(w["domain"], w["params"], precision=precision)
        g.lbm_init_fields(**start(w, nx + ny))
        g.lbm_set_segment(rows)
        assert g.lbm_launch_shape()["kind"] == kind
        g.lbm_step(12)
        got.append({**g.lbm_fields(), **{"state " + k: v for k, v in g.lbm_get_state().items()}})
        g.close()
    for o in got[1:]:
        for k in o:
            assert np.array_equal(o[k], got[0][k]), k


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("nx", [37, 130])
def test_reduced_precision_odd_and_ragged_widths_in_strips(precision, nx):
    """As the parity test of the same widths, on marching strips: the staged rows' last columns and
    the periodic wrap are copied element by element, and with nx = 130 the second strip holds only
    two columns.  Its bars."""
    import os

    import oracle
    from paper_2210_07501_gb300 import Lbm
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    w = WL.channel(nx, 23, 11.3, W=3.0, q_phi=9, q_T=5, sigma0=2e-3, sigma1=-3e-4, sigma2=5e-4,
                   T_hot=1.2, T_cold=0.9, dT=0.6, heat_periods=2, tau_flow=0.9, visc_ratio=1.7,
                   tau_T=1.1, cond_ratio=0.6, tau_phi=0.75)
    from test_gpu_parity import random_init
    init = random_init(w, seed=41 + nx)
    g, ref = Lbm(w["domain"], w["params"], precision=precision), oracle.Oracle(w["domain"], w["params"])
    g.lbm_init_fields(**init)
    g.lbm_set_segment(8)
    assert g.lbm_launch_shape()["kind"] == "strips"
    g.lbm_step(300)
    ref.init(**init)
    ref.step(300)
    a, b = g.lbm_fields(), ref.fields()
    g.close()
    ref.close()
    umax = max(np.max(np.abs(b["u"])), np.max(np.abs(b["v"])))
    bars = {"fp32": {"u": 5e-5, "v": 5e-5, "phi": 1e-4, "T": 3e-6},
            "fp16": {"u": 0.1, "v": 0.1, "phi": 3e-2, "T": 3e-3}}[precision]
    for k, bar in bars.items():
        e = np.max(np.abs(a[k] - b[k])) / (umax if k in ("u", "v") else 1.0)
        assert e <= bar, (k, e)
