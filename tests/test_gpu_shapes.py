"""The launch shapes: what a handle says it uses, and what the autotuner's answer means."""
import numpy as np
import pytest

import lbm_workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("nx,ny", [(300, 70), (523, 2200), (4096, 1040)])
def test_tuned_shape_carries_over(precision, nx, ny):
    """The autotuner's answer, given to lbm_set_segment of another handle of the same channel, selects the
    shape that won: tiles, strips, or tiles where the rule takes strips (FP64 at 523 x 2200)."""
    from paper_2210_07501_gb300 import LBM_SEGMENT_TILES, Lbm
    w = WL.channel(nx, ny, 0.5 * ny, W=4.0, sigma1=1e-4)
    a, b = (Lbm(w["domain"], w["params"], precision=precision) for _ in range(2))
    rule = b.lbm_launch_shape()
    rows = a.lbm_autotune(2)
    won = a.lbm_launch_shape()
    b.lbm_set_segment(rows)
    assert b.lbm_launch_shape() == won
    assert rows == (won["rows"] if won["kind"] == "strips" else LBM_SEGMENT_TILES)
    b.lbm_set_segment(LBM_SEGMENT_TILES)
    assert b.lbm_launch_shape()["kind"] == "tiles"
    b.lbm_set_segment(13)
    assert b.lbm_launch_shape() == {"kind": "strips", "cols": 0, "rows": 13}
    b.lbm_set_segment(0)
    assert b.lbm_launch_shape() == rule
    a.close()
    b.close()


@pytest.mark.parametrize("precision,nx,ny,kind", [
    ("fp32", 200, 100, "tiles"), ("fp32", 4096, 1024, "tiles"), ("fp32", 4096, 1025, "strips"),
    ("fp64", 1024, 1024, "tiles"), ("fp64", 1024, 1025, "strips"), ("fp16", 4096, 1025, "tiles"),
    ("fp32", 3, 524300, "strips")])
def test_rule(precision, nx, ny, kind):
    """Tiles up to 2^22 nodes in FP32, 2^20 in FP64, of any number in FP16, and 65535 rows of tiles."""
    from paper_2210_07501_gb300 import Lbm
    w = WL.channel(nx, ny, 0.5 * ny, W=4.0, sigma1=1e-4)
    g = Lbm(w["domain"], w["params"], precision=precision)
    assert g.lbm_launch_shape()["kind"] == kind
    if ny > 65535 * 8:
        from paper_2210_07501_gb300 import LBM_SEGMENT_TILES
        g.lbm_set_segment(LBM_SEGMENT_TILES)
        assert g.lbm_launch_shape()["kind"] == "strips"
    g.close()


@pytest.mark.parametrize("args,kind", [(["--ny", "96"], None), (["--ny", "96", "--segment", "16"], "strips"),
                                       (["--ny", "96", "--precision", "fp16", "--segment", "16"], "strips")])
def test_bench_names_the_kernel_it_ran(args, kind):
    """The line of the benchmark names the kernel and launch shape in use, as the library reports them
    (kind None: whichever the autotuner took)."""
    import json
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "bench.py", "--steps", "4", "--warmup", "3", "--no-e2e", "--no-cpu-baseline"] + args,
                       cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    line = json.loads(r.stdout.strip().splitlines()[-1])
    kind = kind or line["config"]["launch"]["kind"]
    name = {"tiles": "lbm::tile_kernel", "strips": "lbm::march_kernel"}[kind]
    assert line["config"]["launch"]["kind"] == kind and line["roofline"]["kernel"].startswith(name)
    assert line["config"]["segment_rows"] == (line["config"]["launch"]["rows"] if kind == "strips" else None)
