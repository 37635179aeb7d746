"""One handle per host thread: what the handles share (function attributes of the kernels) is set
once per device and never changed under another thread's launch."""
import os
import subprocess
import threading

import numpy as np
import pytest

import lbm_workloads as WL

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <stdio.h>
#include <thread>
#include <vector>
#include "lbm_once.h"
int main()
{
    static lbm::OncePerDevice once;
    std::atomic<int> calls[70], early{0};
    bool ready[70] = {};
    for (auto &c : calls) c = 0;
    std::vector<std::thread> t;
    for (int k = 0; k < 16; ++k)
        t.emplace_back([&] {
            for (int d = 0; d < 64; ++d) {
                once.run(d, [&] { std::this_thread::yield(); ready[d] = true; ++calls[d]; return 0; });
                if (!ready[d]) ++early;
            }
        });
    for (auto &x : t) x.join();
    int wrong = early;
    for (int d = 0; d < 64; ++d) wrong += calls[d] != 1;
    // an error is returned and the next call tries again; a device past the mask is set up each time
    lbm::OncePerDevice other;
    wrong += other.run(3, [] { return 7; }) != 7;
    int n = 0;
    wrong += other.run(3, [&] { ++n; return 0; }) != 0 || other.run(3, [&] { ++n; return 0; }) != 0 || n != 1;
    wrong += other.run(69, [&] { ++n; return 0; }) != 0 || other.run(69, [&] { ++n; return 0; }) != 0 || n != 3;
    printf("%d\n", wrong);
    return wrong;
}
"""


def test_set_up_once_on_every_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2210_07501_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", csrc, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, timeout=60).stdout.strip() == "0"


def test_kernel_attributes_are_set_once_on_every_device():
    """Attributes hold on one device: a flag per process left the kernels of the second device without
    their shared memory, and nothing ordered a second thread's launch after the settings."""
    for name in ("lbm_step.cu", "lbm_tile.cu"):
        code = open(os.path.join(ROOT, "paper_2210_07501_gb300", "csrc", name)).read()
        assert "cudaFuncSetAttribute" in code and "OncePerDevice" in code and "static bool" not in code, name


def test_no_unordered_first_use():
    """A plain static flag orders nothing: a second thread may see it set and the data behind it not (the
    checksum table of checkpoints had one)."""
    csrc = os.path.join(ROOT, "paper_2210_07501_gb300", "csrc")
    for name in sorted(os.listdir(csrc)):
        assert "static bool" not in open(os.path.join(csrc, name)).read().replace("static bool aligned_rows(", ""), name


@pytest.mark.gpu
def test_two_threads_step_channels_of_different_size():
    """FP64 tiles ask for shared memory by the channel's size.  Two handles of one lattice pair, each
    stepped by its own thread, give the bits they give one after the other."""
    from paper_2210_07501_gb300 import Lbm
    ws = [WL.channel(nx, ny, 0.5 * ny, W=5.0, q_phi=9, q_T=9, sigma1=-1e-4) for nx, ny in ((200, 100), (160, 320))]

    def make():
        return [Lbm(w["domain"], w["params"], precision="fp64") for w in ws]

    def run(g, errors):
        try:
            for _ in range(20):
                g.lbm_step(100)
        except Exception as e:
            errors.append(e)

    errors, together, alone = [], make(), make()
    threads = [threading.Thread(target=run, args=(g, errors)) for g in together]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for g, a in zip(together, alone):
        run(a, errors)
        x, y = g.lbm_fields(), a.lbm_fields()
        for k in x:
            assert np.array_equal(x[k], y[k]), k
        g.close()
        a.close()
    assert not errors, errors
