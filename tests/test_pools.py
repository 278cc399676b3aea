"""The memory pools of work areas: which pool a call allocates from.
The bookkeeping (csrc/efm_pool.h) runs on the host over a fake of the CUDA
calls; on the GPU, a process resets its own context between two searches."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1804_02867_gb300", "csrc")


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("pool") / "pool_driver")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, os.path.join(ROOT, "tests", "host", "pool_driver.cpp"), "-o", exe],
                   check=True)

    def run(*cmds):
        out = subprocess.run([exe], input="\n".join(cmds) + "\n", capture_output=True, text=True, check=True).stdout
        return out.splitlines()

    return run


def test_a_context_keeps_its_pool(driver):
    assert driver("ctx 7", "get", "get", "ctx 8", "get", "ctx 7", "get") == [
        "ok", "pool 1", "pool 1", "ok", "pool 2", "ok", "pool 1"]


def test_a_reset_device_gets_a_new_pool(driver):
    # the same device, a new context: the old handle is not used again
    assert driver("ctx 1", "get", "ctx 2", "get") == ["ok", "pool 1", "ok", "pool 2"]


def test_without_a_pool_the_default_one_serves(driver):
    assert driver("ctx 0", "get") == ["ok", "pool 0"]
    # (a context whose pool could not be made is not asked for one again)
    assert driver("ctx 3", "fail 1", "get", "fail 0", "get") == ["ok", "ok", "pool 0", "ok", "pool 0"]
    many = [f"ctx {i}\nget" for i in range(1, 66)]
    assert driver(*many)[1::2] == [f"pool {i}" for i in range(1, 65)] + ["pool 0"]


RESET_SCRIPT = """
import ctypes
import numpy as np
from paper_1804_02867_gb300 import efmgraph, synth
net = synth.core()
def run():
    w = efmgraph.Network(net, 0)
    sampled = efmgraph.sample_target(w, net.targets[4], 20, 2, 7, 1 << 12)  # before any traversal
    return w, [sampled] + efmgraph.enumerate_targets(w, net.targets[:2], 20, 2, 0, 1 << 14)
w, want = run()
cu, dev = ctypes.CDLL("libcuda.so.1"), ctypes.c_int()
assert cu.cuInit(0) == 0 and cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
assert cu.cuDevicePrimaryCtxReset(dev) == 0  # this process's own context; nothing is in flight
for _ in range(2):
    w, got = run()
    w.close()
    assert len(want[0][0]) > 0  # the walks' minimality test ran
    assert all(np.array_equal(a[0], b[0]) and a[1] == b[1] for a, b in zip(want, got))
print("same")
"""


@pytest.mark.gpu
def test_work_areas_after_a_context_reset():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02867_gb300 import build

    build.build()
    out = subprocess.run([sys.executable, "-c", RESET_SCRIPT], capture_output=True, text=True, cwd=ROOT)
    assert out.stdout.strip() == "same", out.stderr[-2000:]
