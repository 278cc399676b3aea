"""The memory pools of work areas: which pool a call allocates from and when it
gives memory back.  The bookkeeping (csrc/efm_pool.h) runs on the host over a
fake of the CUDA calls; on the GPU, free memory is compared before a network
is loaded and after the last one is freed."""
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
    # the same device, a new context: the old handle is not used again, nor
    # trimmed when a network of the old context is freed
    assert driver("ctx 1", "retain", "get", "ctx 2", "get", "release 1", "retain", "release 2") == [
        "ok", "id 1", "pool 1", "ok", "pool 2", "trims", "id 2", "trims 2"]


def test_the_last_network_gives_the_memory_back(driver):
    assert driver("ctx 5", "retain", "retain", "get", "release 5", "release 5", "get") == [
        "ok", "id 5", "id 5", "pool 1", "trims", "trims 1", "pool 1"]
    # no pool was used: nothing to give back
    assert driver("ctx 5", "retain", "release 5") == ["ok", "id 5", "trims"]


def test_without_a_pool_the_default_one_serves(driver):
    assert driver("ctx 0", "get", "retain", "release 0") == ["ok", "pool 0", "id 0", "trims"]
    # (a context whose pool could not be made is not asked for one again)
    assert driver("ctx 3", "fail 1", "get", "fail 0", "get", "retain", "release 3") == [
        "ok", "ok", "pool 0", "ok", "pool 0", "id 3", "trims"]
    many = [f"ctx {i}\nget" for i in range(1, 66)]
    assert driver(*many)[1::2] == [f"pool {i}" for i in range(1, 65)] + ["pool 0"]


GPU_SCRIPT = """
import torch
from paper_1804_02867_gb300 import efmgraph, synth
torch.zeros(1, device="cuda")
def used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free
net = synth.core()
with efmgraph.Network(net) as nw:  # (modules and the result pools are there)
    efmgraph.enumerate_targets(nw, net.targets[:1], 12, 1, 0, 1 << 12)
before = used()
a, b = efmgraph.Network(net), efmgraph.Network(net)
efmgraph.enumerate_targets(a, net.targets[:1], 12, 1, 0, 1 << 26)
held = used()
a.close()
one = used()
b.close()
print(before, held, one, used(), torch.cuda.mem_get_info()[1])
"""


@pytest.mark.gpu
def test_memory_returns_with_the_last_network():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02867_gb300 import build

    build.build()
    out = subprocess.run([sys.executable, "-c", GPU_SCRIPT], capture_output=True, text=True, check=True, cwd=ROOT)
    before, held, one, after, total = (int(x) for x in out.stdout.split()[-5:])
    assert held - before > 20 << 30  # two arenas of 2^26 states
    assert abs(one - held) < 64 << 20  # a network is still there
    assert after - before <= total // 32 + (64 << 20)


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
