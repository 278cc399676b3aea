"""A process that resets its own context and goes on: networks are loaded anew,
and sampling and traversals give the same answers as before."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
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
def test_calls_after_a_context_reset():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02867_gb300 import build

    build.build()
    out = subprocess.run([sys.executable, "-c", RESET_SCRIPT], capture_output=True, text=True, cwd=ROOT)
    assert out.stdout.strip() == "same", out.stderr[-2000:]
