"""An FP64 network whose digit tiles do not fit in the device's memory runs on the
FP64 FMA kernel, as it did before there were digit tiles."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import numpy as np, torch
import paper_2503_12749_gb300 as gbs
import workloads as wl
gbs.build()
N = 4096
rng = np.random.default_rng(3)
T = (rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))) / (2.0 * np.sqrt(N))
r = rng.uniform(0.3, 0.8, size=N)
small = gbs.gbs_make_network(T[:64, :64].copy(), r[:64], "fp64", 0)  # context and kernels loaded
gbs.gbs_debug_samples(small, 5, 0, 64)
# T's upload, its doubles (0.27 GB each) and the samples' (1.07 GB) fit in 2.1 GB;
# with digits (0.47 GB of T, 1.88 GB of samples) 2.6 GB are wanted
free = torch.cuda.mem_get_info()[0]
filler = torch.empty(free - 2_100_000_000, dtype=torch.uint8, device="cuda")
net = gbs.gbs_make_network(T, r, "fp64", 0)
got = gbs.gbs_debug_samples(net, 5, 0, 300)
gbs.gbs_free_network(net)
del filler
torch.cuda.empty_cache()
net = gbs.gbs_make_network(T, r, "fp64", 0)
want = gbs.gbs_debug_samples(net, 5, 0, 300)
gbs.gbs_free_network(net)
scale = np.abs(want[1]).max()
# FP64 chains of N terms against exact sums: (N + 32) 2^-53 of sums of magnitudes,
# here of the order of 100 times the mean photon number
assert np.all(np.abs(got[1] - want[1]) < 1e-11 * scale), np.abs(got[1] - want[1]).max() / scale
assert np.any(got[1] != want[1])  # (two different kernels)
print("ok")
"""


def test_fma_kernel_without_room_for_digits():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and p.stdout.strip().endswith("ok"), p.stdout + p.stderr
