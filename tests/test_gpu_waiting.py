"""How the host waits for the neighbor lists while earlier work holds the stream:
blocked, where the process asked for it (cudaDeviceScheduleBlockingSync), and with
the same results under each of the device's schedules."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = r"""
import ctypes, sys, time
from paper_2303_12980_gb300.binding import GMPFeaturizer, load_library
assert load_library().cudaSetDeviceFlags(ctypes.c_uint(int(sys.argv[1]))) == 0
import numpy as np, torch
from paper_2303_12980_gb300 import synth
rng = np.random.default_rng(1)
pos, cell = synth.fcc_supercell(rng, 3.6, (4, 4, 4), 0.1)
n = len(pos)
a = (torch.from_numpy(pos).cuda(), torch.zeros(n, dtype=torch.int32, device="cuda"), [0, n], cell[None], [[1, 1, 1]])
F = GMPFeaturizer([0, 1, 2], [0.4, 0.8], 5.0, *synth.gaussian_table(rng, [3], 2))
g = torch.ones((n, F.num_features), device="cuda")
calls = [lambda: F.featurize(*a), lambda: F.featurize_vjp(*a, g)[1], lambda: F.featurize_grad(*a)[3],
         lambda: F.featurize_points(*a, a[0], [0, n])]
for call in calls:
    want = [call() for _ in range(2)][1]
    torch.cuda.synchronize()
    torch.cuda._sleep(800_000_000)  # about 0.4 s
    t, c = time.perf_counter(), time.process_time()
    got = call()
    t, c = time.perf_counter() - t, time.process_time() - c
    torch.cuda.synchronize()
    assert torch.equal(got, want) and t > 0.2, t
    if sys.argv[1] == "4":
        assert c < 0.3 * t, (c, t)
print("waited")
"""


@pytest.mark.parametrize("schedule", [0, 1, 2, 4])  # auto, spin, yield, blocking
def test_wait_as_the_process_asks(schedule):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE, str(schedule)], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "waited" in r.stdout, r.stdout + r.stderr
