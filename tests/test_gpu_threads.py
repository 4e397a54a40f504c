"""Handles of several threads, each on a stream of its own, whose first passes of
the multi-step kernel start together in a new process: the same bits as one
handle alone, and passes in every one of them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import threading
import numpy as np
import torch
from paper_2210_10377_gb300 import binding

m = np.zeros((64, 400), np.uint8)
m[28:36, 90:110] = 1
N = 8
start = threading.Barrier(N)
out, launches = [None] * N, [0] * N

def work(k):
    lat = binding.Lattice(m, 0.6, 0.05, storage="f16dev", stream=torch.cuda.Stream(), torch_alloc=False)
    start.wait()
    lat.step(1)
    lat.step(80)
    launches[k] = lat.launch_count
    out[k] = (lat.populations(), np.stack(lat.force_series("B")))
    lat.close()

threads = [threading.Thread(target=work, args=(k,)) for k in range(N)]
for t in threads:
    t.start()
for t in threads:
    t.join()
for o in out[1:]:
    assert np.array_equal(o[0], out[0][0]) and np.array_equal(o[1], out[0][1])
assert len(set(launches)) == 1 and launches[0] < 81, launches  # three launches a pass
print("ok")
"""


def test_first_passes_of_several_threads():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
