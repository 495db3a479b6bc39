"""Handles before and after a cudaDeviceReset: nothing of the library outlives
the last handle, so the reset leaves no stale memory behind; and handles made
and destroyed by several threads, whose result records share pages."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

from paper_1309_1656_gb300 import fields

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RESET = r"""
import ctypes, sys
import numpy as np
from paper_1309_1656_gb300 import fields, qlbm
st = fields.random_populations(2, (24, 3, 1), seed=5)
def run():
    with qlbm.Lattice(2, (24, 3, 1), 0.8, 1.0, precision="fp64") as lat:
        lat.set_state(st)
        lat.step(3)
        lat.sync()
        return lat.conserved(), lat.get_state()
a = run()
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuDevicePrimaryCtxReset_v2(0) == 0     # what cudaDeviceReset does
b = run()
assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
"""


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1309_1656_gb300 import qlbm
    return qlbm


def test_handles_around_a_device_reset(q):
    r = subprocess.run([sys.executable, "-c", RESET], cwd=ROOT, timeout=300, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]


def test_handles_of_several_threads(q):
    # 8 threads make, use and destroy 40 handles each; up to 5 of a thread's
    # live at once, more than one page of 32 in all
    dims, out = (16, 2, 1), {}
    states = [fields.random_populations(2, dims, seed=s) for s in range(8)]
    want = []
    for st in states:
        with q.Lattice(2, dims, 0.8, 1.0, precision="fp64") as lat:
            lat.set_state(st)
            want.append(lat.conserved())

    def work(i):
        ok = True
        for _ in range(8):
            lats = [q.Lattice(2, dims, 0.8, 1.0, precision="fp64") for _ in range(5)]
            for lat in lats:
                lat.set_state(states[i])
            for lat in lats:
                ok = ok and np.array_equal(lat.conserved(), want[i])
                lat.close()
        out[i] = ok

    threads = [threading.Thread(target=work, args=(i,)) for i in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert out == {i: True for i in range(8)}
