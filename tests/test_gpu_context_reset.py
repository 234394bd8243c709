"""cudaDeviceReset between two calls: what the library keeps for small batches
belonged to the old context and is not used again.  In a process of its own,
whose context no other test needs."""
import os
import subprocess
import sys

import pytest

import oracle

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes
from paper_1810_06800_gb300 import rsa
for name in ("/usr/local/cuda/lib64/libcudart.so", "libcudart.so.13", "libcudart.so"):
    try:
        cuda = ctypes.CDLL(name)
        break
    except OSError:
        pass
else:
    raise SystemExit(77)
def both():
    for run in (rsa.rsa_run_small, rsa.rsa_run_static):
        nj, nc = run(16, 2, [1, 2, 3])
        print(*nj, *nc)
both()
assert cuda.cudaDeviceSynchronize() == 0 and cuda.cudaDeviceReset() == 0
both()
rsa.rsa_mix_release()
both()
"""


def test_small_batches_after_a_device_reset():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                       timeout=120)
    if r.returncode == 77:
        pytest.skip("no shared CUDA runtime to reset the device with")
    assert r.returncode == 0, r.stderr[-2000:]
    nj, nc = oracle.samples(16, 2, [1, 2, 3])
    want = " ".join(str(int(v)) for v in [*nj, *nc])
    assert r.stdout.split("\n")[:-1] == [want] * 6
