"""``lbm_front_heights`` keeps pinned blocks from one call to the next. A
``cudaDeviceReset`` frees them with everything else of the device: simulations
created afterwards read their fronts through new ones. In a process of its own,
which holds no other CUDA state."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = """
import ctypes
import numpy as np
from paper_2303_02210_gb300 import lbm
from paper_2303_02210_gb300 import workloads as wl

lib = lbm.load_library()
rt = ctypes.CDLL("libcudart.so.13")
p = lbm.make_params(wl.lattice_small(seed=3, growth_rate=3e-3), "fp64")

def run():
    h = ctypes.c_void_p()
    assert lib.lbm_create(ctypes.byref(p), None, None, 0, ctypes.byref(h)) == 0, lib.lbm_last_cuda_error()
    assert lib.lbm_step(h, 25) == 0
    front = np.empty(p.width, dtype=np.int32)
    hbar, w = ctypes.c_double(), ctypes.c_double()
    for _ in range(2):
        rc = lib.lbm_front_heights(h, front.ctypes.data, ctypes.byref(hbar), ctypes.byref(w))
        assert rc == 0, lib.lbm_last_cuda_error()
    lib.lbm_destroy(h)
    return front, hbar.value, w.value

a = run()
assert rt.cudaDeviceReset() == 0
# other pinned memory where the blocks were
q = ctypes.c_void_p()
assert rt.cudaHostAlloc(ctypes.byref(q), ctypes.c_size_t(1 << 20), 3) == 0
mine = np.ctypeslib.as_array(ctypes.cast(q, ctypes.POINTER(ctypes.c_uint8)), shape=(1 << 20,))
mine[:] = 7
b = run()
assert np.array_equal(a[0], b[0]) and a[1:] == b[1:], (a, b)
assert (mine == 7).all()
print("fronts equal across a reset")
"""


def test_front_heights_after_a_device_reset():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "fronts equal across a reset" in r.stdout, r.stderr[-2000:]
