"""The library's memory pool: what it keeps between calls goes back when its last user goes.  Each test in a
process of its own (the pool is one per process and device)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(code):
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]


def test_memory_goes_back_with_the_last_model():
    """A model outlives its mechanism: 190 MB of a per-species pass are kept until the model is freed."""
    _run("""
import sys; sys.path.insert(0, "tests")
import numpy as np, torch, paper_2312_13513_gb300 as cg
from oracle import surrogate as osur
from synth.mechanism import h2_mechanism
from helpers import random_states
from gpu_common import to_dev
from test_gpu_surrogate_per_species import _ps_params
h2 = h2_mechanism()
T, p, Y = random_states(h2, 32768, 31, "H2", Tlo=300.0, Thi=2500.0)
prm = _ps_params(h2, osur.features(T, p, Y), 32, (1600, 800, 400))
Td, pd, Yd = to_dev(T, p, Y)
free = []
for _ in range(3):                                   # the first round loads the kernels
    dm = cg.Mechanism(h2)
    model = cg.Surrogate(dm, params=prm)
    dm.close()
    out = cg.surrogate_forward(model, Td, pd, Yd)
    torch.cuda.synchronize()
    kept = torch.cuda.mem_get_info()[0]
    model.close()
    del out
    torch.cuda.empty_cache()
    free.append(torch.cuda.mem_get_info()[0])
    assert free[-1] - kept > 100e6, (free, kept)
assert abs(free[2] - free[1]) < 8e6, free
""")


def test_pool_of_a_context_that_was_reset():
    """A device reset ends the context and the pool with it: a mechanism loaded afterwards works on a pool of
    the new context, with the same results."""
    _run("""
import ctypes
import numpy as np
import paper_2312_13513_gb300 as cg
from paper_2312_13513_gb300 import _lib
from synth.mechanism import h2_mechanism
from synth.states import load_table, quasi_dns_field
L = _lib.load()
rt = ctypes.CDLL("libcudart.so.13")                  # the one the library has loaded
f = quasi_dns_field(load_table("h2_flamelet.npz"), n=2011, seed=3)
rt.cudaMalloc.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
rt.cudaMemcpy.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]

def dev(a):
    a = np.ascontiguousarray(a, np.float64)
    p = ctypes.c_void_p()
    assert rt.cudaMalloc(ctypes.byref(p), a.nbytes) == 0 and rt.cudaMemcpy(p, a.ctypes.data, a.nbytes, 1) == 0
    return p

out = []
for _ in range(3):
    dm = cg.Mechanism(h2_mechanism())
    T, p, Y = dev(f["T"]), dev(f["p"]), dev(f["Y"])
    for _ in range(2):
        assert L.chem_advance(dm.handle, T, p, Y, 5e-7, 2011, 1e-6, 1e-10, None) == 0, L.chem_last_error()
        assert rt.cudaDeviceSynchronize() == 0
    h = np.empty(2011)
    assert rt.cudaMemcpy(h.ctypes.data, T, h.nbytes, 2) == 0
    out.append(h)
    dm.close()
    assert rt.cudaDeviceReset() == 0
assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
""")
