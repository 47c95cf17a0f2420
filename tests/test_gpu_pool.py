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
