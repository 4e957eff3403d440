"""The FLD step's line kernels at the ring lengths where their shared memory passes what a launch
has without asking (static and dynamic part together), in a process that has asked for no more."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STEPS = """
import numpy as np, torch, synth
from tests.test_fld_gpu import RTOL_E, TOL, _step_pair
for nph in (335, 336, 352, 384, 399, 400):  # the shortest first: a longer ring raises the limit for good
    w = synth.disk3d(4, 10, nph, n_nu=32, tau550=10.0, seed=5)
    t, e0, q = synth.fld_fields(w.grid, seed=2)
    got, ref, st = _step_pair(torch, w.grid, w.nu, w.kappa, w.rho, t, q, e0, 1e4, 1e8, 15.0)
    off = np.abs(got / ref - 1).max()
    assert st["rel_change"] < TOL and off < RTOL_E, (nph, off, st)
print("steps ok")
"""


def test_ring_lengths_in_a_fresh_process():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", STEPS], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "steps ok" in r.stdout, (r.returncode, r.stdout[-1000:], r.stderr[-2000:])
