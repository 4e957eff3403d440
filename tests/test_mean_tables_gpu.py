"""The mean opacities from groups of 8 lanes: bin counts off the four bins a warp takes at a time,
bands wide and narrow against kT, a single bin and transparent bins, against the FP64 oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_nu", [1, 2, 3, 5, 31, 32, 79, 128])
@pytest.mark.parametrize("t", [1.0, 20.0, 700.0, 1e5])
def test_planck_and_rosseland_means(n_nu, t):
    """Both sides integrate the bands with 8-point Gauss panels of at most one unit of x in FP64; what
    differs is the order of at most ~200 positive terms and the rounding of the nodes: 1e-12."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_3301_gb300 import Tracer
    w = synth.disk3d(8, 4, 1, n_nu=max(n_nu, 2))
    nu, kappa = w.nu[:n_nu], w.kappa[:n_nu].copy()
    if n_nu == 5:
        kappa[1] = 0.0
    tr = Tracer.from_grid(w.grid)
    tr.set_opacity_table(nu, kappa, w.t_sub)
    tr.set_star(w.t_star, w.r_star)
    p, r = oracle.planck_mean(t, nu, kappa), oracle.rosseland_mean(t, nu, kappa)
    assert abs(tr.planck_mean_opacity(t) - p) <= 1e-12 * p
    assert abs(tr.rosseland_mean_opacity(t) - r) <= 1e-12 * r
    tr.close()
