"""The FP64 mode's shortcuts (power series over thin bins, Taylor classes of the absorbed
fraction, the reduced exponential, the attenuation carried along a lane's cells, bins that
underflow) against the FP64 oracle, to the rounding of the float32 outputs."""
import dataclasses

import numpy as np
import pytest

import synth
from tests import _parity

pytestmark = pytest.mark.gpu

# outputs are rounded to float32 (2^-24 of the value); what is left for the FP64 arithmetic,
# at most 1e-12 of a cell's value (a few hundred roundings of 1.1e-16, amplified 7.4-fold by
# the alternating series), is far below the difference to 6.1e-8
RTOL = 6.1e-8


def _workload(nr, scale, seed):
    """Rays whose per-cell optical depths run over ten decades around `scale` (in units of
    1 / kappa_max), 24 bins with opacities over eight decades, one tenth of the cells without
    dust and one tenth of the dust cells without gas."""
    w = synth.disk3d(nr, 5, 3, 24, 1.0, seed)
    rng = np.random.default_rng(seed)
    kappa = np.geomspace(1e-4, 1e4, 24)
    col = scale / kappa[-1] * 10.0 ** rng.uniform(-5, 0, w.grid.shape)
    rho = col / np.diff(w.grid.r_if)
    rho[rng.random(w.grid.shape) < 0.1] = 0.0
    td = np.where(rng.random(w.grid.shape) < 0.1, 1600.0, 300.0)
    return dataclasses.replace(w, kappa=kappa, rho=rho, tdust=td)


@pytest.mark.parametrize("nr", [1, 7, 64, 131, 300])
# the largest kappa dN of a cell: every bin thin; at the class ends of 5, 8 and 13 terms; the
# series end; the exponential's range; bins that underflow behind a few cells; far beyond it
@pytest.mark.parametrize("scale", [1e-4, 2.09e-3, 4.6e-2, 0.3465, 1.0, 30.0, 3e3, 1e7])
def test_classes(nr, scale):
    from paper_1001_3301_gb300 import Tracer
    w = _workload(nr, scale, seed=nr + 11)
    orc = _parity.oracle_for(w)
    with Tracer.from_grid(w.grid, "fp64") as tr:
        shapes = tr.tunings()
    for shape in shapes:
        q, a, e = _parity.run_gpu(w, "fp64", shape=shape)
        _parity.assert_parity(w, q, a, e, orc, rtol_q=RTOL, rtol_a=RTOL, rtol_energy=1e-11,
                              label=f"nr={nr} scale={scale} {shape}")
