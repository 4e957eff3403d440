"""FP64 mode on rays of many tiles, where a block traces several consecutive tiles: the column
carried from tile to tile, and summed anew in front of a block's first one, against the oracle."""
import dataclasses

import numpy as np
import pytest

import synth
from tests import _parity

pytestmark = pytest.mark.gpu


# cells of the rays and their number: one tile per block (as many waves of tiles as blocks), whole
# waves of several tiles, and a tile count that no wave divides
@pytest.mark.parametrize("nr,rays", [(5000, 3), (16385, 60), (60000, 9), (131072, 8)])
def test_long_rays(nr, rays):
    w = synth.disk3d(nr, rays, 1, n_nu=5, tau550=10.0, seed=nr)
    rng = np.random.default_rng(nr)
    rho = w.rho * (0.5 + rng.random(w.rho.shape))
    rho[rng.random(rho.shape) < 0.02] = 0.0
    w = dataclasses.replace(w, rho=rho)
    orc = _parity.oracle_for(w)
    # the outputs are rounded to float32 (6e-8); the column's FP64 sum over nr cells, in another
    # order than the oracle's, moves an attenuation by tau nr 1.1e-16, 2e-10 at most
    q, a, e = _parity.run_gpu(w, "fp64")
    _parity.assert_parity(w, q, a, e, orc, rtol_q=6.2e-8, rtol_a=6.2e-8, rtol_energy=1e-9, label=f"{nr} x {rays}")
