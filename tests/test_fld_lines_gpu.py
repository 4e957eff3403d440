"""The FLD step's phi-line smoother at the edges of its segments and chunks, against the FP64
direct solve (the same inputs and per-cell bound as the FLD step's own test)."""
import numpy as np
import pytest

import synth
from tests.test_fld_gpu import RTOL_E, TOL, _step_pair, torch  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [
    (12, 24, 15),    # one phi cell short of lines
    (12, 24, 16),    # the shortest ring: four segments of four cells
    (12, 24, 17),    # uneven segments
    (9, 30, 37),     # odd nr: the scalar kernels
    (33, 14, 40),    # two blocks along k, the second with one ring
    (16, 24, 64),    # segments of eight
    (8, 16, 130),    # sixteen segments, uneven
    (8, 10, 144),    # interior of one chunk exactly
    (4, 10, 272),    # an interior longer than a chunk
    (5, 8, 600),     # several chunks
    (4, 6, 1024),    # the longest ring whose sweep stays in shared memory
    (4, 6, 1025),    # beyond it
])
@pytest.mark.parametrize("dt", [1e4, 1e300])
def test_rings(torch, shape, dt):  # noqa: F811
    nr, nth, nph = shape
    w = synth.disk3d(nr, nth, nph, n_nu=32, tau550=10.0, seed=5)
    t, e0, q = synth.fld_fields(w.grid, seed=2)
    got, ref, st = _step_pair(torch, w.grid, w.nu, w.kappa, w.rho, t, q, e0, dt, 1e8, 15.0)
    assert st["rel_change"] < TOL
    assert np.abs(got / ref - 1).max() < RTOL_E, (np.abs(got / ref - 1).max(), st)


def test_partial_ranges(torch):  # noqa: F811
    """A wedge away from the poles (no rows for lines) and one that ends at a pole."""
    for lo, hi in ((0.25, 0.75), (0.0, 0.5), (0.5, 1.0)):
        g = synth.log_grid(12, 20, 32)
        g.theta_if = np.linspace(lo * np.pi, hi * np.pi, 21)
        w = synth.disk3d(12, 20, 32, n_nu=32, tau550=10.0, seed=5)
        t, e0, q = synth.fld_fields(g, seed=2)
        got, ref, st = _step_pair(torch, g, w.nu, w.kappa, w.rho, t, q, e0, 1e4, 1e8, 15.0)
        assert np.abs(got / ref - 1).max() < RTOL_E, (lo, hi, np.abs(got / ref - 1).max(), st)
