"""Fields that pass through shared memory (rays that do not start on vector boundaries) against the
oracle: odd ray lengths around the shapes' segment sizes, arrays off their 16-byte boundary, more
slots than warps (both buffers), a last slot with missing rays, every warp-per-ray shape."""

import numpy as np
import pytest

import synth
from tests import _parity

pytestmark = pytest.mark.gpu


def _trace(w, shape, off):
    """Trace with every field `off` floats past an aligned base."""
    import torch
    from paper_1001_3301_gb300 import Tracer
    n = w.grid.ncells

    def place(x):
        t = torch.zeros(n + off, dtype=torch.float32, device="cuda")
        if x is not None:
            t[off:] = torch.from_numpy(np.ascontiguousarray(x).ravel()).cuda()
        return t[off:].view(w.grid.shape)

    with Tracer.from_grid(w.grid) as tr:
        tr.set_opacity_table(w.nu, w.kappa, w.t_sub)
        tr.set_star(w.t_star, w.r_star)
        shapes = [s for s in tr.tunings() if s[0] > 0]
        if shape is None:
            return shapes
        tr.set_tuning(*shape)
        q, a, e = tr.irradiate(place(w.rho32()), place(w.tdust32()), place(None), place(None), energy=True)
        return q.double().cpu().numpy(), a.double().cpu().numpy(), e


@pytest.mark.parametrize("nr,off", [(3, 0), (63, 0), (65, 0), (127, 0), (129, 0), (191, 0), (193, 0), (255, 0), (257, 0),
                                    (383, 0), (385, 0), (511, 0), (513, 0), (1001, 0), (256, 1), (512, 3), (600, 2)])
def test_staged_fields(nr, off):
    w = synth.disk3d(nr, 33, 7, 24, 10.0, 3)
    w.rho[w.rho < 1e-30] = 0.0
    orc = _parity.oracle_for(w)
    for shape in _trace(w, None, 0):
        q, a, e = _trace(w, shape, off)
        _parity.assert_parity(w, q, a, e, orc, label=f"nr={nr} off={off} {shape}")


def test_many_slots():
    """More rays than resident warps hold at once, so that every warp walks several slots."""
    w = synth.disk3d(135, 160, 130, 8, 1.0, 5)
    orc = _parity.oracle_for(w)
    for shape in _trace(w, None, 0):
        q, a, e = _trace(w, shape, 0)
        _parity.assert_parity(w, q, a, e, orc, label=str(shape))
