"""The shape a context takes without autotuning: it serves the table, and the result meets the
oracle at the sizes where the choice changes."""
import numpy as np
import pytest

import synth
from tests import _parity
from tests.test_tdep_gpu import _oracle, _run, _tg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nr", [64, 256, 257, 300, 383, 384, 385, 512])
def test_separable_table(nr):
    """A separable kappa(nu, T) table needs a kernel with the column weight (rays of 257 to 383
    cells went to the tile kernel, which has none)."""
    w = synth.disk3d(nr, 6, 3, 24, 1.0, 3)
    tg = _tg(12)
    kt = synth.kappa_synth_t(w.nu, tg)
    q, a, e, _ = _run(w, tg, kt, kind=1)
    _parity.assert_parity(w, q, a, e, _oracle(w, tg, kt), label=f"nr={nr}")


@pytest.mark.parametrize("dims", [(1, 1, 1), (8, 4, 1), (64, 24, 1), (64, 40, 40), (200, 40, 30), (300, 30, 30),
                                  (512, 30, 20), (513, 40, 40), (513, 20, 20), (1100, 40, 39)])
def test_plain_table(dims):
    from paper_1001_3301_gb300 import Tracer
    w = synth.disk3d(*dims, n_nu=16, tau550=10.0, seed=3)
    orc = _parity.oracle_for(w)
    for precision in ("fp32_kahan", "fp32_plain"):
        with Tracer.from_grid(w.grid, precision) as tr:
            tr.set_opacity_table(w.nu, w.kappa, w.t_sub)
            tr.set_star(w.t_star, w.r_star)
            assert tr.tuning() in tr.tunings()
        q, a, e = _parity.run_gpu(w, precision)
        _parity.assert_parity(w, q, a, e, orc, rtol_q=1e-5 if precision == "fp32_kahan" else 1e-4,
                              rtol_a=1e-5 if precision == "fp32_kahan" else 1e-4, label=f"{dims} {precision}")
