"""Full-rank kappa(nu, T): the kernel with the bins across the lanes at the edges of its slots (16
bins), chunks (8 cells) and warps (4 rays), against the FP64 oracle within the tracer's bounds, and
the rule that takes the default there."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from tests import _parity

pytestmark = pytest.mark.gpu


def _table(nu, tg):
    return synth.kappa_synth(nu)[:, None] * (0.5 + np.random.default_rng(nu.size).random((nu.size, tg.size)))


def _tracer(w, tg, kt):
    from paper_1001_3301_gb300 import Tracer
    tr = Tracer.from_grid(w.grid)
    tr.set_opacity_table_t(w.nu, tg, kt, w.t_sub)
    tr.set_star(w.t_star, w.r_star)
    return tr


@pytest.mark.parametrize("nr,ntheta,nphi,n_nu,n_t,tau", [
    (8, 3, 1, 15, 32, 1.0), (9, 2, 3, 16, 5, 100.0), (17, 5, 1, 17, 24, 1e-3), (64, 7, 1, 128, 32, 1e5),
    (41, 4, 1, 127, 6, 10.0), (1000, 1, 2, 33, 8, 30.0)])
def test_bins_across_lanes(nr, ntheta, nphi, n_nu, n_t, tau):
    torch = pytest.importorskip("torch")
    w = synth.disk3d(nr, ntheta, nphi, n_nu=n_nu, tau550=tau, seed=nr)
    tg = np.geomspace(10.0, 1400.0, n_t).astype(np.float32).astype(np.float64)
    kt = _table(w.nu, tg)
    rng = np.random.default_rng(nr)
    rho, td = w.rho32().copy(), w.tdust32().copy()
    rho[rng.random(rho.shape) < 0.05] = 0.0            # empty dust cells (their force limit)
    td[rng.random(td.shape) < 0.1] = w.t_sub + 100.0   # sublimated
    td.reshape(-1)[::7] = 5.0                          # below the table
    tr = _tracer(w, tg, kt)
    c = min(s[1] for s in tr.tunings())
    tr.set_tuning(1, c, 4, 1)
    q, a, e = tr.irradiate(torch.from_numpy(rho).cuda(), torch.from_numpy(td).cuda(), energy=True)
    g = w.grid
    orc = oracle.irradiate_tdep(g.r_if, g.theta_if, g.phi_if, w.t_star, w.r_star, w.nu, tg, kt, w.t_sub,
                                rho.astype(np.float64), td.astype(np.float64), nthreads=4)
    _parity.assert_parity(w, q.double().cpu().numpy(), a.double().cpu().numpy(), e, orc, rho=rho, tdust=td)
    tr.close()


@pytest.mark.parametrize("rays,n_nu,takes", [(2047, 64, False), (2048, 64, True), (2048, 63, False), (4096, 32, True),
                                               (4096, 31, False)])
def test_default_rule(rays, n_nu, takes):
    torch = pytest.importorskip("torch")
    w = synth.disk3d(20, rays, 1, n_nu=n_nu)
    tg = np.geomspace(10.0, 1400.0, 9).astype(np.float32).astype(np.float64)
    tr = _tracer(w, tg, _table(w.nu, tg))
    r, t = torch.from_numpy(w.rho32()).cuda(), torch.from_numpy(w.tdust32()).cuda()
    tr.irradiate(r, t)
    assert (tr.tuning()[2:] == (4, 1)) == takes
    out = []
    for s in (tr.tuning(), min(tr.tunings(), key=lambda s: s[3] != 1), max(tr.tunings(), key=lambda s: s[3])):
        tr.set_tuning(*s)
        out.append(tr.irradiate(r, t)[:2])
    for o in out[1:]:  # each within 1e-5 of the exact answer
        for u, v in zip(out[0], o):
            assert float((u - v).abs().max()) <= 2e-5 * float(u.abs().max())
    tr.close()
