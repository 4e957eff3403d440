"""Eq. 16 with a diffuse field on kappa(nu, T) tables, whose Planck mean has a kink at every
temperature point: each cell's T is within the bound of a root of the equation in FP64, on the mean
as the library tabulates it (1024 points of ln T, cubic Hermite with Catmull-Rom tangents, held
outside; the steepest table has more than one root in places)."""
import numpy as np
import pytest

import synth
from tests.test_temperature_gpu import RTOL_T, torch  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

A_CONST = 4 * 5.670374419184429e-5 / 2.99792458e10
LN_HI = 11.512925464970229


def _mean_on_nodes(tr):
    """L(y) = ln kappa_P(e^y) as tabulated."""
    y = np.linspace(0.0, LN_HI, 1024)
    p = np.log([tr.planck_mean_opacity(float(t)) for t in np.exp(y)]).astype(np.float32).astype(np.float64)
    m = np.gradient(p)  # (p[k+1] - p[k-1]) / 2, one-sided at the ends

    def mean(v):
        u = np.clip(v * (1023 / LN_HI), 0.0, 1023.0)
        k = np.minimum(u.astype(int), 1022)
        t = u - k
        q2 = 3 * (p[k + 1] - p[k]) - 2 * m[k] - m[k + 1]
        q3 = 2 * (p[k] - p[k + 1]) + m[k] + m[k + 1]
        return p[k] + t * (m[k] + t * (q2 + t * q3))
    return mean


def _excess(mean, t, a, e):
    """a T^4 - E_R - a_rad / kappa_P(T), relative to a T^4: changes sign at a root."""
    return 1.0 - (e + a * np.exp(-mean(np.log(t)))) / (A_CONST * t ** 4)


def _table(name, nu):
    if name.startswith("full"):
        tg = np.geomspace(10.0, 1500.0, int(name[4:]))
        f = 0.5 + np.random.default_rng(0).random((nu.size, tg.size))
        return tg, synth.kappa_synth(nu)[:, None] * f
    if name == "ice":
        tg = synth.t_grid(24)
        return tg, synth.kappa_synth_t3(nu, tg)
    tg = np.array([10.0, 100.0, 110.0, 1500.0])  # ten-fold within 10 K, up or down by a quarter
    return tg, synth.kappa_synth(nu)[:, None] * np.array([1.0, 1.0] + [10.0 if name == "up" else 0.75] * 2)


@pytest.mark.parametrize("name", ["full24", "full32", "ice", "up", "down"])
@pytest.mark.parametrize("t_lo,t_hi", [(5.0, 3000.0), (0.3, 3e5)])
def test_kinked_means(torch, name, t_lo, t_hi):  # noqa: F811
    from paper_1001_3301_gb300 import Tracer
    nu = synth.nu_bins(79)
    tg, kt = _table(name, nu)
    g = synth.log_grid(64, 63, 64)
    tr = Tracer.from_grid(g)
    tr.set_opacity_table_t(nu, tg, kt, synth.T_SUB_K)
    tr.set_star(synth.T_STAR_K, synth.R_STAR_CM)
    mean = _mean_on_nodes(tr)
    rng = np.random.default_rng(7)
    t = np.exp(rng.uniform(np.log(t_lo), np.log(t_hi), g.shape))
    share = 10 ** rng.uniform(-1, 1, g.shape)
    s = A_CONST * t ** 4 / (1 + share)
    e, a = (s * share).astype(np.float32), (s * np.exp(mean(np.log(t)))).astype(np.float32)
    got = tr.dust_temperature(torch.from_numpy(a).cuda(), torch.from_numpy(e).cuda()).double().cpu().numpy()
    a, e = a.astype(np.float64), e.astype(np.float64)
    # within the bound of a root; where the mean falls nearly as T^-4 a root is no better defined than
    # the equation: there the terms balance to the same bound (4 RTOL_T of a T^4 are RTOL_T of T)
    off = (_excess(mean, got * (1 - RTOL_T), a, e) * _excess(mean, got * (1 + RTOL_T), a, e) > 0) & (
        np.abs(_excess(mean, got, a, e)) > 4 * RTOL_T)
    assert not off.any(), (off.sum(), got[off][:4], a[off][:4], e[off][:4])
    tr.close()
