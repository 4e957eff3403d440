"""Eq. 16 with a diffuse field (E_R given) over its whole range, against the FP64 oracle: sources
from nothing to beyond both ends of the tables, either of them dominant, smooth and steep opacity
tables, whole vectors and a remainder of single cells."""
import numpy as np
import pytest

import oracle
import synth
from tests.test_temperature_gpu import RTOL_T, _tracer, torch  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("table", ["disk", "step"])
@pytest.mark.parametrize("dims", [(40, 25, 20), (7, 3, 1), (1, 1, 1)])
def test_whole_range(torch, table, dims):  # noqa: F811
    w = synth.disk3d(*dims, n_nu=79, tau550=1.0, seed=1)
    kappa = w.kappa if table == "disk" else np.where(w.nu > synth.C_CM_S / 30e-4, 1e3, 1.0)
    tr = _tracer(w, kappa=kappa)
    n = w.grid.ncells
    rng = np.random.default_rng(5)
    a_const = 4 * 5.670374419e-5 / 2.99792458e10
    t_src = 10 ** rng.uniform(np.log10(0.3), np.log10(3e5), n)       # the temperature of the source alone
    kp = np.array([oracle.planck_mean(t, w.nu, kappa) for t in np.geomspace(1.0, 1e5, 64)])
    a = a_const * t_src ** 4 * np.exp(np.interp(np.log(t_src), np.log(np.geomspace(1.0, 1e5, 64)), np.log(kp)))
    e = a_const * (t_src * 10 ** rng.uniform(-2, 2, n)) ** 4         # the field's share from 1e-8 to 1e8
    pick = rng.integers(0, 12, n)
    a[pick == 0] = 0.0
    e[pick == 1] = 0.0
    a[pick == 2] *= 1e-25                                            # far below the table
    a[pick == 3] = 1e-42                                             # subnormal
    a, e = (x.astype(np.float32).reshape(w.grid.shape) for x in (a, e))
    cu = lambda x: torch.from_numpy(x).cuda()
    got = tr.dust_temperature(cu(a), cu(e)).double().cpu().numpy()
    ref = oracle.dust_temperature(a.astype(np.float64), e.astype(np.float64), w.nu, kappa)
    zero = (a == 0.0) & (e == 0.0)
    assert np.all(got[zero] == 0.0)
    # (a subnormal a_rad alone is zero to the hardware functions)
    m = ~zero & ((a > 1e-37) | (e > 0.0))
    rel = np.abs(got[m] / ref[m] - 1)
    assert rel.max() < RTOL_T, (rel.max(), ref[m][np.argmax(rel)], a[m][np.argmax(rel)], e[m][np.argmax(rel)])
    tr.close()
