"""The warp-per-ray batch on fields off their 16-byte boundary, which pass through shared memory
although the rays' lengths are multiples of the vector: against the oracle."""
import numpy as np
import pytest

import synth
from tests import _parity
from tests.test_batch_gpu import _tracers, torch  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 16, 4, 3), (1, 16, 4, 4), (1, 8, 4, 6)])
@pytest.mark.parametrize("off", [1, 2, 3])
def test_unaligned_fields(torch, shape, off):  # noqa: F811
    from paper_1001_3301_gb300 import Batch
    # segments of 8, 16 and 32 lanes, full and partly filled; grids whose last slot misses rays
    ws = [synth.disk3d(nr, 7, 5, n_nu=n_nu, tau550=tau, seed=nr) for nr, n_nu, tau in
          ((64, 32, 1.0), (128, 79, 10.0), (192, 16, 0.3), (256, 79, 100.0), (100, 32, 3.0), (4, 5, 1.0))]
    trs = _tracers(ws)

    def place(x):
        t = torch.full((x.size + off,), float("nan"), dtype=torch.float32, device="cuda")
        t[off:] = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32).ravel()).cuda()
        return t[off:].view(x.shape)

    rho, td = [place(w.rho32()) for w in ws], [place(w.tdust32()) for w in ws]
    q, a = ([place(np.full(w.grid.shape, np.nan)) for w in ws] for _ in range(2))
    with Batch(trs) as b:
        assert b.set_tuning(*shape) == shape
        b.run(rho, td, q, a)
        for w, qq, aa, e in zip(ws, q, a, b.energy()):
            _parity.assert_parity(w, qq.double().cpu().numpy(), aa.double().cpu().numpy(), e, _parity.oracle_for(w),
                                  label=f"{w.grid.nr} {shape} {off}")
    for tr in trs:
        tr.close()
