"""The host-buffer entry point at the cell counts where its number of ray chunks changes: outputs
equal the device path bit for bit, the energy (partials grouped by chunk) to rounding."""
import pytest

import synth

pytestmark = pytest.mark.gpu


# two chunks; four; six, with rays that no chunk count divides; six of odd rays
@pytest.mark.parametrize("nr,ntheta,nphi", [(128, 64, 129), (256, 64, 133), (256, 128, 257), (301, 97, 289)])
def test_chunks(nr, ntheta, nphi):
    torch = pytest.importorskip("torch")
    from paper_1001_3301_gb300 import Tracer
    w = synth.disk3d(nr, ntheta, nphi, n_nu=16, tau550=10.0, seed=8)
    tr = Tracer.from_grid(w.grid)
    tr.set_opacity_table(w.nu, w.kappa, w.t_sub)
    tr.set_star(w.t_star, w.r_star)
    rho, td = torch.from_numpy(w.rho32()), torch.from_numpy(w.tdust32())
    q1, a1, e1 = tr.irradiate(rho.cuda(), td.cuda(), energy=True)
    pq, pa = (torch.full(w.grid.shape, -1.0, dtype=torch.float32).pin_memory() for _ in range(2))
    e2 = tr.irradiate_host(rho.pin_memory(), td.pin_memory(), pq, pa, energy=True)
    assert torch.equal(pq, q1.cpu()) and torch.equal(pa, a1.cpu())
    assert abs(e2.e_abs / e1.e_abs - 1) < 1e-9 and abs(e2.e_esc / e1.e_esc - 1) < 1e-9
    tr.close()
