"""D3Q27 lattices of whole 32 x 8 columns with more planes or rows than a grid has blocks along z
or y: they step on the marching kernel, whose grid counts along x, to its bits."""
import pytest

from paper_2003_11069_gb300 import lbnci

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", [lbnci.LB_FP32, lbnci.LB_FP16DEV])
@pytest.mark.parametrize("ny,nz", [(8, 65537), (8 * 65536, 2)])
def test_whole_columns_longer_than_a_grid_axis(ny, nz, precision, monkeypatch):
    """Bitwise: the same kernel as LBNCI_D3_KERNEL=march selects."""
    nx, N = 32, 32 * ny * nz
    psi = 0.9 * torch.sin(0.9 * torch.arange(N, dtype=torch.float64, device="cuda"))
    rho1, rho2 = 0.5 * (1 + psi), 0.5 * (1 - psi)
    cfg = lbnci.lb_config_make(lattice=lbnci.LB_D3Q27, nx=nx, ny=ny, nz=nz, wall_y=1, wall_z=1, tau=0.8, A_s=0.01,
                               beta=0.7, A_h=0.05, force=(2e-5, 0.0, 0.0), precision=precision)
    got = []
    for kernel in ("", "march"):
        monkeypatch.setenv("LBNCI_D3_KERNEL", kernel) if kernel else monkeypatch.delenv("LBNCI_D3_KERNEL", raising=False)
        with lbnci.Sim(cfg) as sim:
            assert sim.step_path() == lbnci.LB_PATH_D3Q27 and sim.state_form() == lbnci.LB_STATE_PAIRS
            sim.init_fields(rho1, rho2)
            sim.step(2)
            got.append(torch.empty(54 * N, dtype=torch.float64, device="cuda"))
            lbnci.lb_get_populations(sim.h, got[-1])
            if nz > 2:  # (the fields kernels count rows and planes by blocks of 4 and 2)
                assert abs(sim.observables()["mass"][0] / float(rho1.sum()) - 1.0) < 1e-4
    assert torch.equal(*got)
