"""Which step a configuration gets, as far as its workspace shows it (no GPU needed): lattices that
a grid of the streaming D3Q27 kernels cannot hold (more than 65535 blocks along y or z) take the
workspace of the marching step, those just inside take the streaming one's."""
import pytest

from paper_2003_11069_gb300 import lbnci


@pytest.mark.parametrize("precision", [lbnci.LB_FP32, lbnci.LB_FP16DEV])
@pytest.mark.parametrize("other", ["march", "carry"])
@pytest.mark.parametrize("nx,ny,nz,fits", [(32, 8, 65535, True), (32, 8, 65536, False), (64, 8, 65537, False),
                                           (32, 8 * 65535, 2, True), (32, 8 * 65536, 2, False)])
def test_workspace_of_lattices_at_the_limits_of_a_grid_axis(nx, ny, nz, fits, precision, other, monkeypatch):
    cfg = lbnci.lb_config_make(lattice=lbnci.LB_D3Q27, nx=nx, ny=ny, nz=nz, wall_y=1, wall_z=1, precision=precision)
    monkeypatch.delenv("LBNCI_D3_KERNEL", raising=False)
    default = lbnci.lb_workspace_size(cfg)
    monkeypatch.setenv("LBNCI_D3_KERNEL", other)
    assert (default != lbnci.lb_workspace_size(cfg)) == fits
