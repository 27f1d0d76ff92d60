"""The workspace sizes that include/lbnci.h documents for the faster steps are the ones that select
them: at lb_workspace_size() bytes the step runs the kernels without scratch, at the documented size
more the three passes (seen by the kernels launched per step), to the same populations."""
import os
import re

import pytest

from paper_2003_11069_gb300 import lbnci

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include", "lbnci.h")


def _documented(row):
    m = re.search(row + r"\s+(\d+) N \+ (\d+)", open(HEADER).read())
    return int(m.group(1)), int(m.group(2))


@pytest.mark.parametrize("row,lat,dims,precisions,kernels", [
    (r"FP64 with Guo forcing, D2Q9 and D3Q27", lbnci.LB_D2Q9, (36, 17, 1), (lbnci.LB_FP64,), (1, 3)),
    (r"FP64 with Guo forcing, D2Q9 and D3Q27", lbnci.LB_D3Q27, (32, 8, 5), (lbnci.LB_FP64,), (2, 3)),
    (r"FP32 and FP16-dev D2Q9 with nx % 4 != 0", lbnci.LB_D2Q9, (37, 19, 1), (lbnci.LB_FP32, lbnci.LB_FP16DEV), (1, 3)),
    (r"FP32 and FP16-dev D3Q27 with nx % 32 != 0 or ny % 8 != 0", lbnci.LB_D3Q27, (33, 9, 5),
     (lbnci.LB_FP32, lbnci.LB_FP16DEV), (2, 3)),
])
def test_documented_sizes_select_the_passes(row, lat, dims, precisions, kernels, monkeypatch):
    for k in ("LBNCI_D3_KERNEL", "LBNCI_FUSED", "LBNCI_FUSED_SPT"):
        monkeypatch.delenv(k, raising=False)
    per_site, more = _documented(row)
    N = dims[0] * dims[1] * dims[2]
    psi = 0.9 * torch.sin(0.9 * torch.arange(N, dtype=torch.float64, device="cuda"))
    for precision in precisions:
        cfg = lbnci.lb_config_make(lattice=lat, nx=dims[0], ny=dims[1], nz=dims[2], wall_y=1,
                                   wall_z=int(lat == lbnci.LB_D3Q27), tau=0.8, A_s=0.01, beta=0.7, A_h=0.05,
                                   precision=precision)
        least = lbnci.lb_workspace_size(cfg)
        got = []
        for n, launches in ((least, kernels[0]), (least + per_site * N + more, kernels[1])):
            ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
            cfg.workspace, cfg.workspace_bytes = (ws.data_ptr() + 255) & ~255, n
            with lbnci.Sim(cfg) as sim:
                sim.init_fields(0.5 * (1 + psi), 0.5 * (1 - psi))
                before = sim.launches()
                sim.step(2)
                assert sim.launches() - before == 2 * launches
                got.append(torch.empty((18 if lat == lbnci.LB_D2Q9 else 54) * N, dtype=torch.float64, device="cuda"))
                lbnci.lb_get_populations(sim.h, got[-1])
        assert torch.equal(*got)
