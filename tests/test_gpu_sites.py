"""The per-site passes (csrc/lb_sites.cuh): the FP64 step and the fields and observables, against
the kernels that recompute over halos and against the oracle, at the edges of their blocks (one
site, one site more or less than a block, rows that fill no warp), for every storage layout."""
import numpy as np
import pytest

import oracle
from paper_2003_11069_gb300 import inputs, lbnci

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES_2D = [(1, 1), (33, 9), (31, 40), (128, 64), (36, 17)]
SIZES_3D = [(3, 2, 2), (33, 9, 5), (31, 7, 17), (64, 16, 18)]


def _state(lat, nx, ny, nz, seed):
    """Populations of a mixture with interfaces everywhere and a non-equilibrium part."""
    rng = np.random.default_rng(seed)
    N, Q = nx * ny * nz, 9 if lat == lbnci.LB_D2Q9 else 27
    psi = np.clip(1.5 * np.sin(0.9 * np.arange(N) + rng.uniform(-1, 1, N)), -0.95, 0.95)
    p = oracle.make_params(lattice=lat, nx=nx, ny=ny, nz=nz)
    f = oracle.init(p, 0.5 * (1 + psi), 0.5 * (1 - psi))
    return f * (1 + 0.05 * rng.uniform(-1, 1, 2 * Q * N))


def _cfg(lat, nx, ny, nz, walls, precision, A_h=0.05, h_max=4.0):
    return lbnci.lb_config_make(lattice=lat, nx=nx, ny=ny, nz=nz, wall_y=walls[0], wall_z=walls[1], tau=0.8, A_s=0.01,
                                beta=0.7, A_h=A_h, h_max=h_max, force=(2e-5, -1e-5, 0.0), precision=precision)


CASES = [(lbnci.LB_D2Q9, nx, ny, 1, (w, 0)) for nx, ny in SIZES_2D for w in (0, 1)] + \
    [(lbnci.LB_D3Q27, nx, ny, nz, w) for nx, ny, nz in SIZES_3D for w in ((0, 0), (1, 0), (1, 1))]


@pytest.mark.parametrize("lat,nx,ny,nz,walls", CASES)
def test_fp64_passes_equal_the_one_pass_kernels(lat, nx, ny, nz, walls, monkeypatch):
    """Bitwise: the passes round every value as the fused D2Q9 and the marching D3Q27 kernels do."""
    f = _state(lat, nx, ny, nz, 3)
    out = {}
    for mode in ("passes", "halo"):
        for k in ("LBNCI_D3_KERNEL", "LBNCI_FUSED", "LBNCI_FUSED_SPT"):
            monkeypatch.delenv(k, raising=False)
        if mode == "halo":
            monkeypatch.setenv("LBNCI_FUSED", "classic")
            monkeypatch.setenv("LBNCI_D3_KERNEL", "march")
        for A_h, h_max in ((0.05, 4.0), (0.05, 2.5), (0.0, 4.0)):
            with lbnci.Sim(_cfg(lat, nx, ny, nz, walls, lbnci.LB_FP64, A_h, h_max)) as sim:
                sim.set_populations(f)
                sim.step(3)
                out[mode, A_h, h_max] = sim.get_populations()
    for k in [k[1:] for k in out if k[0] == "passes"]:
        assert np.array_equal(out[("passes",) + k], out[("halo",) + k])


@pytest.mark.parametrize("precision", [lbnci.LB_FP64, lbnci.LB_FP32])
def test_passes_need_no_larger_workspace(precision, monkeypatch):
    """A workspace without room for the passes' scratch still steps, to the state of one that has it
    and of a sim that allocates its own memory."""
    monkeypatch.delenv("LBNCI_D3_KERNEL", raising=False)
    f = _state(lbnci.LB_D3Q27, 33, 9, 5, 4)
    cfg = _cfg(lbnci.LB_D3Q27, 33, 9, 5, (1, 1), precision)
    least = lbnci.lb_workspace_size(cfg)
    got = []
    for n in (least, least + 48 * 33 * 9 * 5 + 1024, 0):
        ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
        cfg.workspace, cfg.workspace_bytes = ((ws.data_ptr() + 255) & ~255, n) if n else (None, 0)
        with lbnci.Sim(cfg) as sim:
            sim.set_populations(f)
            sim.step(2)
            got.append(sim.get_populations())
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])


@pytest.mark.parametrize("precision", [lbnci.LB_FP64, lbnci.LB_FP32, lbnci.LB_FP16DEV])
@pytest.mark.parametrize("lat,nx,ny,nz,walls", CASES)
def test_fields_and_observables(lat, nx, ny, nz, walls, precision):
    """Every field and the sums, of a state as it was set and of one a step left, against the
    oracle's of the same populations. FP64: rounding. FP32 arithmetic: densities and u are sums of
    27 terms of order one with 2^-24 relative rounding each, and the gradient one of 18 terms of
    order one, so 100 2^-24 bounds them; the near-contact force is compared where both found the
    same distance, and the distances may differ only at near-ties (a few sites)."""
    p = oracle.make_params(lattice=lat, nx=nx, ny=ny, nz=nz, wall_y=walls[0], wall_z=walls[1], tau=0.8, A_s=0.01,
                           beta=0.7, A_h=0.05, force=(2e-5, -1e-5, 0.0))
    tol = 1e-13 if precision == lbnci.LB_FP64 else 100 * 2.0 ** -24
    N = nx * ny * nz
    if N == 1 and precision != lbnci.LB_FP64:
        pytest.skip("host populations of one site below FP64 are refused (no room to stage them)")
    with lbnci.Sim(_cfg(lat, nx, ny, nz, walls, precision)) as sim:
        sim.set_populations(_state(lat, nx, ny, nz, 5))
        for _ in range(2):
            of = oracle.fields(p, sim.get_populations())
            got = sim.fields()
            psi = torch.empty(N, dtype=torch.float64, device="cuda")
            u = torch.empty(3 * N, dtype=torch.float64, device="cuda")
            obs = sim.observables(psi_out=psi, u_out=u)
            assert np.array_equal(psi.cpu().numpy(), got["psi"])
            assert np.array_equal(u.cpu().numpy().reshape(3, N), got["u"])
            same = got["hit"] == of["hit"]
            assert same.mean() >= (1.0 if precision == lbnci.LB_FP64 else 0.98)
            for k in ("rho1", "rho2", "psi", "grad"):
                assert np.max(np.abs(got[k] - of[k].reshape(got[k].shape))) <= tol, k
            for k in ("frep", "u"):
                d = np.abs(got[k] - of[k].reshape(got[k].shape))[:, same]
                assert np.max(d) <= tol, k
            rho, un = got["rho1"] + got["rho2"], got["u"]
            sums = {"mass": [got["rho1"].sum(), got["rho2"].sum()], "momentum": (rho * un).sum(axis=1),
                    "flow_rate": (rho * un[0]).sum() / nx, "flow_rate_disp": (got["rho1"] * un[0]).sum() / nx}
            # rho of the kernels is the rounded sum of the components
            lim = (2.0 ** -24 if precision != lbnci.LB_FP64 else 1e-15) * 4 * (np.abs(rho * un).sum() + 1e-30)
            assert np.allclose(obs["mass"], sums["mass"], rtol=1e-13, atol=0)
            assert np.max(np.abs(obs["momentum"] - sums["momentum"])) <= lim
            assert abs(obs["flow_rate"] - sums["flow_rate"]) <= lim
            assert abs(obs["flow_rate_disp"] - sums["flow_rate_disp"]) <= lim
            assert obs["n_nci"] == int((got["hit"] > 0).sum()) and obs["n_bad"] == 0
            sim.step(1)


@pytest.mark.parametrize("precision", [lbnci.LB_FP32, lbnci.LB_FP16DEV])
@pytest.mark.parametrize("forcing", [lbnci.LB_FORCE_GUO, lbnci.LB_FORCE_EDM_DISPERSED])
@pytest.mark.parametrize("nx,ny,nz,walls", [(33, 9, 5, (1, 1)), (31, 7, 17, (0, 1)), (70, 20, 18, (1, 0)), (5, 3, 2, (0, 0))])
def test_ragged_ducts_equal_the_marching_step(nx, ny, nz, walls, forcing, precision, monkeypatch):
    """Lattices of no whole 32 x 8 columns: the streaming kernels on the two-population state give
    the marching kernel's populations (the same expressions on the same state)."""
    f = _state(lbnci.LB_D3Q27, nx, ny, nz, 6)
    cfg = _cfg(lbnci.LB_D3Q27, nx, ny, nz, walls, precision)
    cfg.forcing = forcing
    got = []
    for mode in ("", "march"):
        if mode:
            monkeypatch.setenv("LBNCI_D3_KERNEL", mode)
        else:
            monkeypatch.delenv("LBNCI_D3_KERNEL", raising=False)
        with lbnci.Sim(cfg) as sim:
            sim.set_populations(f)
            sim.step(3)
            got.append(sim.get_populations())
    assert np.array_equal(*got)


def test_fields_report_bad_sites_as_before():
    """NaN, infinite and negative densities are counted, whatever path the fields take."""
    for lat, dims in ((lbnci.LB_D2Q9, (40, 24, 1)), (lbnci.LB_D3Q27, (32, 8, 4))):
        for precision in (lbnci.LB_FP64, lbnci.LB_FP32):
            f = _state(lat, *dims, 8).reshape(2, -1, dims[0] * dims[1] * dims[2])
            f[0, 0, 5], f[1, 0, 77], f[0, 0, 100] = np.nan, np.inf, -50.0
            cfg = _cfg(lat, *dims, (1, 0), precision)
            with lbnci.Sim(cfg) as sim:
                sim.set_populations(f.ravel())
                o = sim.observables(allow_numeric=True)
            dt = torch.float64 if precision == lbnci.LB_FP64 else torch.float32
            ref = lbnci.lb_observables_noalloc(cfg, torch.tensor(f.ravel(), dtype=dt, device="cuda"),
                                               allow_numeric=True)
            assert o["n_bad"] == ref["n_bad"] >= 3
            assert o["n_interface"] == ref["n_interface"] and o["n_nci"] == ref["n_nci"]


@pytest.mark.parametrize("precision", [lbnci.LB_FP32, lbnci.LB_FP16DEV])
@pytest.mark.parametrize("nx,ny,wall", [(1, 1, 0), (3, 2, 1), (5, 9, 0), (33, 8, 1), (31, 40, 0), (130, 67, 1),
                                        (1030, 131, 1)])
def test_ragged_2d_passes_equal_the_one_pass_kernel(precision, nx, ny, wall, monkeypatch):
    """Bitwise, for both forcings, several rays and with the scratch or (the documented workspace)
    without: the passes evaluate the expressions of the fused D2Q9 kernel on every site."""
    f = torch.from_numpy(_state(lbnci.LB_D2Q9, nx, ny, 1, 7)).cuda()  # (a single site cannot be staged)
    for forcing in (lbnci.LB_FORCE_GUO, lbnci.LB_FORCE_EDM_DISPERSED):
        for A_h, h_max in ((0.05, 4.0), (0.05, 2.5), (0.0, 4.0)):
            cfg = _cfg(lbnci.LB_D2Q9, nx, ny, 1, (wall, 0), precision, A_h, h_max)
            cfg.forcing = forcing
            out = {}
            for mode in ("passes", "fused", "documented"):
                monkeypatch.delenv("LBNCI_FUSED_SPT", raising=False)
                monkeypatch.delenv("LBNCI_FUSED", raising=False)
                if mode == "fused":
                    monkeypatch.setenv("LBNCI_FUSED", "classic")
                cfg.workspace, cfg.workspace_bytes = None, 0
                with lbnci.Sim(cfg, workspace="torch" if mode == "documented" else None) as sim:
                    lbnci.lb_set_populations(sim.h, f)
                    before = sim.launches()
                    sim.step(3)
                    assert sim.launches() - before == (9 if mode == "passes" else 3)
                    assert sim.step_path() == lbnci.LB_PATH_FUSED2D
                    out[mode] = torch.empty_like(f)
                    lbnci.lb_get_populations(sim.h, out[mode])
            assert torch.equal(out["passes"], out["fused"])
            assert torch.equal(out["documented"], out["fused"])


@pytest.mark.parametrize("precision", [lbnci.LB_FP64, lbnci.LB_FP32, lbnci.LB_FP16DEV])
@pytest.mark.parametrize("lat,nx,ny,nz", [(lbnci.LB_D2Q9, 1, 8 * 65535 + 3, 1), (lbnci.LB_D3Q27, 3, 2, 65537)])
def test_lattices_longer_than_a_grid_axis(lat, nx, ny, nz, precision, monkeypatch):
    """Lattices that the passes' grids cannot hold step on the kernels that count blocks along x, as
    the environment variables select them: the same bits."""
    f = torch.from_numpy(_state(lat, nx, ny, nz, 5)).cuda()
    got = []
    for old in (False, True):
        for k, v in (("LBNCI_D3_KERNEL", "march"), ("LBNCI_FUSED", "classic")):
            monkeypatch.setenv(k, v) if old else monkeypatch.delenv(k, raising=False)
        with lbnci.Sim(_cfg(lat, nx, ny, nz, (1, int(nz > 1)), precision)) as sim:
            lbnci.lb_set_populations(sim.h, f)
            sim.step(2)
            got.append(torch.empty_like(f))
            lbnci.lb_get_populations(sim.h, got[-1])
            if nz > 1:
                o = sim.observables(allow_numeric=True)
                assert np.isfinite(o["mass"][0])
    assert torch.equal(got[0], got[1])
