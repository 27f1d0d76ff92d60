"""The workloads whose speed this framework is measured on, through its public entry points.

Every lattice case is what a simulation program does again and again: advance a lattice (or
an ensemble of lattices) by a number of steps, then read the observables, psi and u. Sizes and
parameters are those of this repository's benchmark, tests and warm-start study:

  droplet2d       the plain-method configuration, FP64: one droplet in a periodic box
  channel2d       packed-emulsion channels on D2Q9, from a test crop to the large channel
  duct3d          packed-emulsion square ducts on D3Q27, the benchmark's default workload
  ensemble        a batch of warm-start channels stepped together
  unet_forward    the surrogate's prediction for a batch of channels
  unet_train      loss and gradients of a training batch

Body forces are set from a Poiseuille velocity u_p (G = 8 rho nu u_p / ny^2), which keeps a
flow at low Mach number however long it runs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2003_11069_gb300 import inputs, lbnci, unet, warmstart

PRECISION = {"fp64": lbnci.LB_FP64, "fp32": lbnci.LB_FP32, "fp16dev": lbnci.LB_FP16DEV}
FORCING = {"guo": lbnci.LB_FORCE_GUO, "edm": lbnci.LB_FORCE_EDM_DISPERSED}
TAU, A_S, BETA, G_TH, H_MIN, H_MAX = 1.0, 0.01, 0.7, 0.05, 2.0, 4.0
NU = (TAU - 0.5) / 3.0
LAM = (0.2, 1.0, 1.0)  # channel weights of the warm-start study's loss


def _lb(kind, nx, ny, nz=1, precision="fp32", forcing="guo", steps=20, A_h=0.005, u_p=0.01):
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "forcing": forcing, "steps": steps,
            "A_h": A_h, "u_p": u_p}


def _net(kind, batch, H=64, W=256, levels=4, base=32):
    return {"kind": kind, "batch": batch, "H": H, "W": W, "levels": levels, "base": base}


def listed():
    cases = {
        # the plain-method FP64 run on its 128 x 128 periodic box: the smallest lattice, latency counts
        "droplet2d_fp64": _lb("droplet2d", 128, 128, precision="fp64", steps=100, A_h=0.05, u_p=0.0),
        # the 512 x 64 crop on which the long accuracy runs are made, 200 steps between two samples
        "channel2d_crop_fp32": _lb("channel2d", 512, 64, steps=200),
        # the soft-flowing-crystal channel of the benchmark (it fits in L2)
        "channel2d_fp32": _lb("channel2d", 2048, 256, steps=50),
        # the large channel (larger than L2) in FP16-deviation storage
        "channel2d_large_fp16dev": _lb("channel2d", 8192, 1024, precision="fp16dev", steps=20),
        # a channel whose length is no multiple of four, with the paper's own forcing
        "channel2d_ragged_edm_fp32": _lb("channel2d", 1030, 131, forcing="edm", steps=50),
        # a three-dimensional parity run in FP64
        "duct3d_fp64": _lb("duct3d", 128, 48, 48, precision="fp64", steps=10),
        # the benchmark's default: the large duct in FP16-deviation storage
        "duct3d_fp16dev": _lb("duct3d", 512, 128, 128, precision="fp16dev", steps=20, A_h=0.03),
        # the smaller duct in FP32 storage
        "duct3d_small_fp32": _lb("duct3d", 384, 96, 96, steps=20, A_h=0.03),
        # a duct of no whole columns, FP32
        "duct3d_ragged_fp32": _lb("duct3d", 150, 66, 66, steps=20, A_h=0.03),
        # the parameter study: 96 channels, lengths 512-1024, widths 64-96, stepped together
        "ensemble_fp32": {"kind": "ensemble", "members": 96, "precision": "fp32", "steps": 40},
        # prediction for a handful of channels
        "unet_forward_b8": _net("unet_forward", 8),
        # the study's training batch
        "unet_train_b32": _net("unet_train", 32),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["droplet2d", "channel2d", "channel2d", "channel2d", "duct3d", "duct3d", "duct3d", "ensemble",
                       "unet_forward", "unet_train"])
    if kind == "ensemble":
        return {"kind": kind, "members": _log(rng, 4, 96), "precision": rng.choice(["fp32", "fp32", "fp16dev"]),
                "steps": rng.randint(20, 40)}
    if kind.startswith("unet"):
        return _net(kind, _log(rng, 1, 32), H=8 * rng.randint(4, 8), W=8 * rng.randint(12, 32),
                    levels=rng.choice([3, 4, 4]))
    precision = rng.choice(["fp32", "fp32", "fp16dev", "fp64"])
    forcing = rng.choice(["guo", "guo", "guo", "edm"])
    A_h = rng.choice([0.0, 0.005, 0.01])
    if kind == "droplet2d":
        n = _log(rng, 96, 512)
        return _lb(kind, n, n + rng.randint(-8, 8), precision=precision, forcing=forcing, steps=rng.randint(50, 150),
                   A_h=A_h, u_p=0.0)
    if kind == "channel2d":
        nx, ny = _log(rng, 256, 8192), _log(rng, 64, 1024)
        if rng.random() < 0.6:
            nx = (nx + 31) // 32 * 32
        if precision == "fp64":
            nx, ny = min(nx, 1000), min(ny, 150)
        steps = max(10, min(200, int(1.6e8 / (nx * ny))))
        if precision == "fp64":
            steps = min(steps, 30)
        return _lb(kind, nx, ny, precision=precision, forcing=forcing, steps=steps, A_h=A_h,
                   u_p=rng.uniform(0.002, 0.02))
    nx, ny, nz = _log(rng, 64, 512), _log(rng, 32, 128), _log(rng, 32, 128)
    if rng.random() < 0.6:
        nx, ny = (nx + 31) // 32 * 32, (ny + 7) // 8 * 8
    if precision == "fp64":
        nx, ny, nz = min(nx, 150), min(ny, 48), min(nz, 48)
    return _lb(kind, nx, ny, nz, precision=precision, forcing=forcing, steps=rng.randint(8, 10 if precision == "fp64"
                                                                                         else 20), A_h=A_h,
               u_p=rng.uniform(0.002, 0.02))


# ------------------------------------------------------------------ inputs
def _force(c):
    return 0.0 if c["kind"] == "droplet2d" else 8.0 * NU * c["u_p"] / c["ny"] ** 2


def _lattice_fields(c, seed):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    rng = np.random.default_rng(seed)
    if c["kind"] == "droplet2d":
        ctr = (nx / 2 + rng.uniform(-2, 2), ny / 2 + rng.uniform(-2, 2), 0.0)
        fl = inputs.droplet(nx, ny, radius=0.234 * min(nx, ny) * rng.uniform(0.95, 1.05), center=ctr)
    elif c["kind"] == "duct3d":
        fl = inputs.duct_emulsion_3d(nx, ny, nz, seed=seed)
    else:
        # long channels are periods of a shorter one, side by side (the flow is periodic along x)
        k = 4 if nx % 4 == 0 and nx * ny > 2_000_000 else 1
        fl = inputs.channel_emulsion_2d(nx // k, ny, seed=seed)
        if k > 1:
            fl = inputs.Fields(nx, ny, 1, *(np.tile(r.reshape(ny, nx // k), (1, k)).ravel()
                                            for r in (fl.rho1, fl.rho2)))
    return fl


def _ensemble_channels(c, seed):
    """One study's channels (sizes and parameters); the seed packs the droplets."""
    chs = warmstart.channels(c["members"], 20, ah_range=(0.0, 0.01))
    for k, ch in enumerate(chs):
        ch.fields = inputs.channel_emulsion_2d(ch.nx, ch.ny, seed=seed + 1000 * k, area_fraction=ch.area_fraction)
    return chs


def _unet_data(c, seed):
    """Features of warm-start channels, targets of their shape (psi and a flow profile) and parameters."""
    chs = warmstart.channels(c["batch"], seed)
    X = np.stack([warmstart.features(ch, c["H"], c["W"]) for ch in chs])
    rng = np.random.default_rng(seed + 1)
    y = (np.arange(c["H"]) + 0.5) / c["H"]
    prof = (4.0 * y * (1.0 - y))[None, :, None].astype(np.float32)
    T = np.empty(X.shape[:3] + (3,), np.float32)
    T[..., 0] = X[..., 1]
    T[..., 1] = prof * (0.8 + 0.2 * X[..., 1])
    T[..., 2] = 0.05 * rng.standard_normal(X.shape[:3]).astype(np.float32)
    shapes = _unet_shapes(c)
    return X, T, unet.flatten(inputs.unet_params([("", s) for s in shapes], seed + 2))


def _unet_shapes(c):
    C = [c["base"] << k for k in range(c["levels"])]
    out, cin = [], 5
    for w in C:
        out += [(w, 3, 3, cin), (w, 3, 3, w)]
        cin = w
    for k in range(c["levels"] - 2, -1, -1):
        out += [(C[k], 3, 3, C[k + 1]), (C[k], 3, 3, 2 * C[k]), (C[k], 3, 3, C[k])]
    return out + [(3, C[0])]


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind.startswith("unet"):
        X, T, params = _unet_data(c, seed)
        net = unet.Net(unet.make_config(levels=c["levels"], base=c["base"], H=c["H"], W=c["W"], max_batch=c["batch"]))
        net.set_params(params)
        s = {"kind": kind, "net": net, "X": torch.tensor(X, device="cuda")}
        if kind == "unet_forward":
            s["y"] = torch.empty((c["batch"], c["H"], c["W"], 3), device="cuda")
        else:
            s["T"], s["grads"] = torch.tensor(T, device="cuda"), torch.empty(net.nparams, device="cuda")
        return s
    if kind == "ensemble":
        chs = _ensemble_channels(c, seed)
        ens = lbnci.Ensemble([warmstart._config(ch, precision=PRECISION[c["precision"]]) for ch in chs])
        for m, ch in zip(ens.members, chs):
            m.init_fields(ch.fields.rho1, ch.fields.rho2)
        ens.tune()
        N = [m.N for m in ens.members]
        psi, u = (torch.empty(k * sum(N), dtype=torch.float64, device="cuda") for k in (1, 3))
        return {"kind": kind, "ens": ens, "steps": c["steps"], "psi": psi, "u": u, "psi_of": psi.split(N),
                "u_of": u.split([3 * n for n in N])}
    fl = _lattice_fields(c, seed)
    three = kind == "duct3d"
    cfg = lbnci.lb_config_make(lattice=lbnci.LB_D3Q27 if three else lbnci.LB_D2Q9, nx=c["nx"], ny=c["ny"], nz=c["nz"],
                               wall_y=int(kind != "droplet2d"), wall_z=int(three), tau=TAU, A_s=A_S, beta=BETA,
                               A_h=c["A_h"], h_min=H_MIN, h_max=H_MAX, g_th=G_TH, force=(_force(c), 0.0, 0.0),
                               precision=PRECISION[c["precision"]], forcing=FORCING[c["forcing"]])
    sim = lbnci.Sim(cfg)
    sim.init_fields(fl.rho1, fl.rho2)
    return {"kind": kind, "sim": sim, "steps": c["steps"], "fp64": c["precision"] == "fp64",
            "psi": torch.empty(sim.N, dtype=torch.float64, device="cuda"),
            "u": torch.empty(3 * sim.N, dtype=torch.float64, device="cuda")}


def run(state):
    s, kind = state, state["kind"]
    if kind == "unet_forward":
        return s["net"].forward(s["X"], s["y"])
    if kind == "unet_train":
        loss = s["net"].loss_grad(s["X"], s["T"], lam=LAM, grads=s["grads"])
        return {"loss": loss, "grads": s["grads"]}
    if kind == "ensemble":
        s["ens"].step(s["steps"])
        obs = [m.observables(psi_out=p, u_out=u, allow_numeric=True)
               for m, p, u in zip(s["ens"].members, s["psi_of"], s["u_of"])]
        # the fields of an FP32 lattice are FP32 numbers: a study keeps them as such
        return {"psi": s["psi"].float(), "u": s["u"].float(), "flow": _flow(obs)}
    s["sim"].step(s["steps"])
    o = s["sim"].observables(psi_out=s["psi"], u_out=s["u"], allow_numeric=True)
    out = {"psi": s["psi"], "u": s["u"]} if s["fp64"] else {"psi": s["psi"].float(), "u": s["u"].float()}
    out.update(mass=o["mass"], counts=np.array([o["n_interface"], o["n_nci"], o["n_bad"]]))
    if kind != "droplet2d":  # nothing drives the droplet: its flow rate is rounding
        out["flow"] = _flow([o])
    return out


def _flow(obs):
    return np.array([[o["flow_rate"], o["flow_rate_disp"]] for o in obs])


# ------------------------------------------------------------------ what a pass cannot do without
# bytes of state per site: two components' populations, or, on D3Q27 with Guo forcing below
# FP64, the totals, two rest populations and the four recolouring coefficients
_STATE = {("2d", "fp64"): 144, ("2d", "fp32"): 72, ("2d", "fp16dev"): 44, ("3d", "fp64"): 432, ("3d", "fp32"): 128,
          ("3d", "fp16dev"): 76, ("3d-edm", "fp64"): 432, ("3d-edm", "fp32"): 216, ("3d-edm", "fp16dev"): 116}


def _conv_layers(c):
    """(pixels, C_in, C_out) of the 3x3 convolutions, first layer first."""
    C, P = [c["base"] << k for k in range(c["levels"])], c["batch"] * c["H"] * c["W"]
    out, cin = [], 5
    for k, w in enumerate(C):
        out += [(P >> 2 * k, cin, w), (P >> 2 * k, w, w)]
        cin = w
    for k in range(c["levels"] - 2, -1, -1):
        out += [(P >> 2 * k, C[k + 1], C[k]), (P >> 2 * k, 2 * C[k], C[k]), (P >> 2 * k, C[k], C[k])]
    return out


def work(case):
    c, kind = case, case["kind"]
    if kind.startswith("unet"):
        P, L = c["batch"] * c["H"] * c["W"], _conv_layers(c)
        params = sum(9 * i * o + o for _, i, o in L) + 3 * c["base"] + 3
        fwd = sum(2 * 9 * p * i * o for p, i, o in L) + 2 * P * 3 * c["base"]
        if kind == "unet_forward":
            return {"bytes": P * (5 + 3) * 4 + 2 * params, "flops": fwd}
        acts = 2 * sum(p * o for p, _, o in L)  # BF16 activations: written, read again by the backward pass
        return {"bytes": P * (5 + 3) * 4 + 8 * params + 2 * acts, "flops": 3 * fwd - 2 * 9 * L[0][0] * 5 * c["base"]}
    if kind == "ensemble":  # 768 x 80 sites a channel in the mean
        N, d = 768 * 80 * c["members"], "2d"
    else:
        N, d = c["nx"] * c["ny"] * c["nz"], "3d" if kind == "duct3d" else "2d"
        d += "-edm" if d == "3d" and c["forcing"] == "edm" else ""
    per_site = 2 * _STATE[d, c["precision"]]
    out = 32 if c["precision"] == "fp64" else 16
    return {"bytes": N * (c["steps"] * per_site + per_site // 2 + out),
            "flops": N * c["steps"] * (400 if d == "2d" else 1000)}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _exact_lattice(D, nx, ny, nz, walls, G, A_h, forcing, rho1, rho2, steps):
    """Colour-gradient lattice Boltzmann with near-contact forces, from densities at rest."""
    dev, Q, w_of = _dev(), 3 ** D, (4 / 9, 1 / 9, 1 / 36) if D == 2 else (8 / 27, 2 / 27, 1 / 54, 1 / 216)
    cs = [tuple((0, 1, -1)[i // 3 ** a % 3] for a in range(3)) for i in range(Q)]
    w = [w_of[sum(v * v for v in c)] for c in cs]
    opp = [cs.index(tuple(-v for v in c)) for c in cs]
    shape, smax = (nz, ny, nx), int(H_MAX) if A_h > 0 else 0
    r0 = [torch.as_tensor(r, device=dev).reshape(shape) for r in (rho1, rho2)]
    f = [[w[i] * r for i in range(Q)] for r in r0]

    def pull(fk):
        out = []
        for i, c in enumerate(cs):
            t = torch.roll(fk[i], (c[2], c[1], c[0]), (0, 1, 2))
            for axis, comp, wall in ((1, c[1], walls[0]), (0, c[2], walls[1])):
                if wall and comp:  # halfway bounce-back: the site's own opposite population
                    at = (slice(None),) * axis + ((0 if comp > 0 else shape[axis] - 1),)
                    t[at] = fk[opp[i]][at]
            out.append(t)
        return out

    def pad(a, axis, wall):
        n = a.shape[axis]
        lo, hi = (0, n - 1) if wall else (n - 1, 0)
        return torch.cat([a.narrow(axis, lo, 1), a, a.narrow(axis, hi, 1)], axis)

    def dot(c, v):
        r = 0.0
        for a in range(D):
            if c[a]:
                r = r + c[a] * v[a]
        return r

    def macro(fp):
        rho = [sum(fp[k]) for k in (0, 1)]
        rt = rho[0] + rho[1]
        psi = (rho[0] - rho[1]) / rt
        pp = pad(pad(pad(psi, 2, False), 1, walls[0]), 0, walls[1])
        grad = [torch.zeros_like(psi) for _ in range(3)]
        for i, c in enumerate(cs):
            v = pp[1 + c[2]:1 + c[2] + nz, 1 + c[1]:1 + c[1] + ny, 1 + c[0]:1 + c[0] + nx]
            for a in range(D):
                if c[a]:
                    grad[a] += 3.0 * w[i] * c[a] * v
        g = (grad[0] ** 2 + grad[1] ** 2 + grad[2] ** 2).sqrt()
        m = [torch.where(g > 0, q / torch.where(g > 0, g, 1.0), 0.0) for q in grad]
        A = torch.zeros_like(psi)
        if smax:
            z, y, x = (g > G_TH).nonzero(as_tuple=True)
            n, gs = [-q[z, y, x] for q in m], g[z, y, x]
            As, live = torch.zeros_like(gs), torch.ones_like(gs, dtype=torch.bool)
            for s in range(1, smax + 1):
                d = [torch.sign(q) * torch.floor((s * q).abs() + 0.5) for q in n]
                px, py, pz = (x + d[0].long()) % nx, y + d[1].long(), z + d[2].long()
                for q, hi, wall in ((py, ny, walls[0]), (pz, nz, walls[1])):
                    if wall:
                        live &= (q >= 0) & (q < hi)
                py, pz = py % ny, pz % nz
                facing = -sum(m[a][pz, py, px] * n[a] for a in range(D)) < 0
                found = live & (g[pz, py, px] > G_TH) & facing
                As[found] = A_h if s <= H_MIN else A_h * (H_MIN / s) ** 3
                live &= ~found
            A[z, y, x] = As
        F = [G[a] + A * m[a] * 0.5 * g for a in range(3)]
        tot = [a + b for a, b in zip(*fp)]
        j = [sum((c[a] * t for c, t in zip(cs, tot) if c[a]), torch.zeros_like(psi)) for a in range(3)]
        u = [(j[a] + 0.5 * F[a]) / rt for a in range(3)]
        return rho, rt, psi, m, g, F, j, u, tot

    def feq(i, rho, v):
        cv = dot(cs[i], v)
        return w[i] * rho * (1 + 3 * cv + 4.5 * cv * cv - 1.5 * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2))

    om = 1.0 / TAU
    for _ in range(steps):
        fp = [pull(fk) for fk in f]
        rho, rt, _, m, g, F, j, u, tot = macro(fp)
        del fp
        uF = sum(u[a] * F[a] for a in range(3))
        seg = BETA * rho[0] * rho[1] / rt
        if forcing == "edm":
            ue = [j[a] / rt for a in range(3)]
            inv = [torch.where(r > 0, 1.0 / torch.where(r > 0, r, 1.0), 0.0) for r in rho]
            uk = [[ue[a] + (G[a] * rho[k] / rt + (F[a] - G[a] if k == 0 else 0.0)) * inv[k] for a in range(3)]
                  for k in (0, 1)]
        for i in range(Q):
            c = cs[i]
            cm = dot(c, m)
            if forcing == "edm":
                fs = tot[i] - om * (tot[i] - feq(i, rt, ue))
            else:
                cF = dot(c, F)
                fs = tot[i] - om * (tot[i] - feq(i, rt, u))
                fs = fs + (1 - 0.5 * om) * w[i] * (3 * (cF - uF) + 9 * dot(c, u) * cF)
            fs = fs + A_S * g * (w[i] * cm * cm - w[i] / 3)
            rc = seg * w[i] * (cm / math.sqrt(max(1, sum(v * v for v in c))))
            f[0][i], f[1][i] = rho[0] / rt * fs + rc, rho[1] / rt * fs - rc
            if forcing == "edm":
                for k in (0, 1):
                    f[k][i] = f[k][i] + feq(i, rho[k], uk[k]) - feq(i, rho[k], ue)
    rho, rt, psi, _, _, _, _, u, _ = macro([pull(fk) for fk in f])
    flow = [float((r * u[0]).sum()) / nx for r in (rt, rho[0])]
    return psi.reshape(-1), torch.stack(u).reshape(-1), [float(r.sum()) for r in rho], flow


def _exact_unet(c, X, T, params, grads):
    dev, shapes = _dev(), _unet_shapes(c)
    flat = torch.as_tensor(params, device=dev).double().requires_grad_(grads)
    layers, at = [], 0
    for s in shapes:
        n = math.prod(s)
        wt = flat[at:at + n].reshape(s)
        layers.append((wt.permute(0, 3, 1, 2) if len(s) == 4 else wt[:, :, None, None], flat[at + n:at + n + s[0]]))
        at += n + s[0]
    nn = torch.nn.functional

    def forward(x):
        it = iter(layers)

        def conv(h):
            wt, b = next(it)
            return torch.relu(nn.conv2d(nn.pad(h, (1, 1, 0, 0), mode="circular"), wt, b, padding=(1, 0)))
        skips, h = [], x.permute(0, 3, 1, 2)
        for k in range(c["levels"]):
            h = conv(conv(h))
            if k < c["levels"] - 1:
                skips.append(h)
                h = nn.max_pool2d(h, 2)
        for skip in reversed(skips):
            h = conv(nn.interpolate(h, scale_factor=2, mode="nearest"))
            h = conv(conv(torch.cat([h, skip], 1)))
        wt, b = next(it)
        return nn.conv2d(h, wt, b).permute(0, 2, 3, 1)

    X, T = (torch.as_tensor(a, device=dev).double() for a in (X, T))
    if not grads:
        return torch.cat([forward(x) for x in X.split(4)])
    lam, total = torch.tensor(LAM, dtype=torch.float64, device=dev), 0.0
    for x, t in zip(X.split(4), T.split(4)):
        loss = (lam * (forward(x) - t) ** 2).sum() / (X.shape[0] * X.shape[1] * X.shape[2])
        loss.backward()
        total += float(loss.detach())
    return {"loss": np.float64(total), "grads": flat.grad}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind.startswith("unet"):
        with torch.set_grad_enabled(kind == "unet_train"):
            return _exact_unet(c, *_unet_data(c, seed), kind == "unet_train")
    with torch.no_grad():
        if kind == "ensemble":
            got = [_exact_lattice(2, ch.nx, ch.ny, 1, (1, 0), (ch.force, 0.0, 0.0), ch.A_h, "guo", ch.fields.rho1,
                                  ch.fields.rho2, c["steps"]) for ch in _ensemble_channels(c, seed)]
            return {"psi": torch.cat([g[0] for g in got]), "u": torch.cat([g[1] for g in got]),
                    "flow": np.array([g[3] for g in got])}
        fl, three = _lattice_fields(c, seed), kind == "duct3d"
        psi, u, mass, flow = _exact_lattice(3 if three else 2, c["nx"], c["ny"], c["nz"],
                                            (int(kind != "droplet2d"), int(three)), (_force(c), 0.0, 0.0), c["A_h"],
                                            c["forcing"], fl.rho1, fl.rho2, c["steps"])
        return {"psi": psi, "u": u, "mass": np.array(mass), "counts": None,
                "flow": None if kind == "droplet2d" else np.array([flow])}
