"""Both kernels of the U-Net's convolutions against the oracle and exact sums: tcgen05.mma (the
default) and mma.sync (the kernel of operands that the other cannot take and of
LBNCI_UNET_MMA=sync), and networks whose batch changes from call to call (their launches are planned
per batch)."""
import numpy as np
import pytest

from oracle import unet_oracle as U
from paper_2003_11069_gb300 import inputs, unet

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [  # B, H, W, C_in, C_out, up: whole and cut tiles, one row, one tile, odd columns, many splits
    (1, 1, 128, 32, 32, 0), (2, 5, 128, 32, 32, 0), (1, 33, 256, 32, 64, 0), (1, 18, 130, 64, 32, 0),
    (1, 40, 384, 64, 32, 0), (3, 2, 254, 32, 96, 0), (1, 17, 40, 256, 128, 0), (1, 8, 34, 96, 160, 0),
    (1, 1, 2, 32, 32, 0), (4, 31, 31, 64, 64, 0), (2, 12, 256, 64, 32, 1), (1, 34, 200, 128, 64, 1),
    (1, 16, 36, 64, 32, 1), (1, 2, 2, 64, 64, 1), (3, 14, 34, 32, 32, 1),
]


def _integers(shape, g):
    return torch.randint(-2, 3, shape, device="cuda", generator=g).to(torch.bfloat16)


@pytest.mark.parametrize("mma", ["tcgen05", "sync"])
@pytest.mark.parametrize("B,H,W,Ci,Co,up", SHAPES)
def test_weight_gradient_of_small_integers_is_exact(B, H, W, Ci, Co, up, mma, monkeypatch):
    """Operands of -2 .. 2: every product and every partial sum is an integer of at most 4 P < 2^24, so
    FP32 sums are exact in any order and a pixel left out or taken twice shows."""
    assert 4 * B * H * W < 2 ** 24
    monkeypatch.setenv("LBNCI_UNET_MMA", mma)
    g = torch.Generator(device="cuda").manual_seed(B + 10 * H + W + Ci)
    hi, wi = (H // 2, W // 2) if up else (H, W)
    x, dy = _integers((B, hi, wi, Ci), g), _integers((B, H, W, Co), g)
    work = torch.empty(unet.conv3x3_wgrad_work(B, H, W, Ci, Co) // 4 + 1, device="cuda")
    dw, db = torch.full((Co * 9 * Ci,), 0.5, device="cuda"), torch.full((Co,), 0.5, device="cuda")
    unet.conv3x3_wgrad(x, Ci, B, H, W, Ci, up, dy, Co, Co, dw, db, work)
    xin = x.double().repeat_interleave(2, 1).repeat_interleave(2, 2) if up else x.double()
    xin = torch.cat([xin[:, :, -1:], xin, xin[:, :, :1]], 2)                      # periodic columns
    xin = torch.nn.functional.pad(xin, (0, 0, 0, 0, 1, 1))                        # zero rows
    for tap in range(9):
        xs = xin[:, tap // 3:tap // 3 + H, tap % 3:tap % 3 + W]
        exact = torch.einsum("bhwo,bhwc->oc", dy.double(), xs)
        assert torch.equal(dw.view(Co, 9, Ci)[:, tap].double(), exact), tap
    assert torch.equal(db.double(), dy.double().sum(dim=(0, 1, 2)))


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)


@pytest.mark.parametrize("levels,H,W", [(2, 16, 32), (4, 16, 32), (4, 32, 96)])
def test_network_of_the_default_kernels_against_the_oracle(levels, H, W, monkeypatch):
    """Output, loss and every gradient are as near to FP64 as BF16 storage permits: within 1.5x the
    distance of the oracle that rounds to BF16 where the network stores it, plus 1e-3."""
    monkeypatch.delenv("LBNCI_UNET_MMA", raising=False)
    B, lam = 2, [1.0, 0.5, 2.0]
    cfg = unet.make_config(levels=levels, base=32, H=H, W=W, max_batch=B)
    params = inputs.unet_params(U.layer_shapes(levels, 32, 5, 3), levels, bias_scale=0.05)
    rng = np.random.default_rng(levels + H)
    x, t = (rng.normal(size=(B, H, W, c)).astype(np.float32).astype(np.float64) for c in (5, 3))
    L_e, g_e, y_e = U.loss_and_grads(params, x, t, levels=levels, lam=lam, emulate_bf16=True)
    L_0, g_0, y_0 = U.loss_and_grads(params, x, t, levels=levels, lam=lam, emulate_bf16=False)
    with unet.Net(cfg) as net:
        net.set_params(unet.flatten(params))
        y = net.forward(x.astype(np.float32)).astype(np.float64)
        G = torch.zeros(net.nparams, device="cuda")
        L = net.loss_grad(torch.tensor(x, dtype=torch.float32, device="cuda"),
                          torch.tensor(t, dtype=torch.float32, device="cuda"), lam=lam, grads=G)
    assert _rel(y, y_0) <= 1.5 * _rel(y_e, y_0) + 1e-3
    assert abs(L - L_0) <= 1.5 * abs(L_e - L_0) + 1e-3 * L_0
    got = unet.unflatten(G.cpu().numpy().astype(np.float64), unet.layer_shapes(cfg))
    for k, ((gw, gb), (ew, eb), (rw, rb)) in enumerate(zip(got, g_e, g_0)):
        assert _rel(gw, rw) <= 1.5 * _rel(ew, rw) + 1e-3, ("weight", k)
        assert _rel(gb, rb) <= 1.5 * _rel(eb, rb) + 1e-3, ("bias", k)


def test_a_batch_that_changes_from_call_to_call(monkeypatch):
    """Outputs, loss and gradients of every call are those of a network made for it alone."""
    monkeypatch.delenv("LBNCI_UNET_MMA", raising=False)
    H, W, most = 24, 96, 5
    params = unet.flatten(inputs.unet_params(U.layer_shapes(3, 32, 5, 3), 4, bias_scale=0.05))
    g = torch.Generator(device="cuda").manual_seed(9)
    X = torch.randn((most, H, W, 5), device="cuda", generator=g)
    T = torch.randn((most, H, W, 3), device="cuda", generator=g)

    def both(net, B):
        y, G = torch.empty((B, H, W, 3), device="cuda"), torch.zeros(net.nparams, device="cuda")
        net.forward(X[:B], y)
        return y, net.loss_grad(X[:B], T[:B], grads=G), G

    def make():
        net = unet.Net(unet.make_config(levels=3, base=32, H=H, W=W, max_batch=most))
        net.set_params(params)
        return net
    with make() as net:
        for B in (most, 2, most, 1, 3, 2):
            y, loss, G = both(net, B)
            with make() as fresh:
                y1, loss1, G1 = both(fresh, B)
            assert torch.equal(y, y1) and loss == loss1 and torch.equal(G, G1), B
