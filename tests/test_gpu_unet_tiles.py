"""The tensor-memory convolutions (csrc/unet_conv.cuh) at the edges of their tiles: strips of whole
rows, patches and linear tiles, partial strips, one-row and odd images, periodic columns on both
sides, upsampled inputs, channel slices. The convolution adds the same products in the same order
as the mma.sync kernel, so outputs are compared bit for bit; weight gradients are sums of P products
(P pixels), exact in FP32 up to the summation: |got - exact| <= P 2^-23 sum|terms|, as for the other
kernel; a network's gradients under both kernels differ by that rounding alone."""
import numpy as np
import pytest

from oracle import unet_oracle as U
from paper_2003_11069_gb300 import inputs, unet

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [  # B, H, W, C_in, C_out, up, x padding, y padding
    (1, 1, 128, 32, 32, 0, 0, 0), (2, 5, 128, 32, 32, 0, 32, 64), (1, 33, 256, 32, 64, 0, 0, 0),
    (1, 18, 130, 64, 32, 0, 0, 0), (2, 3, 100, 64, 64, 0, 0, 64), (1, 40, 384, 64, 32, 0, 64, 0),
    (1, 7, 200, 128, 64, 0, 0, 0), (1, 4, 96, 128, 32, 0, 0, 0), (3, 2, 254, 32, 96, 0, 0, 0),
    (1, 2, 256, 64, 32, 1, 0, 32), (2, 12, 256, 64, 32, 1, 0, 0), (1, 34, 200, 128, 64, 1, 0, 0),
    (1, 6, 512, 64, 64, 1, 0, 0), (2, 16, 64, 128, 128, 0, 0, 0), (1, 17, 40, 256, 128, 0, 0, 0),
    (1, 8, 34, 96, 160, 0, 0, 0), (2, 32, 48, 32, 64, 0, 0, 0), (1, 16, 36, 64, 32, 1, 0, 0),
    (1, 1, 2, 32, 32, 0, 0, 0), (1, 64, 8, 512, 64, 0, 0, 0),
]


def _data(B, H, W, Ci, Co, up, xp, yp, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed + 100 * H + W + Ci)
    hi, wi = (H // 2, W // 2) if up else (H, W)
    x = torch.randn((B, hi, wi, Ci + xp), device="cuda", generator=g).to(torch.bfloat16)
    w = (torch.randn((Co, 9, Ci), device="cuda", generator=g) / (3 * Ci ** 0.5)).to(torch.bfloat16)
    b = torch.randn(Co, device="cuda", generator=g)
    return x, w, b


@pytest.mark.parametrize("B,H,W,Ci,Co,up,xp,yp", SHAPES)
def test_convolution_bits_equal_mma_sync(B, H, W, Ci, Co, up, xp, yp, monkeypatch):
    x, w, b = _data(B, H, W, Ci, Co, up, xp, yp)
    out = []
    for mma in ("tcgen05", "sync"):
        monkeypatch.setenv("LBNCI_UNET_MMA", mma)
        for relu, bias in ((1, b), (0, None)):
            y = torch.full((B, H, W, Co + yp), 7.0, device="cuda", dtype=torch.bfloat16)
            unet.conv3x3(x, Ci + xp, B, H, W, Ci, up, w, bias, relu, y, Co + yp, Co)
            out.append(y)
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3])


@pytest.mark.parametrize("B,H,W,Ci,Co,up", [s[:6] for s in SHAPES if s[3] <= 256])
def test_weight_gradient(B, H, W, Ci, Co, up):
    x, _, _ = _data(B, H, W, Ci, Co, up, 0, 0, seed=3)
    dy = torch.randn((B, H, W, Co), device="cuda").to(torch.bfloat16)
    work = torch.empty(unet.conv3x3_wgrad_work(B, H, W, Ci, Co) // 4 + 1, device="cuda")
    dw, db = torch.zeros(Co * 9 * Ci, device="cuda"), torch.zeros(Co, device="cuda")
    unet.conv3x3_wgrad(x, Ci, B, H, W, Ci, up, dy, Co, Co, dw, db, work)
    xin = x.double().repeat_interleave(2, 1).repeat_interleave(2, 2) if up else x.double()
    xin = torch.cat([xin[:, :, -1:], xin, xin[:, :, :1]], 2)                      # periodic columns
    xin = torch.nn.functional.pad(xin, (0, 0, 0, 0, 1, 1))                        # zero rows
    for tap in range(9):
        xs = xin[:, tap // 3:tap // 3 + H, tap % 3:tap % 3 + W]
        exact = torch.einsum("bhwo,bhwc->oc", dy.double(), xs)
        scale = torch.einsum("bhwo,bhwc->oc", dy.double().abs(), xs.abs())
        got = dw.view(Co, 9, Ci)[:, tap].double()
        assert bool(((got - exact).abs() <= B * H * W * 2.0 ** -23 * scale).all()), tap
    d = dy.double().sum(dim=(0, 1, 2))
    assert bool(((db.double() - d).abs() <= B * H * W * 2.0 ** -23 * dy.double().abs().sum(dim=(0, 1, 2))).all())


@pytest.mark.parametrize("H,W,B,levels", [(32, 256, 2, 3), (16, 200, 1, 2), (24, 96, 3, 3)])
def test_network_outputs_equal_and_gradients_agree(H, W, B, levels, monkeypatch):
    """The whole network, whose layers take every kind of tile and whose data gradients carry the
    ReLU masks: outputs bit for bit; gradients to the rounding of their FP32 sums (2^-23 per term
    relative to sum|terms|, which a gradient of random data exceeds by at most sqrt(P) ~ 100)."""
    cfg = unet.make_config(levels=levels, base=32, H=H, W=W, max_batch=B)
    params = unet.flatten(inputs.unet_params(U.layer_shapes(levels, 32, 5, 3), 4, bias_scale=0.05))
    g = torch.Generator(device="cuda").manual_seed(9)
    X = torch.randn((B, H, W, 5), device="cuda", generator=g)
    T = torch.randn((B, H, W, 3), device="cuda", generator=g)
    got = []
    for mma in ("tcgen05", "sync"):
        monkeypatch.setenv("LBNCI_UNET_MMA", mma)
        with unet.Net(cfg) as net:
            net.set_params(params)
            y = torch.empty((B, H, W, 3), device="cuda")
            net.forward(X, y)
            G, G2 = torch.zeros(net.nparams, device="cuda"), torch.zeros(net.nparams, device="cuda")
            loss = net.loss_grad(X, T, grads=G)
            net.loss_grad(X, T, grads=G2)
            torch.cuda.synchronize()
            assert torch.equal(G, G2)
            got.append((y, loss, G))
    assert torch.equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
    a, b = got[0][2].double(), got[1][2].double()
    assert float((a - b).norm() / b.norm()) <= 100 * 2.0 ** -23


@pytest.mark.parametrize("out_ch", [1, 2, 5, 8])
def test_head_gradient_for_other_output_counts(out_ch):
    """The 1x1 head's weight and bias gradients (the last layer's) from the activations' own
    gradient identity: dL/db = sum dy and, with the head's weights scaled, dL/dy . y = sum over the
    head's weights and biases of theta dL/dtheta (y is linear in them); FP32 sums of P = 1152
    terms, 2^-23 each relative to sum|terms|, which random data exceeds the sum of by about 100."""
    H, W, B = 16, 24, 3
    cfg = unet.make_config(levels=2, base=32, out_ch=out_ch, H=H, W=W, max_batch=B)
    shapes = U.layer_shapes(2, 32, 5, out_ch)
    params = unet.flatten(inputs.unet_params(shapes, 4, bias_scale=0.05))
    g = torch.Generator(device="cuda").manual_seed(9)
    X = torch.randn((B, H, W, 5), device="cuda", generator=g)
    T = torch.randn((B, H, W, out_ch), device="cuda", generator=g)
    with unet.Net(cfg) as net:
        net.set_params(params)
        y = torch.empty((B, H, W, out_ch), device="cuda")
        net.forward(X, y)
        G = torch.zeros(net.nparams, device="cuda")
        net.loss_grad(X, T, grads=G)
        torch.cuda.synchronize()
    gw, gb = unet.unflatten(G.cpu().numpy().astype(np.float64), unet.layer_shapes(cfg))[-1]
    w, b = unet.unflatten(np.asarray(params, dtype=np.float32).astype(np.float64), unet.layer_shapes(cfg))[-1]
    w = torch.from_numpy(np.ascontiguousarray(w)).float().bfloat16().double().numpy()  # the head multiplies BF16 weights
    dy = (2.0 / (B * H * W) * (y.double() - T.double())).reshape(-1, out_ch).cpu().numpy()
    tol = 100 * 2.0 ** -23
    assert np.all(np.abs(gb - dy.sum(0)) <= tol * np.abs(dy).sum(0))
    terms = dy * (y.double().reshape(-1, out_ch).cpu().numpy() - np.asarray(b))
    assert np.all(np.abs((gw * w).reshape(out_ch, -1).sum(1) - terms.sum(0)) <= tol * (np.abs(terms).sum(0) +
                                                                                     np.abs(gw * w).reshape(out_ch, -1).sum(1)))
