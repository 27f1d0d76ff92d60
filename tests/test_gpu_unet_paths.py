"""Which kernel a single U-Net convolution or weight gradient takes, and that each of them is right:
tcgen05.mma with operands copied by TMA is the default, mma.sync (csrc/unet_kernels.cuh) the kernel
of operands that it cannot take and of LBNCI_UNET_MMA=sync."""
import pytest

from oracle import unet_oracle as U
from paper_2003_11069_gb300 import inputs, lbnci, unet

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _wgrad(x, dy, up, work_offset=0):
    """dw and db of x [B][h][w][C_in] and dy [B][H][W][C_out], with the scratch work_offset bytes
    into an allocation (whose own alignment is 256)."""
    B, H, W, Co = dy.shape
    Ci = x.shape[3]
    n = unet.conv3x3_wgrad_work(B, H, W, Ci, Co)
    raw = torch.empty(n + 64, device="cuda", dtype=torch.uint8)
    work = raw[work_offset:work_offset + n]
    assert work.data_ptr() % 16 == work_offset % 16
    dw, db = torch.full((Co * 9 * Ci,), 7.0, device="cuda"), torch.full((Co,), 7.0, device="cuda")
    unet.conv3x3_wgrad(x, Ci, B, H, W, Ci, up, dy, Co, Co, dw, db, work)
    torch.cuda.synchronize()
    return dw, db


@pytest.mark.parametrize("B,H,W,Ci,Co,up", [(2, 9, 40, 32, 32, 0), (3, 16, 64, 64, 128, 0), (2, 18, 36, 64, 32, 1)])
def test_weight_gradient_scratch_of_eight_byte_alignment(B, H, W, Ci, Co, up, monkeypatch):
    """The tcgen05 reduction loads 16-byte pieces of the scratch: at an offset of 8 bytes the mma.sync
    kernel runs instead (the same bits as LBNCI_UNET_MMA=sync selects), at 16 the tcgen05 kernel (the
    bits of an aligned scratch)."""
    g = torch.Generator(device="cuda").manual_seed(5)
    hi, wi = (H // 2, W // 2) if up else (H, W)
    x = torch.randn((B, hi, wi, Ci), device="cuda", generator=g).to(torch.bfloat16)
    dy = torch.randn((B, H, W, Co), device="cuda", generator=g).to(torch.bfloat16)
    monkeypatch.delenv("LBNCI_UNET_MMA", raising=False)
    tc, at8, at16 = _wgrad(x, dy, up), _wgrad(x, dy, up, 8), _wgrad(x, dy, up, 16)
    monkeypatch.setenv("LBNCI_UNET_MMA", "sync")
    sync = _wgrad(x, dy, up)
    assert torch.equal(at8[0], sync[0]) and torch.equal(at8[1], sync[1])
    assert torch.equal(at16[0], tc[0]) and torch.equal(at16[1], tc[1])
    assert not torch.equal(tc[0], sync[0])  # the two kernels add in different orders


def _net(B=2, seed=3):
    cfg = unet.make_config(levels=2, base=32, H=16, W=32, max_batch=B)
    net = unet.Net(cfg)
    net.set_params(unet.flatten(inputs.unet_params(U.layer_shapes(2, 32, 5, 3), seed, bias_scale=0.05)))
    g = torch.Generator(device="cuda").manual_seed(seed)
    return net, torch.randn((B, 16, 32, 5), device="cuda", generator=g), torch.randn((B, 16, 32, 3), device="cuda", generator=g)


def test_an_expired_wait_is_reported_to_its_own_network(monkeypatch):
    """LBNCI_UNET_FAIL_TEST=1 sets the error word from the host as a kernel whose wait ran out would
    (no wait is made to run out). The network whose launch it was reports it once, at its next call
    that synchronises; another network, called before, does not; no update is applied meanwhile, and
    the updates that follow are those of a network that never failed."""
    monkeypatch.delenv("LBNCI_UNET_MMA", raising=False)
    (a, X, T), (b, _, _), (c, _, _) = _net(), _net(), _net()
    Y = torch.empty((2, 16, 32, 3), device="cuda")
    with a, b, c:
        start = a.get_params()
        monkeypatch.setenv("LBNCI_UNET_FAIL_TEST", "1")
        a.forward(X, Y)                      # device output: not synchronised, not checked
        monkeypatch.delenv("LBNCI_UNET_FAIL_TEST")
        b.forward(X.cpu().numpy())           # checked: not b's
        assert b.loss_grad(X, T) > 0
        for _ in range(2):
            a.train_step(X, T)               # the word is set: left out
        assert (a.get_params() == start).all()
        with pytest.raises(lbnci.LBError, match="2 parameter updates left out"):
            a.loss_grad(X, T)
        for _ in range(3):                   # cleared; Adam goes on at its first step
            assert a.train_step(X, T, want_loss=True) == c.train_step(X, T, want_loss=True)
        assert (a.get_params() == c.get_params()).all()
        assert not (a.get_params() == start).all()


def test_an_expired_wait_of_a_single_call_is_told_apart(monkeypatch):
    """The next synchronising network call reports it with its own results complete."""
    monkeypatch.delenv("LBNCI_UNET_MMA", raising=False)
    x = torch.zeros((1, 8, 16, 32), device="cuda", dtype=torch.bfloat16)
    w, y = torch.zeros((32, 9, 32), device="cuda", dtype=torch.bfloat16), torch.empty_like(x)
    net, X, T = _net()
    with net:
        loss = net.loss_grad(X, T)
        monkeypatch.setenv("LBNCI_UNET_FAIL_TEST", "1")
        unet.conv3x3(x, 32, 1, 8, 16, 32, 0, w, None, 0, y, 32, 32)
        monkeypatch.delenv("LBNCI_UNET_FAIL_TEST")
        torch.cuda.synchronize()
        with pytest.raises(lbnci.LBError, match="single convolution"):
            net.loss_grad(X, T)
        assert net.loss_grad(X, T) == loss


@pytest.mark.parametrize("B,H,W,Ci,Co,up", [(2, 17, 32, 32, 32, 0), (1, 10, 40, 64, 64, 0), (2, 18, 36, 64, 32, 1),
                                            (1, 3, 16, 32, 64, 0)])
@pytest.mark.parametrize("row", [0, -1])
def test_weight_gradient_of_an_infinite_input(row, B, H, W, Ci, Co, up, monkeypatch):
    """An infinite x reaches the sums that it is a term of and no other: the entries of dw that are
    finite are those of the mma.sync kernel, and agree (P products exact in FP32, each sum within
    P 2^-23 sum|terms| of the exact one), in tiles that are cut off by the image's last row too."""
    g = torch.Generator(device="cuda").manual_seed(H + Ci)
    hi, wi = (H // 2, W // 2) if up else (H, W)
    x = torch.randn((B, hi, wi, Ci), device="cuda", generator=g).to(torch.bfloat16)
    dy = torch.randn((B, H, W, Co), device="cuda", generator=g).to(torch.bfloat16)
    finite = x.clone()
    finite[0, row, 1, 2] = 0
    x[0, row, 1, 2] = float("inf")
    out = {}
    for mma in ("tcgen05", "sync"):
        monkeypatch.setenv("LBNCI_UNET_MMA", mma)
        out[mma] = _wgrad(x, dy, up)[0].view(Co, 9, Ci).double()
    monkeypatch.setenv("LBNCI_UNET_MMA", "sync")
    scale = _wgrad(finite.abs(), dy.abs(), up)[0].view(Co, 9, Ci).double()
    ok = torch.ones((Co, 9, Ci), dtype=torch.bool, device="cuda")
    ok[:, :, 2] = False
    if not up:  # no pixel lies beyond the image: one row of taps never meets its first or last row
        ok[:, slice(0, 3) if row else slice(6, 9), 2] = True
    assert torch.equal(torch.isfinite(out["sync"]), ok)
    assert torch.equal(torch.isfinite(out["tcgen05"]), ok)
    assert bool(((out["tcgen05"] - out["sync"])[ok].abs() <= 2.1 * B * H * W * 2.0 ** -23 * scale[ok]).all())
