"""Which kernel a single U-Net convolution or weight gradient takes, and that each of them is right:
tcgen05.mma with operands copied by TMA is the default, mma.sync (csrc/unet_kernels.cuh) the kernel
of operands that it cannot take and of LBNCI_UNET_MMA=sync."""
import pytest

from paper_2003_11069_gb300 import unet

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
