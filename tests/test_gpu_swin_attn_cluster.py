"""The wide attention half over a cluster, at the edges of its range: every cluster size, windows of fewer and of 64 tokens, an odd number of
windows (half a unit; five and seven where a cluster of eight takes three units and more), one window, seams in both directions, outputs that
are not 32-byte aligned, and the sizes on both sides of the rule that takes it."""
import pytest
import torch

from paper_2404_13528_b200 import binding as sm
from paper_2404_13528_b200 import synth
from tests.gpu_util import check_status, launched, stream, to_dev
from tests.test_gpu_swin import PARAM_NAMES, case

pytestmark = pytest.mark.gpu


def device_block(config_id, B, H, W, C, window, shift):
    """An attention half's parameter block and input; the tensors that it points into come along."""
    dev = {k: to_dev(v) for k, v in synth.swin_inputs(config_id, B, H, W, C, C // 32, window, 0, "bf16").items()}
    p = sm.SwinParams()
    p.dtype, p.B, p.H, p.W, p.C, p.heads, p.window, p.shift, p.mlp_ratio, p.ln_eps = sm.BF16, B, H, W, C, C // 32, window, shift, 0, 1e-5
    for name in PARAM_NAMES:
        if name in dev:
            setattr(p, name, dev[name].data_ptr())
    return p, dev["x"], dev


@pytest.mark.parametrize("C", [128, 192, 256, 384, 512])
@pytest.mark.parametrize("B,H,W,window,shift", [(1, 7, 7, 7, 0), (1, 21, 7, 7, 3), (3, 14, 7, 7, 3), (2, 16, 16, 8, 4), (1, 4, 12, 4, 1), (5, 7, 7, 7, 0), (7, 7, 7, 7, 3)])
def test_attention_half(C, B, H, W, window, shift):
    case(800 + C + window, B=B, H=H, W=W, C=C, heads=C // 32, window=window, shift=shift, mlp_ratio=0, dtype="bf16")


@pytest.mark.parametrize("C,B,H,W", [(192, 5, 28, 28), (128, 9, 28, 28), (256, 4, 28, 21), (384, 11, 14, 14), (512, 15, 14, 7), (512, 16, 14, 7)])
def test_one_wave_and_beyond(C, B, H, W):
    case(900 + C, B=B, H=H, W=W, C=C, heads=C // 32, window=7, shift=3, mlp_ratio=4, dtype="bf16", images=[0, B - 1])


@pytest.mark.parametrize("C,B,H,W,one_kernel", [
    (128, 1, 7, 7, True), (192, 5, 28, 28, True), (256, 4, 28, 21, True), (384, 1, 7, 7, True), (512, 5, 7, 7, True), (512, 7, 7, 7, True),
    (512, 4, 7, 7, False), (128, 64, 28, 28, False), (192, 1, 77, 77, False), (256, 8, 28, 28, False), (384, 16, 28, 28, False), (512, 16, 14, 14, False)])
def test_which_kernel(C, B, H, W, one_kernel):
    p, x, keep = device_block(970 + C, B, H, W, C, 7, 3)
    for mode in (sm.ELIMINATE, sm.ELIMINATE_UNFUSED, sm.EXPLICIT):
        n = sm.smartmem_swin_block_workspace_bytes(p, mode)
        ws, y = torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty_like(x)
        labels = launched(lambda: sm.smartmem_swin_block(p, x.data_ptr(), y.data_ptr(), ws.data_ptr(), n, mode, stream()))
        assert (labels == ["swin_attn_cluster"]) == (one_kernel and mode == sm.ELIMINATE), (mode, labels)
    check_status()


@pytest.mark.parametrize("C,B,H,W", [(128, 3, 14, 7), (192, 3, 14, 7), (256, 3, 14, 7), (384, 3, 14, 7), (512, 7, 7, 7)])
def test_output_aligned_to_16_bytes(C, B, H, W):
    """The rows leave as two 16-byte stores instead of one of 32: the same bits, and nothing beside them."""
    p, x, keep = device_block(980 + C, B, H, W, C, 7, 3)
    n = sm.smartmem_swin_block_workspace_bytes(p, sm.ELIMINATE)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    outs = []
    for first in (16, 8):                                    # (allocations are 32-byte aligned and more)
        buf = torch.full((x.numel() + 32,), float("nan"), dtype=x.dtype, device="cuda")
        y = buf[first:first + x.numel()]
        assert y.data_ptr() % 32 == (0 if first == 16 else 16)
        labels = launched(lambda: sm.smartmem_swin_block(p, x.data_ptr(), y.data_ptr(), ws.data_ptr(), n, sm.ELIMINATE, stream()))
        assert labels == ["swin_attn_cluster"]
        assert torch.isnan(buf[:first]).all() and torch.isnan(buf[first + x.numel():]).all()
        outs.append(y)
    check_status()
    assert torch.isfinite(outs[0].float()).all() and torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("C,B,H,W", [(128, 9, 28, 28), (192, 5, 28, 28), (256, 4, 28, 21), (384, 11, 14, 14), (512, 15, 14, 7)])
def test_every_call_gives_the_same_bits(C, B, H, W):
    """Full waves, call after call while copies on another stream hold up loads: the heads of a CTA and the two threads of a row share memory,
    and no result may depend on which of them is late."""
    p, x, keep = device_block(950 + C, B, H, W, C, 7, 3)
    n = sm.smartmem_swin_block_workspace_bytes(p, sm.ELIMINATE)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    outs = [torch.full_like(x, float("nan")) for _ in range(100)]
    a, b = torch.empty(2, 64 << 20, dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        for _ in range(40):
            b.copy_(a)
    for y in outs:
        sm.smartmem_swin_block(p, x.data_ptr(), y.data_ptr(), ws.data_ptr(), n, sm.ELIMINATE, stream())
    torch.cuda.synchronize()
    check_status()
    assert torch.isfinite(outs[0].float()).all()
    for y in outs[1:]:
        assert torch.equal(y, outs[0])
