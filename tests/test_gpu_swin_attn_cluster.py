"""The wide attention half over a cluster, at the edges of its range: every cluster size, windows of fewer and of 64 tokens, an odd number of
windows (half a unit), one window, seams in both directions, and the sizes on both sides of the rule that takes it."""
import pytest

from tests.test_gpu_swin import case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [128, 192, 256, 384, 512])
@pytest.mark.parametrize("B,H,W,window,shift", [(1, 7, 7, 7, 0), (1, 21, 7, 7, 3), (3, 14, 7, 7, 3), (2, 16, 16, 8, 4), (1, 4, 12, 4, 1)])
def test_attention_half(C, B, H, W, window, shift):
    case(800 + C + window, B=B, H=H, W=W, C=C, heads=C // 32, window=window, shift=shift, mlp_ratio=0, dtype="bf16")


@pytest.mark.parametrize("C,B,H,W", [(192, 5, 28, 28), (128, 9, 28, 28), (256, 4, 28, 21), (384, 11, 14, 14), (512, 15, 14, 7), (512, 16, 14, 7)])
def test_one_wave_and_beyond(C, B, H, W):
    case(900 + C, B=B, H=H, W=W, C=C, heads=C // 32, window=7, shift=3, mlp_ratio=4, dtype="bf16", images=[0, B - 1])
