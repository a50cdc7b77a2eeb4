"""The fp32 halves at the edges of their tiles: every number of tokens a window can have, both head dimensions, both sides of the choice
of threads and tiles, shifted and not, and hidden sizes on both sides of the MLP half's tiles."""
import pytest

from tests.test_gpu_swin import case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window,d,heads,shift", [
    (1, 16, 1, 0), (2, 32, 2, 1), (3, 16, 3, 1), (4, 32, 3, 2), (5, 32, 1, 2),      # 256 threads
    (6, 16, 8, 3), (6, 32, 2, 0), (7, 16, 1, 3), (7, 32, 6, 3), (8, 32, 1, 4), (8, 16, 3, 0),   # 512
])
def test_attention_half(window, d, heads, shift):
    case(700 + 10 * window + heads, B=2, H=2 * window, W=3 * window, C=heads * d, heads=heads, window=window, shift=shift, mlp_ratio=0, dtype="f32")


@pytest.mark.parametrize("window,d,heads,B", [(7, 32, 2, 1), (6, 16, 2, 3), (8, 32, 2, 2), (7, 32, 4, 1), (7, 32, 3, 16)])
def test_attention_half_parts(window, d, heads, B):
    """The tokens of a window over four CTAs a head (a short last part at 7 x 7), over two, and not shared out (48 windows)."""
    case(740 + window + heads, B=B, H=window, W=3 * window, C=heads * d, heads=heads, window=window, shift=2, mlp_ratio=0, dtype="f32")


@pytest.mark.parametrize("C,heads,mlp_ratio,B", [(16, 1, 1, 1), (48, 3, 3, 1), (32, 1, 4, 3), (96, 3, 2, 1), (192, 6, 4, 1)])
def test_mlp_half(C, heads, mlp_ratio, B):
    case(760 + C + mlp_ratio, B=B, H=7, W=14, C=C, heads=heads, window=7, shift=3, mlp_ratio=mlp_ratio, dtype="f32")
