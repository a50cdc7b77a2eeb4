"""What is not finite stays where it belongs: a token that is infinite makes its own window's outputs (its own sequence's in a decoder
layer) not finite, and no other element changes by a bit.  Two windows, or the rows on both sides of a sequence's end, share a tile of the
tensor core, where a probability of zero times another window's infinite value would be NaN."""
import pytest
import torch

from paper_2404_13528_b200 import binding as sm
from paper_2404_13528_b200 import synth
from tests.gpu_util import to_dev
from tests.test_gpu_llama import run_layer
from tests.test_gpu_swin import run_block

pytestmark = pytest.mark.gpu


def other_windows(B, H, W, window, shift, token):
    """[B, H, W] mask of the tokens that are not in `token`'s window."""
    b, r, c = token
    win = lambda n, size: ((torch.arange(n) - shift) % n // window, ((torch.tensor(size) - shift) % n) // window)   # noqa: E731
    (rows, rw), (cols, cw) = win(H, r), win(W, c)
    own = (rows == rw)[:, None] & (cols == cw)[None, :]
    mask = torch.ones(B, H, W, dtype=torch.bool)
    mask[b] = ~own
    return mask.cuda()


@pytest.mark.parametrize("B,H,W,C,heads,window,shift,mlp_ratio", [
    (2, 14, 14, 64, 2, 7, 3, 4), (3, 14, 7, 96, 3, 7, 0, 0), (1, 16, 16, 96, 3, 8, 4, 4),       # narrow: the fused attention half
    (3, 14, 7, 128, 4, 7, 0, 4), (1, 14, 21, 192, 6, 7, 3, 0), (2, 16, 16, 256, 8, 8, 4, 0),    # wide, few windows: over a cluster
    (3, 14, 7, 384, 12, 7, 3, 0), (5, 7, 7, 512, 16, 7, 0, 0), (7, 7, 7, 512, 16, 7, 3, 0),
    (2, 8, 8, 32, 2, 4, 2, 0), (1, 14, 14, 48, 3, 7, 3, 0),                                     # heads of 16
])
@pytest.mark.parametrize("mode", [sm.ELIMINATE, sm.ELIMINATE_UNFUSED, sm.EXPLICIT])
def test_windows(B, H, W, C, heads, window, shift, mlp_ratio, mode):
    cfg = dict(B=B, H=H, W=W, C=C, heads=heads, window=window, shift=shift, mlp_ratio=mlp_ratio, dtype="bf16", mode=mode)
    inp = synth.swin_inputs(610, B, H, W, C, heads, window, mlp_ratio, "bf16")
    dev = {k: to_dev(v) for k, v in inp.items()}
    clean = run_block(inp, dev, **cfg)
    assert torch.isfinite(clean.float()).all()
    for token in [(0, 0, 0), (0, H - 1, W - 1), (B - 1, H - 1, 0), (B // 2, H // 2, W // 2)]:
        x = dev["x"].clone()
        x[token][3] = float("inf")
        y = run_block(inp, dev, x_dev=x, **cfg)
        mask = other_windows(B, H, W, window, shift, token)
        assert torch.equal(y[mask], clean[mask]), f"token {token} reached another window"
        assert not torch.isfinite(y[~mask].float()).any()


@pytest.mark.parametrize("B,S,hidden", [(2, 40, 256), (3, 100, 256), (2, 129, 512), (4, 333, 1024), (3, 1290, 256), (24, 200, 512)])
@pytest.mark.parametrize("mode", [sm.ELIMINATE, sm.EXPLICIT])
def test_sequences(B, S, hidden, mode):
    dev = {k: to_dev(v) for k, v in synth.attn_layer_inputs(611, S, hidden, B=B).items()}
    cfg = dict(B=B, S=S, hidden=hidden, heads=hidden // 128, add_residual=0, mode=mode)
    clean = run_layer(dev, **cfg)
    assert torch.isfinite(clean.float()).all()
    for b in (0, B - 1):
        x = dev["x"].clone()
        x[b, 0, 5] = float("inf")
        y = run_layer(dict(dev, x=x), **cfg)
        others = [i for i in range(B) if i != b]
        assert torch.equal(y[others], clean[others]), f"sequence {b} reached another one"
        assert not torch.isfinite(y[b, 0].float()).any()
