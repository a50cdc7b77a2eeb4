"""GPU parity of the GEMM for few rows (reduction split over a cluster) and of the decode attention at the edges of its tiles."""
import pytest

from paper_2404_13528_b200 import binding as sm
from paper_2404_13528_b200 import synth
from tests.gpu_util import assert_close_bf16, to_dev, to_host_f64
from tests.test_gpu_chains import run_plan
from tests.test_gpu_decode import check_case
from tests.test_gpu_swin import case as block

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (2, 128, 64),            # one k-block: no split
    (16, 136, 192),          # three k-blocks over three CTAs, a ragged column tile
    (17, 384, 1024),         # one row beyond a 16-row step
    (64, 1024, 4096),        # the widest X with two CTAs per SM
    (65, 256, 512),          # the narrowest with one
    (128, 40, 2048),         # most rows, fewer columns than a tile
    (1, 136, 512), (16, 136, 576),   # the shortest reductions, a ragged column tile; nine k-blocks over eight CTAs
    (16, 136, 448), (17, 136, 704),  # a k-block fewer: the tiled kernel
    (17, 128, 768), (31, 264, 1088),
    (3, 32776, 256), (31, 65528, 256),   # four k-blocks, a large W: no split
    (129, 512, 2048), (256, 512, 2048), (200, 384, 1536), (160, 768, 3072),  # several row tiles, the last one short
    (300, 72, 2048), (1024, 256, 4096),  # ten and seven row tiles
    (64, 768, 3072), (65, 768, 3072),    # a large W: one row tile, two
])
def test_few_row_linear(M, N, K):
    x = synth.normal(401, 0, (M, K), dtype="bf16")
    w = synth.normal(401, 1, (N, K), std=K ** -0.5, dtype="bf16")
    out = run_plan([sm.make_op(sm.OP_LINEAR, side_input=(1, 0))], [sm.make_desc((M, K)), sm.make_desc((N, K))], sm.ELIMINATE,
                   [to_dev(x), to_dev(w)], (M, N))
    assert_close_bf16(to_host_f64(out), synth.to_f64(x) @ synth.to_f64(w).T, f"{M} x {N} x {K}")


@pytest.mark.parametrize("B,C,heads,window", [(4, 384, 12, 7), (5, 256, 8, 7), (3, 512, 16, 8)])
def test_block_of_few_rows(B, C, heads, window):
    """Bias and residual of a block's second MLP product in several row tiles."""
    block(57, B=B, H=window, W=window, C=C, heads=heads, window=window, shift=2, mlp_ratio=4, dtype="bf16")


@pytest.mark.parametrize("B,pos,hidden,heads", [
    (1, 31, 256, 2), (1, 32, 256, 2), (2, 63, 256, 2), (2, 64, 256, 2),      # edges of a 32-row box and of a 64-position stage
    (1, 300, 256, 2),                                                        # shares of a cluster, one of them ragged
    (128, 70, 512, 4),                                                       # CTAs that walk over several sequence-heads
])
def test_decode_tile_edges(B, pos, hidden, heads):
    check_case(45, B, pos, pos + 3, hidden, heads, 1)
