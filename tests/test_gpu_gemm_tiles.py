"""GPU parity of the linear layer at sizes where each tile width, and pairs of CTAs with an odd number of row tiles, are chosen."""
import pytest

from paper_2404_13528_b200 import binding as sm
from paper_2404_13528_b200 import synth
from tests.gpu_util import assert_close_bf16, to_dev, to_host_f64
from tests.test_gpu_chains import run_plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (129, 512, 512),         # 64 wide: few tiles
    (300, 576, 192),         # 64 wide, ragged last row tile
    (3000, 768, 192),        # 96 wide
    (700, 520, 320),         # columns no width divides
    (300, 1024, 2048),       # pairs of CTAs, 128 wide, three row tiles: the last pair's second CTA has no rows
    (257, 2048, 4096),       # pairs, one row in the third tile
    (650, 3072, 1024),       # pairs, 256 wide
    (400, 19200, 384),       # pairs, 256 wide, two tiles of the last round in halves
    (513, 15616, 384),       # the same with 32 tiles in halves, one row in the last pair
])
def test_linear_tile_choices(M, N, K):
    x = synth.normal(402, 0, (M, K), dtype="bf16")
    w = synth.normal(402, 1, (N, K), std=K ** -0.5, dtype="bf16")
    out = run_plan([sm.make_op(sm.OP_LINEAR, side_input=(1, 0))], [sm.make_desc((M, K)), sm.make_desc((N, K))], sm.ELIMINATE,
                   [to_dev(x), to_dev(w)], (M, N))
    assert_close_bf16(to_host_f64(out), synth.to_f64(x) @ synth.to_f64(w).T, f"{M} x {N} x {K}")
