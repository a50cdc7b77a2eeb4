"""GPU parity of the row-norm, ragged-transpose, batched-score and fp32 block kernels at the edges of their tiles."""
import numpy as np
import pytest

from oracle import chains
from paper_2404_13528_b200 import binding as sm
from paper_2404_13528_b200 import synth
from tests.gpu_util import assert_close_bf16, to_dev, to_host_bits, to_host_f64
from tests.test_gpu_chains import CH2A, CH2B, patch_merging_case, run_plan
from tests.test_gpu_swin import case
from tests.test_planner import _ops_from_chain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,C,H,W", [
    (3, 9, 5, 13),            # odd on both sides: 2-byte loads and stores
    (2, 66, 8, 9),            # 16-byte loads, 4-byte stores, two tiles each way
    (1, 136, 7, 10),          # 4-byte loads, 16-byte stores; one image
    (2, 100, 3, 4),           # a tile shorter than a pass
    (4, 64, 8, 8), (1, 8, 1, 8),
])
def test_ragged_channels_last_copies_bit_exact(B, C, H, W):
    x = synth.normal(501, 0, (B, C, H, W), dtype="bf16")
    chain = CH2B(B, C, H, W)
    out = run_plan(_ops_from_chain(chain) + [sm.make_op(sm.OP_COPY)], [sm.make_desc((B, C, H, W))], sm.ELIMINATE, [to_dev(x)], (B, H * W, C))
    assert np.array_equal(to_host_bits(out), chains.apply_layout_chain(x, chain))


@pytest.mark.parametrize("B,S,H,D", [
    (20, 200, 8, 64),         # one 256-wide tile per 128 rows, clipped at row and column 200
    (40, 136, 4, 32), (10, 264, 16, 128),   # the shortest reduction; two k-blocks, eight columns in the second tile
    (8, 192, 10, 64), (8, 288, 9, 32), (3, 480, 9, 128), (4, 576, 8, 64),   # 96-wide tiles where they fill the columns, 256-wide for 480
    (6, 504, 8, 64), (37, 200, 8, 128), (20, 264, 5, 128),   # the tiles' rows stored one by one: a last tile of 248 columns, of 72 rows, of 8 by 8
])
def test_batched_scores_clipped_tiles(B, S, H, D):
    q = synth.normal(502, 0, (B, S, H * D), dtype="bf16")
    k = synth.normal(502, 1, (B, S, H * D), dtype="bf16")
    ops = _ops_from_chain(CH2A(B, S, H, D)) + [sm.make_op(sm.OP_BMM_NT, side_input=(1, 0))]
    out = run_plan(ops, [sm.make_desc((B, S, H * D))] * 2, sm.ELIMINATE, [to_dev(q), to_dev(k)], (B, H, S, S))
    ref = chains.chain_2a_scores(synth.to_f64(q), synth.to_f64(k), H)
    assert_close_bf16(to_host_f64(out), ref, f"{B} x {S}")


@pytest.mark.parametrize("C", [8, 24, 40, 64, 72, 136, 192, 256])
def test_row_norm_widths(C):
    """4 C from 32 to 1024 elements: every split of a row over lanes, with and without idle ones."""
    patch_merging_case(2, 6, 10, C)


@pytest.mark.parametrize("cfg", [
    dict(B=2, H=14, W=21, C=96, heads=3, window=7, shift=3, mlp_ratio=4),     # three CTAs per window, ragged last 16 rows
    dict(B=1, H=8, W=16, C=64, heads=2, window=8, shift=4, mlp_ratio=2),      # T = 64
    dict(B=1, H=7, W=7, C=32, heads=1, window=7, shift=0, mlp_ratio=1),       # no cluster in the attention half
    dict(B=1, H=6, W=4, C=128, heads=8, window=2, shift=1, mlp_ratio=4),      # T = 4, eight heads
    dict(B=1, H=4, W=4, C=192, heads=6, window=4, shift=2, mlp_ratio=4),      # hidden features over eight CTAs
    dict(B=1, H=4, W=4, C=320, heads=10, window=4, shift=0, mlp_ratio=4),     # beyond both kernels: kernel by kernel
])
def test_fp32_blocks(cfg):
    case(503, dtype="f32", **cfg)


@pytest.mark.parametrize("cfg,fused", [
    (dict(B=1, H=28, W=56, C=32, heads=2, window=7, shift=3, mlp_ratio=4), True),      # 98 groups of sixteen rows: one kernel
    (dict(B=2, H=28, W=56, C=32, heads=2, window=7, shift=3, mlp_ratio=4), False),     # 196: three
    (dict(B=1, H=28, W=56, C=16, heads=1, window=7, shift=0, mlp_ratio=1), False),
    (dict(B=2, H=28, W=56, C=64, heads=2, window=7, shift=3, mlp_ratio=4), True),
])
def test_fp32_mlp_half_by_size(cfg, fused):
    p = sm.SwinParams()
    p.dtype = sm.F32
    for k, v in cfg.items():
        setattr(p, k, v)
    rows = cfg["B"] * cfg["H"] * cfg["W"] * cfg["C"] * 4
    assert (sm.smartmem_swin_block_workspace_bytes(p, sm.ELIMINATE) < 2 * rows) == fused      # only the tensor between the halves
    case(507, dtype="f32", images=[cfg["B"] - 1], **cfg)


@pytest.mark.parametrize("cfg", [
    dict(B=1, H=7, W=7, C=192, heads=6, window=7, shift=0, mlp_ratio=4),      # one tile of 49 rows, hidden features over four CTAs
    dict(B=3, H=14, W=14, C=192, heads=6, window=7, shift=3, mlp_ratio=2),    # over two CTAs, ragged last 76 rows
    dict(B=1, H=16, W=8, C=128, heads=4, window=4, shift=2, mlp_ratio=4),     # exactly one tile, the widest slice (256)
    dict(B=2, H=14, W=14, C=128, heads=4, window=7, shift=3, mlp_ratio=1),    # one CTA per tile
    dict(B=1, H=14, W=14, C=192, heads=6, window=7, shift=3, mlp_ratio=3),    # 576 does not split into whole blocks: kernel by kernel
    dict(B=1, H=48, W=48, C=128, heads=4, window=8, shift=4, mlp_ratio=4),    # 2304 rows, the fewest that two CTAs per tile take
    dict(B=1, H=40, W=56, C=128, heads=4, window=8, shift=0, mlp_ratio=4),    # 2240: kernel by kernel
    dict(B=3, H=14, W=14, C=128, heads=4, window=7, shift=3, mlp_ratio=6),    # four CTAs per tile, ragged last 76 rows
    dict(B=1, H=14, W=14, C=64, heads=2, window=7, shift=3, mlp_ratio=12),    # the narrowest, four CTAs per tile
])
def test_mlp_over_a_cluster(cfg):
    case(504, dtype="bf16", **cfg)


@pytest.mark.parametrize("cfg", [
    dict(B=1, H=7, W=7, C=256, heads=8, window=7, shift=3, mlp_ratio=4),      # one tile of 49 rows, slices of 64 columns, GELU
    dict(B=7, H=14, W=14, C=256, heads=8, window=7, shift=3, mlp_ratio=4),    # slices of 128, ragged last 92 rows
    dict(B=17, H=16, W=8, C=256, heads=8, window=8, shift=0, mlp_ratio=3),    # slices of 128 (QKV and fc1)
    dict(B=37, H=16, W=8, C=256, heads=8, window=8, shift=4, mlp_ratio=4),    # a full wave: slices of 192 and 256
    dict(B=38, H=16, W=8, C=256, heads=8, window=8, shift=4, mlp_ratio=4),    # one tile more: kernel by kernel
    dict(B=5, H=14, W=14, C=128, heads=4, window=7, shift=3, mlp_ratio=0),    # the narrowest rows
])
def test_norm_linear_in_one_wave(cfg):
    case(505, dtype="bf16", **cfg)


@pytest.mark.parametrize("B,H,W,C", [
    (1, 2, 2, 64), (1, 2, 2, 96),             # one row
    (3, 26, 22, 64),                          # 429 rows of 256: three tiles of 192, ragged last 45
    (20, 64, 62, 64),                         # 19840 rows: two rounds of 192-row tiles
    (15, 62, 62, 96),                         # 14415 rows of 384: one round of 256-row tiles, ragged last 79
    (5, 124, 124, 96),                        # 19220 rows: two rounds of 192-row tiles, ragged last 20
    (1, 2, 2, 128), (3, 26, 22, 128),         # rows of 512, two slices of the columns
    (9, 62, 64, 128), (10, 62, 64, 128),      # 8928 rows in one round; 9920 are two: kernel by kernel
])
def test_merge_in_one_kernel(B, H, W, C):
    patch_merging_case(B, H, W, C)


@pytest.mark.parametrize("M,K,N", [
    (300, 256, 384),                          # three slices of the columns over two tiles
    (1568, 256, 1280), (1568, 256, 1408),     # ten slices: 70 pairs of 74; eleven are 77: two kernels
    (9472, 384, 384), (9473, 384, 384),       # two slices, 37 tiles: every pair; a row more
    (3200, 384, 960),                         # five slices, 13 tiles
    (6144, 512, 384), (6145, 512, 384),       # rows of 512 in three slices: 24 tiles, and one more than fits a round
    (18944, 512, 128), (18945, 512, 128),     # in one: 74 tiles, and a second round
    (1, 256, 128), (1, 384, 192), (1, 128, 64),   # one row
])
def test_norm_linear_chains(M, K, N):
    """LayerNorm -> linear, rows as they lie, at the edges of the rule that makes one kernel of them."""
    x, g, b = synth.normal(506, 0, (M, K), dtype="bf16"), synth.normal(506, 1, (K,), 0.02, 1.0, "bf16"), synth.normal(506, 2, (K,), 0.02, 0.0, "bf16")
    w = synth.normal(506, 3, (N, K), std=K ** -0.5, dtype="bf16")
    ops = [sm.make_op(sm.OP_LAYERNORM, side_input=(1, 2), eps=1e-5), sm.make_op(sm.OP_LINEAR, side_input=(3, 0))]
    out = run_plan(ops, [sm.make_desc(t.shape) for t in (x, g, b, w)], sm.ELIMINATE, [to_dev(t) for t in (x, g, b, w)], (M, N))
    xf = synth.to_f64(x)
    xn = (xf - xf.mean(-1, keepdims=True)) / np.sqrt(xf.var(-1, keepdims=True) + 1e-5) * synth.to_f64(g) + synth.to_f64(b)
    assert_close_bf16(to_host_f64(out), xn @ synth.to_f64(w).T, f"{M} x {K} -> {N}")
