"""The work that users of the library have it do, as cases that can be timed: sizes, inputs, the call, what one call
cannot do without, and how far another correct implementation's results may lie.

Every case goes through the library's public entry points in the mode a program runs in production (ELIMINATE), with
the parameter block, plan, workspace and cache that such a program keeps between calls.  Kinds of work:

  swin           smartmem_swin_block: one shifted-window block, attention half and MLP half (bf16; fp32 for small models)
  prefill        smartmem_attn_layer: one decoder attention layer over whole prompts
  decode         smartmem_attn_decode: the same layer for one new token per sequence against a key/value cache
  scores         smartmem_run_chain: reshape -> transpose -> batched q k^T
  merge          smartmem_run_chain: patch merging (gather of 2x2 neighbours -> LayerNorm -> linear) between two stages
  channels_last  smartmem_run_chain: NCHW -> [B, HW, C] as a copy
"""
import math

import torch

from paper_2404_13528_b200 import binding as sm


# ------------------------------------------------------------------------------------------------ the cases
def swin(name, B, H, W, C, window, shift, mlp_ratio=4, dtype="bf16", head_dim=32):
    return dict(name=name, kind="swin", B=B, H=H, W=W, C=C, head_dim=head_dim, window=window, shift=shift,
                mlp_ratio=mlp_ratio, dtype=dtype)


def prefill(name, B, S, hidden, rotary_dim=0, residual=0):
    return dict(name=name, kind="prefill", B=B, S=S, hidden=hidden, rotary_dim=rotary_dim, residual=residual)


def decode(name, B, pos, hidden, rotary_dim=0, residual=0):
    return dict(name=name, kind="decode", B=B, pos=pos, hidden=hidden, rotary_dim=rotary_dim, residual=residual)


def scores(name, B, S, heads, head_dim):
    return dict(name=name, kind="scores", B=B, S=S, heads=heads, head_dim=head_dim)


def merge(name, B, H, W, C):
    return dict(name=name, kind="merge", B=B, H=H, W=W, C=C)


def channels_last(name, B, C, H, W):
    return dict(name=name, kind="channels_last", B=B, C=C, H=H, W=W)


def listed():
    return [
        # the smallest call: attention half of a tiny fp32 block, 64 tokens; latency and launches are all there is
        swin("swin_fp32_8x8_c32", 1, 8, 8, 32, window=4, shift=2, mlp_ratio=0, dtype="f32", head_dim=16),
        # interactive use: one image through a first-stage block
        swin("swin_1x56x56_c96", 1, 56, 56, 96, window=7, shift=3),
        # batch inference: the first-stage block at the benchmark's batch
        swin("swin_32x56x56_c96", 32, 56, 56, 96, window=7, shift=3),
        # a later, wide stage at a large batch: the contractions dominate
        swin("swin_64x14x14_c512", 64, 14, 14, 512, window=7, shift=3),
        # a second-stage block at a small odd batch: ragged row tiles, no shift
        swin("swin_5x28x28_c192", 5, 28, 28, 192, window=7, shift=0),
        # a whole prompt through a decoder layer of a 4096-wide model
        prefill("prefill_1x2048_h4096", 1, 2048, 4096),
        # two short prompts of odd length, partial rotary embedding, residual added: serving traffic
        prefill("prefill_2x333_h2048_rot32", 2, 333, 2048, rotary_dim=32, residual=1),
        # decoding at a large batch with full caches: the caches are the traffic
        decode("decode_64x2047_h4096", 64, 2047, 4096),
        # decoding for one user: the weights are the traffic
        decode("decode_1x1000_h4096", 1, 1000, 4096),
        # head split and transpose eliminated into a batched q k^T
        scores("scores_8x1024_16x64", 8, 1024, 16, 64),
        # patch merging after the first stage at the benchmark's batch
        merge("merge_32x56x56_c96", 32, 56, 56, 96),
        # a convolution's output handed to token-wise layers: the eliminated chain as one copy
        channels_last("channels_last_8x256x64x64", 8, 256, 64, 64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the kinds and ranges above.  Sizes run over their logarithm; the totals are bounded by the largest
    listed case of the kind."""
    kind = rng.choice(["swin", "swin", "swin", "swin_fp32", "prefill", "prefill", "decode", "decode", "scores", "merge",
                       "channels_last"])
    if kind == "swin":
        C = rng.choice([64, 96, 128, 192, 256, 384, 512])          # 32-wide heads, stages one to three
        window = rng.choice([7, 7, 7, 8])
        most = {64: 8, 96: 8, 128: 8, 192: 4, 256: 4, 384: 2, 512: 2}[C]
        H, W = window * rng.randint(1, most), window * rng.randint(1, most)
        B = max(1, min(_log_int(rng, 1, 64), 32 * 56 * 56 * 96 // (H * W * C), 64 * 14 * 14 * 512 * 512 // (H * W * C * C)))
        case = swin("", B, H, W, C, window, rng.choice([0, window // 2]))
    elif kind == "swin_fp32":
        d = rng.choice([16, 32])
        heads = rng.randint(1, 3)
        window = rng.choice([4, 7])
        case = swin("", rng.randint(1, 3), window * rng.randint(1, 3), window * rng.randint(1, 3), heads * d, window,
                    rng.choice([0, window // 2]), mlp_ratio=rng.choice([0, 4]), dtype="f32", head_dim=d)
    elif kind == "prefill":
        hidden = rng.choice([1024, 2048, 4096])
        B = _log_int(rng, 1, 8)
        case = prefill("", B, _log_int(rng, 16, 2048 // B), hidden, rng.choice([0, 0, 32, 64]), rng.choice([0, 1]))
    elif kind == "decode":
        hidden = rng.choice([1024, 2048, 4096])
        B = _log_int(rng, 1, 64)
        case = decode("", B, min(_log_int(rng, 16, 8000), 64 * 2047 // B), hidden, rng.choice([0, 0, 32, 64]),
                      rng.choice([0, 1]))
    elif kind == "scores":
        case = scores("", rng.randint(1, 8), 8 * _log_int(rng, 4, 128), rng.randint(2, 16), rng.choice([32, 64, 128]))
    elif kind == "merge":
        C = rng.choice([64, 96, 128, 192, 256])
        most = 28 if C < 192 else 14
        H, W = 2 * rng.randint(3, most), 2 * rng.randint(3, most)
        case = merge("", max(1, min(_log_int(rng, 1, 32), 32 * 56 * 56 * 96 // (H * W * C))), H, W, C)
    else:
        C, H, W = _log_int(rng, 16, 512), _log_int(rng, 7, 64), _log_int(rng, 7, 64)
        case = channels_last("", max(1, min(_log_int(rng, 1, 32), 8 * 256 * 64 * 64 // (C * H * W))), C, H, W)
    del case["name"]
    return case


# ------------------------------------------------------------------------------------------------ inputs
class _Plan:
    """A chain's plan, kept by the program for as long as it runs the chain."""

    def __init__(self, ops, shapes):
        self.handle = sm.smartmem_plan(ops, [sm.make_desc(s) for s in shapes], sm.ELIMINATE)
        self.workspace_bytes = sm.smartmem_plan_workspace_bytes(self.handle)

    def __del__(self):
        sm.smartmem_plan_destroy(self.handle)


class _State:
    pass


def prepare(case, seed):
    """Activations N(0, 1), weights and tables N(0, 0.02), scales 1 + N(0, 0.02): the library's synthetic recipe."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dtype = torch.float32 if case.get("dtype") == "f32" else torch.bfloat16

    def normal(*shape, std=1.0, mean=0.0):
        return torch.empty(shape, dtype=dtype, device="cuda").normal_(mean, std, generator=gen)

    def weight(*shape):
        return normal(*shape, std=0.02)

    def scale(*shape):
        return normal(*shape, std=0.02, mean=1.0)

    s = _State()
    s.kind = kind = case["kind"]
    if kind == "swin":
        B, H, W, C, r, ws = (case[k] for k in ("B", "H", "W", "C", "mlp_ratio", "window"))
        heads = C // case["head_dim"]
        s.weights = dict(ln1_g=scale(C), ln1_b=weight(C), w_qkv=weight(3 * C, C), b_qkv=weight(3 * C),
                         rel_bias_table=weight((2 * ws - 1) ** 2, heads), w_proj=weight(C, C), b_proj=weight(C))
        if r:
            s.weights.update(ln2_g=scale(C), ln2_b=weight(C), w_fc1=weight(r * C, C), b_fc1=weight(r * C),
                             w_fc2=weight(C, r * C), b_fc2=weight(C))
        p = sm.SwinParams()
        p.dtype = sm.F32 if dtype == torch.float32 else sm.BF16
        p.B, p.H, p.W, p.C, p.heads, p.window, p.shift, p.mlp_ratio = B, H, W, C, heads, ws, case["shift"], r
        p.ln_eps = 1e-5
        for k, t in s.weights.items():
            setattr(p, k, t.data_ptr())
        s.p, s.x = p, normal(B, H, W, C)
        s.y = torch.empty_like(s.x)
        s.workspace_bytes = sm.smartmem_swin_block_workspace_bytes(p, sm.ELIMINATE)
    elif kind in ("prefill", "decode"):
        B, hidden = case["B"], case["hidden"]
        s.weights = dict(rms_g=scale(hidden), w_qkv=weight(3 * hidden, hidden), w_o=weight(hidden, hidden))
        p = sm.AttnParams()
        p.dtype, p.B, p.hidden, p.heads, p.head_dim, p.causal = sm.BF16, B, hidden, hidden // 128, 128, 1
        p.add_residual, p.rotary_dim, p.rms_eps, p.rope_theta = case["residual"], case["rotary_dim"], 1e-5, 10000.0
        for k, t in s.weights.items():
            setattr(p, k, t.data_ptr())
        s.p = p
        if kind == "prefill":
            p.S = case["S"]
            s.x = normal(B, p.S, hidden)
            s.workspace_bytes = sm.smartmem_attn_layer_workspace_bytes(p, sm.ELIMINATE)
        else:
            s.pos = case["pos"]
            p.S = (s.pos + 256) // 256 * 256                          # caches grow in blocks of 256 positions
            s.x = normal(B, hidden)
            s.k_cache, s.v_cache = normal(B, p.S, hidden), normal(B, p.S, hidden)
            s.k_new, s.v_new = s.k_cache[:, s.pos], s.v_cache[:, s.pos]
            s.workspace_bytes = sm.smartmem_attn_decode_workspace_bytes(p, sm.ELIMINATE)
        s.y = torch.empty_like(s.x)
    else:
        B = case["B"]
        if kind == "scores":
            S, nh, d = case["S"], case["heads"], case["head_dim"]
            s.inputs = [normal(B, S, nh * d), normal(B, S, nh * d)]
            ops = [sm.make_op(sm.OP_RESHAPE, shape=(B, S, nh, d)), sm.make_op(sm.OP_TRANSPOSE, perm=(0, 2, 1, 3)),
                   sm.make_op(sm.OP_BMM_NT, side_input=(1, 0))]
            out = (B, nh, S, S)
        elif kind == "merge":
            H, W, C = case["H"], case["W"], case["C"]
            s.inputs = [normal(B, H, W, C), scale(4 * C), weight(4 * C), weight(2 * C, 4 * C)]
            ops = [sm.make_op(sm.OP_RESHAPE, shape=(B, H // 2, 2, W // 2, 2, C)),
                   sm.make_op(sm.OP_TRANSPOSE, perm=(0, 1, 3, 4, 2, 5)),
                   sm.make_op(sm.OP_RESHAPE, shape=(B, (H // 2) * (W // 2), 4 * C)),
                   sm.make_op(sm.OP_LAYERNORM, side_input=(1, 2), eps=1e-5), sm.make_op(sm.OP_LINEAR, side_input=(3, 0))]
            out = (B, (H // 2) * (W // 2), 2 * C)
        else:
            C, H, W = case["C"], case["H"], case["W"]
            s.inputs = [normal(B, C, H, W)]
            ops = [sm.make_op(sm.OP_TRANSPOSE, perm=(0, 2, 3, 1)), sm.make_op(sm.OP_RESHAPE, shape=(B, H * W, C)),
                   sm.make_op(sm.OP_COPY)]
            out = (B, H * W, C)
        s.plan = _Plan(ops, [tuple(t.shape) for t in s.inputs])
        s.y = torch.empty(out, dtype=dtype, device="cuda")
        s.workspace_bytes = s.plan.workspace_bytes
    s.workspace = torch.empty(max(s.workspace_bytes, 16), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    stream = torch.cuda.current_stream().cuda_stream
    if s.kind == "swin":
        sm.smartmem_swin_block(s.p, s.x.data_ptr(), s.y.data_ptr(), s.workspace.data_ptr(), s.workspace_bytes, sm.ELIMINATE,
                               stream)
        return s.y
    if s.kind == "prefill":
        sm.smartmem_attn_layer(s.p, s.x.data_ptr(), s.y.data_ptr(), s.workspace.data_ptr(), s.workspace_bytes, sm.ELIMINATE,
                               stream)
        return s.y
    if s.kind == "decode":
        sm.smartmem_attn_decode(s.p, s.pos, s.x.data_ptr(), s.k_cache.data_ptr(), s.v_cache.data_ptr(), s.y.data_ptr(),
                                s.workspace.data_ptr(), s.workspace_bytes, sm.ELIMINATE, stream)
        return {"y": s.y, "k_new": s.k_new, "v_new": s.v_new, "k_cache": s.k_cache, "v_cache": s.v_cache}
    sm.smartmem_run_chain(s.plan.handle, [t.data_ptr() for t in s.inputs], [s.y.data_ptr()], s.workspace.data_ptr(),
                          s.workspace_bytes, stream)
    return s.y


# ------------------------------------------------------------------------------------------------ work and tolerance
def work(case):
    """Inputs and weights read once, results written once; multiply-adds counted as two operations."""
    k, B = case["kind"], case["B"]
    if k == "swin":
        C, r, T = case["C"], case["mlp_ratio"], case["window"] ** 2
        M, params = B * case["H"] * case["W"], (4 + 2 * r) * C * C
        size = 4 if case["dtype"] == "f32" else 2
        return {"bytes": size * (2 * M * C + params), "flops": 2 * M * params + 4 * M * T * C}
    if k == "prefill":
        h, S = case["hidden"], case["S"]
        return {"bytes": 2 * (2 * B * S * h + 4 * h * h), "flops": 8 * B * S * h * h + 2 * B * S * (S + 1) * h}
    if k == "decode":
        h, pos = case["hidden"], case["pos"]
        return {"bytes": 2 * (4 * h * h + 2 * B * pos * h + 4 * B * h), "flops": 8 * B * h * h + 4 * B * (pos + 1) * h}
    if k == "scores":
        S, nh, d = case["S"], case["heads"], case["head_dim"]
        return {"bytes": 2 * (2 * B * S * nh * d + B * nh * S * S), "flops": 2 * B * nh * S * S * d}
    n = B * case["C"] * case["H"] * case["W"]
    if k == "merge":
        return {"bytes": 2 * (n + 8 * case["C"] ** 2 + n // 2), "flops": 4 * n * case["C"]}
    return {"bytes": 4 * n, "flops": 0}


def tolerance(case):
    """bf16 results carry a rounding of 2^-9 of their own on top of bf16 intermediates; a few elements of the first
    positions of a causal layer, whose softmax runs over a handful of keys, see an unaveraged rounding of q and k."""
    if case["kind"] == "channels_last":
        return "exact"
    if case.get("dtype") == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-2, "max": 1e-1}
