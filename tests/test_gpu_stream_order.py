"""What a call reads may be written by the call right before it on the stream: keys, weights, scales.  Each consumer is run behind the
copy that makes its operand, without and with a synchronisation in between, and the results are compared bit for bit."""
import pytest
import torch

from paper_2404_13528_b200 import binding as sm
from tests.gpu_util import check_status, launched, stream

pytestmark = pytest.mark.gpu

ROUNDS = 12


class Chain:
    """A plan with its workspace, run without a synchronisation."""

    def __init__(self, ops, shapes, mode=sm.ELIMINATE, dtype=sm.BF16):
        self.plan = sm.smartmem_plan(ops, [sm.make_desc(s, dtype) for s in shapes], mode)
        self.steps = sm.smartmem_plan_num_steps(self.plan)
        self.bytes = sm.smartmem_plan_workspace_bytes(self.plan)
        self.ws = torch.empty(max(self.bytes, 16), dtype=torch.uint8, device="cuda")

    def __call__(self, inputs, out):
        sm.smartmem_run_chain(self.plan, [t.data_ptr() for t in inputs], [out.data_ptr()], self.ws.data_ptr(), self.bytes, stream())

    def __del__(self):
        sm.smartmem_plan_destroy(self.plan)


def bf16(seed, *shape, std=1.0, mean=0.0, dtype=torch.bfloat16):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(mean, std, generator=gen)


def transposer(rows, cols, dtype=sm.BF16):
    """[cols, rows] -> [rows, cols] as a copy."""
    return Chain([sm.make_op(sm.OP_TRANSPOSE, perm=(1, 0)), sm.make_op(sm.OP_COPY)], [(cols, rows)], dtype=dtype)


def roller(n, dtype=sm.BF16):
    """[n] -> [n], rotated, as a copy."""
    return Chain([sm.make_op(sm.OP_ROLL, shift=5, axis=0), sm.make_op(sm.OP_COPY)], [(n,)], dtype=dtype)


def compare(sources, make, use, out_like):
    """make(source) writes the operand, use(out) reads it; every round has another source and another output."""
    def run(sync):
        outs = [torch.full_like(out_like, float("nan")) for _ in range(ROUNDS)]
        torch.cuda.synchronize()
        for i, out in enumerate(outs):
            make(sources[i % len(sources)])
            if sync:
                torch.cuda.synchronize()
            use(out)
            if sync:
                torch.cuda.synchronize()
        check_status()
        return outs

    for i, (a, b) in enumerate(zip(run(False), run(True))):
        assert not torch.isnan(b.float()).any()
        assert torch.equal(a, b), f"round {i}: another result behind a synchronisation"


@pytest.mark.parametrize("M,N,K", [(16, 16, 128), (31, 24, 128), (16, 16, 4096)])
def test_explicit_copies_then_scores(M, N, K):
    """Both operands of a product for few rows come from copies of the same call."""
    ops = [sm.make_op(sm.OP_ROLL, shift=3, axis=0), sm.make_op(sm.OP_BMM_NT, side_input=(1, 0))]
    chain = Chain(ops, [(M, K), (N, K)], sm.EXPLICIT)
    assert chain.steps == (3, 2)
    sources = [(bf16(10 + i, M, K), bf16(20 + i, N, K)) for i in range(3)]
    current = []
    compare(sources, lambda s: current.__setitem__(slice(None), s), lambda out: chain(current, out), torch.empty(M, N, dtype=torch.bfloat16, device="cuda"))


@pytest.mark.parametrize("M,N,K", [(16, 16, 128), (31, 2048, 1024)])
def test_keys_of_one_call_scores_of_the_next(M, N, K):
    keys, q = torch.empty(N, K, dtype=torch.bfloat16, device="cuda"), bf16(30, M, K)
    make, scores = transposer(N, K), Chain([sm.make_op(sm.OP_BMM_NT, side_input=(1, 0))], [(M, K), (N, K)])
    compare([bf16(31 + i, K, N) for i in range(3)], lambda s: make([s], keys), lambda out: scores([q, keys], out),
            torch.empty(M, N, dtype=torch.bfloat16, device="cuda"))


@pytest.mark.parametrize("M,N,K", [(3, 512, 1024), (100, 2048, 2048), (300, 512, 512)])
def test_weights_then_linear(M, N, K):
    w, x = torch.empty(N, K, dtype=torch.bfloat16, device="cuda"), bf16(40, M, K)
    make, linear = transposer(N, K), Chain([sm.make_op(sm.OP_LINEAR, side_input=(1, 0))], [(M, K), (N, K)])
    compare([bf16(41 + i, K, N, std=0.05) for i in range(3)], lambda s: make([s], w), lambda out: linear([x, w], out),
            torch.empty(M, N, dtype=torch.bfloat16, device="cuda"))


@pytest.mark.parametrize("which", ["w", "gamma"])
@pytest.mark.parametrize("C", [64, 96, 128])
def test_weights_then_patch_merging(C, which):
    B, H, W = 2, 14, 14
    x, K, N = bf16(50, B, H, W, C), 4 * C, 2 * C
    g, b, w = bf16(51, K, std=0.1, mean=1.0), bf16(52, K, std=0.1), bf16(53, N, K, std=0.05)
    chain = Chain([sm.make_op(sm.OP_RESHAPE, shape=(B, H // 2, 2, W // 2, 2, C)), sm.make_op(sm.OP_TRANSPOSE, perm=(0, 1, 3, 4, 2, 5)),
                   sm.make_op(sm.OP_RESHAPE, shape=(B, H * W // 4, K)), sm.make_op(sm.OP_LAYERNORM, side_input=(1, 2), eps=1e-5),
                   sm.make_op(sm.OP_LINEAR, side_input=(3, 0))], [(B, H, W, C), (K,), (K,), (N, K)])
    if which == "w":
        make, target, sources = transposer(N, K), w, [bf16(54 + i, K, N, std=0.05) for i in range(3)]
    else:
        make, target = roller(K), g
        sources = [bf16(57 + i, K, std=0.1, mean=1.0) for i in range(3)]
    compare(sources, lambda s: make([s], target), lambda out: chain([x, g, b, w], out),
            torch.empty(B, H * W // 4, N, dtype=torch.bfloat16, device="cuda"))


@pytest.mark.parametrize("B", [1, 70, 130])
def test_weights_then_decode_step(B):
    hidden, pos, s_max = 512, 40, 64
    x, k, v = bf16(60, B, hidden), bf16(61, B, s_max, hidden), bf16(62, B, s_max, hidden)
    rms_g, w_qkv, w_o = bf16(63, hidden, std=0.1, mean=1.0), torch.empty(3 * hidden, hidden, dtype=torch.bfloat16, device="cuda"), bf16(64, hidden, hidden, std=0.05)
    make, p = transposer(3 * hidden, hidden), sm.AttnParams()
    p.dtype, p.B, p.S, p.hidden, p.heads, p.head_dim, p.causal, p.rms_eps, p.rope_theta = sm.BF16, B, s_max, hidden, hidden // 128, 128, 1, 1e-5, 10000.0
    p.rms_g, p.w_qkv, p.w_o = rms_g.data_ptr(), w_qkv.data_ptr(), w_o.data_ptr()
    n = sm.smartmem_attn_decode_workspace_bytes(p, sm.ELIMINATE)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    compare([bf16(65 + i, hidden, 3 * hidden, std=0.05) for i in range(3)], lambda s: make([s], w_qkv),
            lambda out: sm.smartmem_attn_decode(p, pos, x.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr(), ws.data_ptr(), n, sm.ELIMINATE, stream()),
            torch.empty_like(x))


@pytest.mark.parametrize("which", ["rms_g", "w_qkv", "x"])
@pytest.mark.parametrize("B,S,hidden", [(1, 20, 512), (2, 32, 3072)])
def test_operands_then_decoder_layer_of_few_rows(B, S, hidden, which):
    """RMSNorm is part of the QKV product, which is the call's first kernel."""
    par = dict(x=bf16(90, B * S, hidden), rms_g=bf16(91, hidden, std=0.1, mean=1.0), w_qkv=bf16(92, 3 * hidden, hidden, std=0.05),
               w_o=bf16(93, hidden, hidden, std=0.05))
    p = sm.AttnParams()
    p.dtype, p.B, p.S, p.hidden, p.heads, p.head_dim, p.causal, p.rms_eps, p.rope_theta = sm.BF16, B, S, hidden, hidden // 128, 128, 1, 1e-5, 10000.0
    p.rms_g, p.w_qkv, p.w_o = par["rms_g"].data_ptr(), par["w_qkv"].data_ptr(), par["w_o"].data_ptr()
    n = sm.smartmem_attn_layer_workspace_bytes(p, sm.ELIMINATE)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    target, std = par[which], 0.05 if which == "w_qkv" else 1.0

    def use(out):
        sm.smartmem_attn_layer(p, par["x"].data_ptr(), out.data_ptr(), ws.data_ptr(), n, sm.ELIMINATE, stream())

    assert launched(lambda: use(torch.empty_like(par["x"])))[0] == "gemm_splitk"
    make = roller(target.numel()) if target.dim() == 1 else transposer(*target.shape)
    compare([bf16(94 + i, *reversed(target.shape), std=std) for i in range(3)], lambda s: make([s], target), use, torch.empty_like(par["x"]))


@pytest.mark.parametrize("which,dtype,C,head_dim,H,half,first", [
    ("w_qkv", sm.BF16, 192, 32, 14, -1, "swin_attn_cluster"), ("w_proj", sm.BF16, 192, 32, 14, -1, "swin_attn_cluster"),
    ("b_qkv", sm.BF16, 192, 32, 14, -1, "swin_attn_cluster"), ("rel_bias_table", sm.BF16, 192, 32, 14, -1, "swin_attn_cluster"),
    ("w_qkv", sm.BF16, 192, 32, 77, -1, "gemm_ln_wave"),       # norm + QKV in one kernel: more windows than one wave of clusters
    ("w_qkv", sm.BF16, 512, 32, 14, -1, "layernorm"),          # kernel by kernel
    ("w_qkv", sm.F32, 32, 16, 8, -1, "swin_attn_f32"),
    ("w_fc1", sm.BF16, 192, 32, 14, 1, "gemm_ln_wave"), ("w_fc1", sm.BF16, 256, 32, 14, 1, "gemm_ln_wave"),   # the MLP half on its own
    ("w_fc1", sm.F32, 32, 16, 8, 1, "swin_mlp_f32"),
    ("w_fc1", sm.BF16, 128, 32, 49, 1, "mlp_cluster"),         # the same over a cluster
])
def test_weights_then_block(which, dtype, C, head_dim, H, half, first):
    td = torch.float32 if dtype == sm.F32 else torch.bfloat16
    ws_, heads = (4 if H == 8 else 7), C // head_dim
    par = dict(ln1_g=bf16(70, C, std=0.1, mean=1.0, dtype=td), ln1_b=bf16(71, C, std=0.1, dtype=td), w_qkv=bf16(72, 3 * C, C, std=0.05, dtype=td),
               b_qkv=bf16(73, 3 * C, std=0.05, dtype=td), rel_bias_table=bf16(74, (2 * ws_ - 1) ** 2, heads, std=0.1, dtype=td),
               w_proj=bf16(75, C, C, std=0.05, dtype=td), b_proj=bf16(76, C, std=0.05, dtype=td), ln2_g=bf16(77, C, std=0.1, mean=1.0, dtype=td),
               ln2_b=bf16(78, C, std=0.1, dtype=td), w_fc1=bf16(79, 4 * C, C, std=0.05, dtype=td), b_fc1=bf16(80, 4 * C, std=0.05, dtype=td),
               w_fc2=bf16(81, C, 4 * C, std=0.05, dtype=td), b_fc2=bf16(82, C, std=0.05, dtype=td))
    p = sm.SwinParams()
    p.dtype, p.B, p.H, p.W, p.C, p.heads, p.window, p.shift, p.mlp_ratio, p.ln_eps = dtype, 1, H, H, C, heads, ws_, 1, 4, 1e-5
    for name, t in par.items():
        setattr(p, name, t.data_ptr())
    x = bf16(83, 1, H, H, C, dtype=td)
    n = sm.smartmem_swin_block_workspace_bytes(p, sm.ELIMINATE)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    target = par[which]
    flat = target.dim() == 1 or which == "rel_bias_table"
    make = roller(target.numel(), dtype) if flat else transposer(*target.shape, dtype)

    def use(out):
        if half < 0:
            sm.smartmem_swin_block(p, x.data_ptr(), out.data_ptr(), ws.data_ptr(), n, sm.ELIMINATE, stream())
        else:
            sm.smartmem_swin_block_half(p, x.data_ptr(), out.data_ptr(), ws.data_ptr(), n, sm.ELIMINATE, half, stream())

    assert launched(lambda: use(torch.empty_like(x)))[0] == first
    shape, std = ((target.numel(),), 0.1) if flat else (tuple(reversed(target.shape)), 0.05)
    compare([bf16(84 + i, *shape, std=std, dtype=td) for i in range(3)], lambda s: make([s], target), use, torch.empty_like(x))
