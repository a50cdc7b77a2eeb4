"""The per-step calls through the CPython extension take what ctypes takes and refuse what ctypes refuses.  No device is needed: every
call is refused on the host, by the binding or (no workspace) by the library."""
import ctypes

import pytest

from paper_2404_13528_b200 import binding as sm


def swin_params():
    p = sm.SwinParams()
    p.dtype, p.B, p.H, p.W, p.C, p.heads, p.window, p.shift, p.mlp_ratio, p.ln_eps = sm.BF16, 1, 14, 14, 96, 3, 7, 3, 0, 1e-5
    for name in ("ln1_g", "ln1_b", "w_qkv", "b_qkv", "rel_bias_table", "w_proj", "b_proj"):
        setattr(p, name, 16)
    return p


def attn_params():
    p = sm.AttnParams()
    p.dtype, p.B, p.S, p.hidden, p.heads, p.head_dim, p.causal, p.rms_eps, p.rope_theta = sm.BF16, 1, 16, 256, 2, 128, 1, 1e-5, 1e4
    p.rms_g = p.w_qkv = p.w_o = 16
    return p


CALLS = [(lambda p, x=16, n=0, st=0: sm.smartmem_swin_block(p, x, 32, 48, n, sm.ELIMINATE, st), swin_params, attn_params),
         (lambda p, x=16, n=0, st=0: sm.smartmem_attn_layer(p, x, 32, 48, n, sm.ELIMINATE, st), attn_params, swin_params),
         (lambda p, x=16, n=0, st=0: sm.smartmem_attn_decode(p, 3, x, 64, 80, 32, 48, n, sm.ELIMINATE, st), attn_params, swin_params)]


@pytest.fixture(params=["extension", "ctypes"])
def path(request, monkeypatch):
    monkeypatch.setattr(sm, "_fast", sm._NoFast if request.param == "ctypes" else None)
    if request.param == "extension":
        assert sm._bind_fast() is not sm._NoFast


@pytest.mark.parametrize("call,own,other", CALLS)
def test_parameter_blocks(path, call, own, other):
    class Derived(type(own())):
        pass

    derived = Derived.from_buffer_copy(own())
    for good in (own(), derived):
        with pytest.raises(sm.SmartmemError) as e:
            call(good)
        assert e.value.code == sm.ERR_WORKSPACE
    # another block, the block's bytes, too few bytes, nothing
    for bad in (other(), bytes(own()), b"\0" * 8, bytearray(4096), None, 16):
        with pytest.raises((TypeError, ctypes.ArgumentError)):
            call(bad)


@pytest.mark.parametrize("call,own,other", CALLS)
def test_addresses(path, call, own, other):
    for kw, code in ((dict(x=None), sm.ERR_INVALID_ARG), (dict(x=ctypes.c_void_p(16)), sm.ERR_WORKSPACE), (dict(st=None), sm.ERR_WORKSPACE),
                     (dict(st=ctypes.c_void_p(0)), sm.ERR_WORKSPACE), (dict(x=24), sm.ERR_ALIGNMENT)):
        with pytest.raises(sm.SmartmemError) as e:
            call(own(), **kw)
        assert e.value.code == code
    for kw in (dict(x=1.5), dict(n="0"), dict(st=[])):
        with pytest.raises((TypeError, ctypes.ArgumentError)):
            call(own(), **kw)


def test_chain_lists(path):
    plan = sm.smartmem_plan([sm.make_op(sm.OP_TRANSPOSE, perm=(1, 0)), sm.make_op(sm.OP_BMM_NT, side_input=(1, 0))],
                            [sm.make_desc((64, 16)), sm.make_desc((64, 16))], sm.EXPLICIT)
    try:
        for ins, outs, code in (([16, 32], [48], sm.ERR_WORKSPACE), ((16, ctypes.c_void_p(32)), (48,), sm.ERR_WORKSPACE),
                                ([16, None], [48], sm.ERR_INVALID_ARG), ([16, 32], [None], sm.ERR_INVALID_ARG), ([16, 24], [48], sm.ERR_ALIGNMENT)):
            with pytest.raises(sm.SmartmemError) as e:
                sm.smartmem_run_chain(plan, ins, outs, 64, 0, 0)
            assert e.value.code == code
        for ins in ([16, 1.5], 16, [16, object()]):
            with pytest.raises((TypeError, ctypes.ArgumentError)):
                sm.smartmem_run_chain(plan, ins, [48], 64, 0, 0)
    finally:
        sm.smartmem_plan_destroy(plan)
