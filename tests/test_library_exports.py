"""The C-ABI library loads without a GPU and exports every symbol include/smartmem.h declares."""
import ctypes
import os
import re

import pytest

from paper_2404_13528_b200 import binding as sm

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_symbols():
    text = open(os.path.join(ROOT, "include", "smartmem.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(smartmem_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported_and_bound():
    names = declared_symbols()
    assert len(names) >= 18
    L = ctypes.CDLL(sm.LIB_PATH)
    for n in names:
        assert hasattr(L, n), f"{n} declared in smartmem.h but not exported"
        assert n in sm.EXPORTED, f"{n} has no entry in the Python binding"
        assert hasattr(sm, n), f"binding lacks a function named {n}"


@pytest.mark.parametrize("mode,B,S,code", [
    (sm.ELIMINATE, 1, 1 << 30, sm.ERR_WORKSPACE),           # heads do not count: the cache's rows hold all of them
    (sm.ELIMINATE, 2, 1 << 30, sm.ERR_UNSUPPORTED),
    (sm.EXPLICIT, 1, 1 << 30, sm.ERR_UNSUPPORTED), (sm.EXPLICIT, 1, (1 << 30) - 1, sm.ERR_WORKSPACE),
])
def test_decode_cache_rows_limit(mode, B, S, code):
    p = sm.AttnParams()
    p.dtype, p.B, p.S, p.hidden, p.heads, p.head_dim, p.rms_eps, p.rope_theta = sm.BF16, B, S, 256, 2, 128, 1e-5, 1e4
    p.rms_g = p.w_qkv = p.w_o = 16
    with pytest.raises(sm.SmartmemError) as e:              # refused on the host, nothing is launched: no workspace is given
        sm.smartmem_attn_decode(p, 3, 16, 32, 48, 64, 80, 0, mode, 0)
    assert e.value.code == code


def test_host_only_calls_work_without_a_gpu():
    assert sm.smartmem_status_string(sm.OK) == "ok"
    assert sm.smartmem_launch_count() >= 0
    p = sm.SwinParams()
    p.dtype, p.B, p.H, p.W, p.C, p.heads, p.window, p.shift, p.mlp_ratio = sm.BF16, 2, 14, 14, 64, 2, 7, 3, 4
    e = sm.smartmem_swin_block_workspace_bytes(p, sm.ELIMINATE)
    x = sm.smartmem_swin_block_workspace_bytes(p, sm.EXPLICIT)
    u = sm.smartmem_swin_block_workspace_bytes(p, sm.ELIMINATE_UNFUSED)
    mc = 2 * 14 * 14 * 64 * 2
    # only what the chosen path writes is reserved.  ELIMINATE (attention half and MLP half each one kernel): the tensor between
    # the halves; kernel by kernel: qkv (3), attention output, the tensor between the halves; EXPLICIT adds the layout copies
    assert mc <= e < 2 * mc
    assert 5 * mc <= u < 6 * mc
    assert x >= u + 10 * mc
    p.C, p.heads = 512, 16                        # wide block: LayerNorm outputs and the hidden activation are materialised
    mcw = 2 * 14 * 14 * 512 * 2
    assert sm.smartmem_swin_block_workspace_bytes(p, sm.ELIMINATE) >= (1 + 3 + 1 + 1 + 1 + 4) * mcw
