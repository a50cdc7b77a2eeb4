"""Runs the cases of perf/cases.py, and a few for kernels that none of them takes, for a profiler: every case is warmed up, then one pass
of it is made inside a cudaProfilerStart / Stop range, so that `ncu --profile-from-start off` captures each of its kernels once.  Prints
how many kernels each pass launched.

    python profiles/capture.py [NAME ...]        default: all, and a step of 16 sequences in place of the one of 64
"""
import os
import sys

import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from paper_2404_13528_b200 import binding as sm  # noqa: E402
from perf import cases  # noqa: E402


def every():
    out = [c for c in cases.listed() if c["name"] != "decode_64x2047_h4096"]
    out.append(cases.decode("decode_16x2047_h4096", 16, 2047, 4096))          # (half a gigabyte of cache)
    out.append(cases.swin("swin_10x28x28_c128", 10, 28, 28, 128, window=7, shift=3))
    out.append(cases.swin("swin_fp32_1x28x28_c96", 1, 28, 28, 96, window=7, shift=3, dtype="f32"))
    unfused = dict(next(c for c in out if c["name"] == "swin_32x56x56_c96"), name="swin_32x56x56_c96_unfused")
    return out + [unfused]


def one_pass(case, state):
    if not case["name"].endswith("_unfused"):
        return cases.run(state)
    n = sm.smartmem_swin_block_workspace_bytes(state.p, sm.ELIMINATE_UNFUSED)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    sm.smartmem_swin_block(state.p, state.x.data_ptr(), state.y.data_ptr(), ws.data_ptr(), n, sm.ELIMINATE_UNFUSED,
                           torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()


def main(names):
    for case in every():
        if names and case["name"] not in names:
            continue
        state = cases.prepare(case, 1)
        for _ in range(3):
            one_pass(case, state)
        torch.cuda.synchronize()
        before = sm.smartmem_launch_count()
        torch.cuda.cudart().cudaProfilerStart()
        one_pass(case, state)
        torch.cuda.synchronize()
        torch.cuda.cudart().cudaProfilerStop()
        print(case["name"], sm.smartmem_launch_count() - before, flush=True)
        del state
        torch.cuda.empty_cache()


if __name__ == "__main__":
    main(sys.argv[1:])
