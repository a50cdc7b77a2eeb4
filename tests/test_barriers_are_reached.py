"""A wait of a kernel may run out for one warp and not for another, which then stands at a barrier for good.  So no barrier without a limit
lies in a block that a warp only enters while its own waits have succeeded (`if (ok ...)`)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_13528_b200", "csrc")
BARRIER = re.compile(r"bar\.sync|bar\.red|__syncthreads\(|cluster_sync\w*\(|cluster_wait\(|cluster_arrive\w*\(")
GUARD = re.compile(r"if\s*(constexpr\s*)?\(\s*ok\b")


def guarded_barriers(text):
    """Barriers inside blocks headed by `if (ok`, as (guard, barrier) lines."""
    text = re.sub(r"//[^\n]*", "", text)
    found, stack, head = [], [], 0
    for m in re.finditer(r"[{};]|" + BARRIER.pattern, text):
        token = m.group()
        if token == "{":
            stack.append(text[head:m.start()])
        elif token == "}":
            if stack:
                stack.pop()
        elif token != ";":
            here = stack + [text[head:m.start()]]
            found += [(h.strip(), token) for h in here if GUARD.search(h)]
            continue
        head = m.end()
    return found


def test_the_scan_sees_them():
    assert guarded_barriers('if (ok) { x; asm volatile("bar.sync 1, 64;"); }')
    assert guarded_barriers("if (ok && y) ptx::cluster_sync();")
    assert guarded_barriers("if (ok) { if (z) { __syncthreads(); } }")
    assert not guarded_barriers("if (ok) { x; } __syncthreads(); // if (ok) bar.sync")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))), ids=os.path.basename)
def test_every_warp_comes_to_its_barriers(path):
    with open(path) as f:
        assert guarded_barriers(f.read()) == []
