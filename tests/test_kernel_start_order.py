"""Order of a kernel's first steps in the sources (no GPU): wait for the previous grid before any access to global memory, let the
next one start behind that wait, and, where the kernel has tensor memory, only when its CTA holds its columns - a CTA of the next
kernel could otherwise hold them while it waits for this kernel."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_12499_b200", "csrc")
IN_ORDER = {"selftest_wait_kernel"}      # launched without the attribute: it starts behind the kernel before it


def kernels():
    """(file, name, body without comments) of every kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\b", text):
            head = re.sub(r"__launch_bounds__\s*\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)", "", text[m.end():])
            name = re.match(r"\s*(\w+)\s*\(", head).group(1)
            start = at = head.index("{")
            depth = 0
            while True:
                depth += (head[at] == "{") - (head[at] == "}")
                if depth == 0:
                    break
                at += 1
            yield os.path.basename(path), name, head[start:at + 1]


def fault(body):
    """What is wrong with the order of a kernel's first steps (None: nothing)."""
    waits, starts = [[m.start() for m in re.finditer(f + r"\s*\(\s*\)", body)] for f in ("previous_grid_done", "next_grid_may_start")]
    if len(waits) != 1 or len(starts) != 1:
        return "one wait for the previous grid and one start of the next"
    if not waits[0] < starts[0]:
        return "the next grid starts before the previous one is done"
    allocs = [m.start() for m in re.finditer(r"\btmem_alloc\s*\(", body)]
    if allocs and not (allocs[-1] < starts[0] and "__syncthreads()" in body[allocs[-1]:starts[0]]):
        return "the next grid starts before tensor memory is allocated"
    return None


@pytest.mark.parametrize("source,name,body", [pytest.param(*k, id="%s-%s" % k[:2]) for k in kernels() if k[1] not in IN_ORDER])
def test_order_of_first_steps(source, name, body):
    assert fault(body) is None


def test_order_is_told_apart():
    good = "{ if (warp == 1) tmem_alloc(slot, 128); __syncthreads(); previous_grid_done(); next_grid_may_start(); }"
    assert fault(good) is None
    assert fault("{ previous_grid_done(); next_grid_may_start(); tmem_alloc(slot, 128); __syncthreads(); }")
    assert fault("{ tmem_alloc(slot, 128); previous_grid_done(); next_grid_may_start(); __syncthreads(); }")
    assert fault("{ next_grid_may_start(); previous_grid_done(); }")
    assert fault("{ previous_grid_done(); }")
    assert sum("tmem_alloc" in body for _, _, body in kernels()) >= 10
