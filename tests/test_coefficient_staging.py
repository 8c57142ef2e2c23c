"""Source-level check of the rule that the line-coefficient classes state: every thread of a block stages
them in the constructor, and a block barrier separates that from the first line that uses them."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_03179_gb300", "csrc")
CONSTRUCTED = re.compile(r"const Coef8?<[^>]*> (\w+)\((?:&?s\w+)\);")
BARRIER = re.compile(r"__syncthreads\(\)|named_sync\(")


def kernels():
    out = []
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for part in open(p).read().split("__global__")[1:]:
            m = CONSTRUCTED.search(part)
            if m:
                name = re.search(r"\b(k_\w+)\s*\(", part).group(1)
                out.append(pytest.param(part[m.end():], m.group(1), id=f"{os.path.basename(p)}:{name}"))
    return out


def test_the_kernels_are_found():
    assert len(kernels()) >= 7


@pytest.mark.parametrize("body,coef", kernels())
def test_a_barrier_precedes_the_first_line(body, coef):
    use = re.search(r"\bline8?<[^;]*>\(" + coef + r",", body)
    assert use is not None
    before = body[:use.start()]
    # a helper that is defined before the barrier but called after it would have to be looked at by hand
    assert BARRIER.search(before), before[-300:]
