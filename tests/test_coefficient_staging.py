"""Source-level check of the rule that the line-coefficient classes state: every thread of a block stages
them (in the constructor, or by stage()), and a block barrier separates that from the first line that
uses them."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_03179_gb300", "csrc")
STAGED = re.compile(r"const Coef<[^>]*> (\w+)\(&s\w+\);|\b(\w+)\.stage\(s\w+\);")
BARRIER = re.compile(r"__syncthreads\(\)|named_sync\(")


def kernels():
    out = []
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for part in open(p).read().split("__global__")[1:]:
            m = STAGED.search(part)
            if m or re.search(r"\bCoef8?<[^>]*> \w+[;(]", part):
                name = re.search(r"\b(k_\w+)\s*\(", part).group(1)
                assert m, f"{name} never stages its coefficients"
                out.append(pytest.param(part[m.end():], m.group(1) or m.group(2), id=f"{os.path.basename(p)}:{name}"))
    return out


def test_the_kernels_are_found():
    assert len(kernels()) >= 7


@pytest.mark.parametrize("body,coef", kernels())
def test_a_barrier_precedes_the_first_line(body, coef):
    # the FP32 form, which stages nothing, may use them at once
    code = re.sub(r"if constexpr \(Coef8<T>::SHARED == 1\)[^;]*;", "", body)
    use = re.search(r"\bline8?<[^;]*>\(" + coef + r",", code)
    assert use is not None
    before = code[:use.start()]
    # a helper that is defined before the barrier but called after it would have to be looked at by hand
    assert BARRIER.search(before), before[-300:]
