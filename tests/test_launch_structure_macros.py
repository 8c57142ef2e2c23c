"""Source-level check of the programmatic-dependent-launch rule for kernels whose names reach `launch_dep`
through a macro or a generic lambda (the finite-difference kernels): each of their definitions calls
`pdl_wait()`, and no launch by an indirect name escapes the check."""
import re

import pytest
from test_launch_structure import _kernel_bodies, _sources

# a macro or function parameter that stands for a kernel in a launch_dep call, and how its callers name it
INDIRECT = {"K": re.compile(r"\bFD_LAUNCH(?:_TILED)?\(\s*(k_\w+)"), "kernel": re.compile(r"\bgo\(\s*(k_\w+)")}


def launched_indirectly(src):
    return {name for text in src.values() for r in INDIRECT.values() for name in r.findall(text)}


def kernels_that_never_wait(src):
    out = []
    for name in sorted(launched_indirectly(src)):
        bodies = [b for text in src.values() for b in _kernel_bodies(name, text)]
        if not bodies or any("pdl_wait();" not in b for b in bodies):
            out.append(name)
    return out


def test_kernels_launched_through_macros_wait():
    src = _sources()
    names = launched_indirectly(src)
    assert {"k_fd_apply", "k_fd_first", "k_fd_step", "k_fd_resid", "k_fd_resid_restrict", "k_fd_smooth_restrict",
            "k_fd_prolong_resid", "k_fd_adj_step"} <= names
    assert kernels_that_never_wait(src) == []


def test_every_indirect_name_is_one_of_these():
    for f, text in _sources().items():
        body = text.replace("inline void launch_dep(void (*k)(KArgs...)", "")
        for arg in re.findall(r"launch_dep\(\s*([A-Za-z_]\w*)", body):
            assert arg.startswith("k_") or arg in INDIRECT, (f, arg)


@pytest.mark.parametrize("name", ["k_fd_apply", "k_fd_step", "k_fd_prolong_resid", "k_fd_adj_step"])
def test_a_missing_wait_is_found(name):
    src = dict(_sources())
    for f, text in src.items():
        for body in _kernel_bodies(name, text):
            text = text.replace(body, body.replace("pdl_wait();", ""))
        src[f] = text
    assert kernels_that_never_wait(src) == [name]
