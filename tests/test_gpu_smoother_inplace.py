"""SEM smoothing with the iterate and the right-hand side in one buffer: the result of separate buffers, for
the separate kernels at every order's branches and for the fused smoother; and the kernel that reads the
one while it writes the other declares neither as free of aliases."""
import os
import re

import numpy as np
import pytest

import workloads as W
from oracle import problems as P
from oracle.chebyshev import smooth as oracle_smooth

torch = pytest.importorskip("torch")
import paper_2210_03179_gb300 as cm  # noqa: E402

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_03179_gb300", "csrc")


def test_the_start_kernel_allows_one_buffer():
    text = open(os.path.join(CSRC, "chebyshev.cu")).read()
    for kernel in ("k_smooth_begin",):
        args = re.search(r"__global__[^;{]*?\b" + kernel + r"\s*\(([^)]*)\)", text).group(1)
        for name in ("rin", "x"):      # rin is b, which may be x
            decl = next(a for a in args.split(",") if re.search(r"\b" + name + r"$", a.strip()))
            assert "__restrict__" not in decl, decl


needs_gpu = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")


@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("N", [3, 5, 7])
@pytest.mark.parametrize("kind", ["1st", "opt4th"])
@pytest.mark.parametrize("order", [1, 2, 3, 4])
def test_one_buffer(N, kind, order):
    from gpu_util import N as host, T, relerr
    v = W.sem_box_vertices(3, 2, 4)
    H = P.sem_hierarchy(v, (N, 1) if N == 3 else (N, 3, 1))
    L = H.levels[0]
    s = cm.Solver("sem", verts=v, orders=(N, 1) if N == 3 else (N, 3, 1), kind=kind, prec="mixed",
                  lmax=[x.lmax for x in H.levels[:-1]])
    b = np.random.default_rng(order).uniform(-1, 1, L.n) * ~L.dirichlet
    tol = {cm.CHEBMG_F64: 1e-12, cm.CHEBMG_F32: 1e-4}   # as the smoother with two buffers is tested
    for dt, ty in ((cm.CHEBMG_F64, torch.float64), (cm.CHEBMG_F32, torch.float32)):
        for variant in (0, 2 if dt == cm.CHEBMG_F64 else 1) if N == 7 else (None,):
            if variant is not None:
                cm.chebmg_set_fused_smoother(s.ctx, 0, dt, variant)
            for zero in (True, False):
                x = T(b, ty)
                cm.chebmg_smooth(s.ctx, 0, dt, x, x, order, zero)
                ref = oracle_smooth(L, b, order, kind, L.lmax, 0.1, x0=None if zero else b)
                assert relerr(host(x), ref) < tol[dt], (dt, variant, zero)
    s.close()
