"""The finite-difference step kernels at the edges of their tiles and branches, against the oracle:
grids below, at and above a tile, every order's branch, a zero and a nonzero guess, right-hand side
and iterate in one buffer, coarsening by two and by another factor, dense coarse problems, batches."""
import numpy as np
import pytest

from oracle import multigrid as M
from oracle import problems as P
from oracle.chebyshev import smooth as oracle_smooth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2210_03179_gb300 as cm  # noqa: E402
from gpu_util import N, T, relerr  # noqa: E402

TOL = {cm.CHEBMG_F64: 1e-12, cm.CHEBMG_F32: 1e-4}     # as the other smoother tests


@pytest.mark.parametrize("m,Lx", [(3, 1.0), (31, 1.0), (33, 4.0), (65, 1.0)])
@pytest.mark.parametrize("kind", ["1st", "opt4th"])
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5])
def test_smoother(m, Lx, kind, order):
    H = P.fd_hierarchy(m, Lx=Lx, coarsest=max(1, m // 2), kind=kind)
    L = H.levels[0]
    s = cm.Solver("fd2d", m=m, Lx=Lx, coarsening=2, coarsest=max(1, m // 2), kind=kind, prec="mixed", lmax=[L.lmax])
    b, x0 = np.random.default_rng(order).uniform(-1, 1, (2, L.n))
    for dt, ty in ((cm.CHEBMG_F64, torch.float64), (cm.CHEBMG_F32, torch.float32)):
        for zero in (True, False):
            x = T(x0, ty)
            cm.chebmg_smooth(s.ctx, 0, dt, T(b, ty), x, order, zero)
            assert relerr(N(x), oracle_smooth(L, b, order, kind, L.lmax, 0.1, x0=None if zero else x0)) < TOL[dt]
        x = T(b, ty)
        cm.chebmg_smooth(s.ctx, 0, dt, x, x, order, True)      # in place
        assert relerr(N(x), oracle_smooth(L, b, order, kind, L.lmax, 0.1)) < TOL[dt]
    s.close()


@pytest.mark.parametrize("m,c,coarsest", [(31, 2, 7), (47, 2, 11), (80, 3, 8), (127, 2, 31), (63, 2, 1)])
@pytest.mark.parametrize("k,sided", [(1, "symmetric"), (2, "symmetric"), (2, "one-sided")])
def test_cycle_and_batch(m, c, coarsest, k, sided):
    H = P.fd_hierarchy(m, c=c, coarsest=coarsest, kind="4th", k=k, sided=sided)
    s = cm.Solver("fd2d", m=m, coarsening=c, coarsest=coarsest, kind="4th", order=k, sided=sided,
                  lmax=[L.lmax for L in H.levels[:-1]])
    R = np.random.default_rng(m).uniform(-1, 1, (18, m * m))
    ref = np.stack([M.vcycle(H, r) for r in R])
    z = torch.empty(m * m, dtype=torch.float64, device="cuda")
    cm.chebmg_vcycle(s.ctx, T(R[0]), z)
    assert relerr(N(z), ref[0]) < 1e-12
    Z = torch.empty(18, m * m, dtype=torch.float64, device="cuda")
    cm.chebmg_vcycle_batched(s.ctx, T(R), Z)
    assert relerr(N(Z), ref) < 1e-12
    s.close()
