"""The SEM smoother's update kernels where their branches change: odd and even orders (x is updated
every other step), order 1 (no stored direction), a zero weight, vectors that are not 16-byte
aligned, and the restriction residual left behind a pre-smoother, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import multigrid as M
from oracle import problems as P
from oracle.chebyshev import smooth as oracle_smooth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2210_03179_gb300 as cm  # noqa: E402
from gpu_util import N, T, relerr  # noqa: E402

# FP64 as every operator test; FP32: at most 6 operator applications of about 1e-6 each
TOL = {cm.CHEBMG_F64: 1e-12, cm.CHEBMG_F32: 1e-4}


@pytest.fixture(scope="module")
def hierarchy():
    v = W.sem_box_vertices(3, 2, 3)
    return v, P.sem_hierarchy(v, (7, 3, 1))


@pytest.mark.parametrize("kind", ["1st", "opt4th"])
@pytest.mark.parametrize("order", [1, 2, 3, 5])
@pytest.mark.parametrize("shift", [0, 1])
def test_orders_and_alignment(hierarchy, kind, order, shift):
    v, H = hierarchy
    L = H.levels[0]
    s = cm.Solver("sem", verts=v, orders=(7, 3, 1), kind=kind, prec="mixed", lmax=[x.lmax for x in H.levels[:-1]])
    rng = np.random.default_rng(order)
    b, x0 = rng.uniform(-1, 1, (2, L.n))
    b[L.dirichlet] = x0[L.dirichlet] = 0.0
    for dt, ty in ((cm.CHEBMG_F64, torch.float64), (cm.CHEBMG_F32, torch.float32)):
        for zero in (True, False):
            bt = torch.empty(L.n + 1, dtype=ty, device="cuda")[shift:shift + L.n]
            xt = torch.empty(L.n + 1, dtype=ty, device="cuda")[shift:shift + L.n]
            bt.copy_(T(b, ty))
            xt.copy_(T(x0, ty))
            cm.chebmg_smooth(s.ctx, 0, dt, bt, xt, order, zero)
            ref = oracle_smooth(L, b, order, kind, L.lmax, 0.1, x0=None if zero else x0)
            assert relerr(N(xt), ref) < TOL[dt], (dt, zero)
    s.close()


@pytest.mark.parametrize("betas", [(0.0,), (1.1, 0.0), (0.0, 1.2, 0.0)])
def test_zero_weights(hierarchy, betas):
    v, H = hierarchy
    L = H.levels[0]
    s = cm.Solver("sem", verts=v, orders=(7, 3, 1), kind="4th", lmax=[x.lmax for x in H.levels[:-1]])
    cm.chebmg_set_smoother_weights(s.ctx, betas)
    b = np.random.default_rng(3).uniform(-1, 1, L.n) * ~L.dirichlet
    x = torch.full((L.n,), 7.0, dtype=torch.float64, device="cuda")
    cm.chebmg_smooth(s.ctx, 0, cm.CHEBMG_F64, T(b), x, len(betas), True)
    ref = oracle_smooth(L, b, len(betas), "4th", L.lmax, 0.1, betas=np.array(betas))
    assert np.abs(N(x) - ref).max() <= 1e-12 * max(np.abs(ref).max(), 1e-300)
    s.close()


@pytest.mark.parametrize("k,sided", [(1, "symmetric"), (3, "symmetric"), (1, "one-sided")])
def test_residual_after_the_smoother(hierarchy, k, sided):
    v, H = hierarchy
    HH = P.sem_hierarchy(v, (7, 3, 1), kind="4th", k=k, sided=sided, lmax=[x.lmax for x in H.levels[:-1]])
    s = cm.Solver("sem", verts=v, orders=(7, 3, 1), kind="4th", order=k, sided=sided,
                  lmax=[x.lmax for x in H.levels[:-1]])
    r = np.random.default_rng(5).uniform(-1, 1, HH.levels[0].n) * ~HH.levels[0].dirichlet
    z = torch.empty(len(r), dtype=torch.float64, device="cuda")
    cm.chebmg_vcycle(s.ctx, T(r), z)
    assert relerr(N(z), M.vcycle(HH, r)) < 1e-8     # the coarse solve stops at 1e-10
    s.close()
