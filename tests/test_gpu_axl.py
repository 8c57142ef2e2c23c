"""The line-pass operator of the orders without a kernel of their own (2, 4, 5, 6, 8, 9): one
element, full and ragged last blocks, ids from the lattice and from a map, batches, both
precisions, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle.sem import SemLevel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2210_03179_gb300 as cm  # noqa: E402
from gpu_util import N, T, relerr  # noqa: E402

TOL = {cm.CHEBMG_F64: 1e-12, cm.CHEBMG_F32: 2e-5}     # those of the other operator tests


@pytest.mark.parametrize("order", [2, 4, 5, 6, 8, 9])
@pytest.mark.parametrize("mesh", [(2, 1, 1), (5, 2, 1), (3, 3, 2)])
@pytest.mark.parametrize("boxed", [True, False])
def test_operator(order, mesh, boxed):
    v = W.sem_box_vertices(*mesh)
    L = SemLevel(v, order)
    dirichlet = L.dirichlet.copy()
    kw = dict(orders=(order, 1), prec="mixed", lmax=[1.0])
    if boxed:
        s = cm.Solver("sem", verts=v, **kw)
    else:
        s = cm.Solver("sem_mesh", coords=L.coords.reshape(L.E, -1, 3), gid=L.gid.reshape(L.E, -1), n=L.n,
                      dirichlet=dirichlet, **kw)
    X = np.random.default_rng(order).uniform(-1, 1, (3, L.n))
    ref = np.stack([L.apply_A(x) for x in X])
    for dt, ty in ((cm.CHEBMG_F64, torch.float64), (cm.CHEBMG_F32, torch.float32)):
        y = torch.full((L.n,), 3.0, dtype=ty, device="cuda")
        cm.chebmg_apply_A(s.ctx, 0, dt, T(X[0], ty), y)
        assert relerr(N(y), ref[0]) < TOL[dt]
        Y = torch.empty((3, L.n), dtype=ty, device="cuda")
        cm.chebmg_apply_A_batched(s.ctx, 0, dt, T(X, ty), Y)
        assert relerr(N(Y), ref) < TOL[dt]
    s.close()


# FP64 takes the line passes above four elements per SM (one at orders 8 and 9) and a thread per point
# up to there: both sides of the line on 152 SMs.
@pytest.mark.parametrize("order,mesh", [(o, m) for o in (4, 5, 6) for m in ((19, 8, 4), (29, 7, 3))] +
                         [(o, m) for o in (8, 9) for m in ((19, 4, 2), (17, 3, 3))])
@pytest.mark.parametrize("boxed", [True, False])
def test_operator_about_the_line(order, mesh, boxed):
    v = W.sem_box_vertices(*mesh)
    L = SemLevel(v, order)
    kw = dict(orders=(order, 1), prec="fp64", lmax=[1.0])
    if boxed:
        s = cm.Solver("sem", verts=v, **kw)
    else:
        s = cm.Solver("sem_mesh", coords=L.coords.reshape(L.E, -1, 3), gid=L.gid.reshape(L.E, -1), n=L.n,
                      dirichlet=L.dirichlet.copy(), **kw)
    x = np.random.default_rng(order).uniform(-1, 1, L.n)
    y = torch.full((L.n,), 3.0, dtype=torch.float64, device="cuda")
    cm.chebmg_apply_A(s.ctx, 0, cm.CHEBMG_F64, T(x), y)
    assert relerr(N(y), L.apply_A(x)) < TOL[cm.CHEBMG_F64]
    s.close()
