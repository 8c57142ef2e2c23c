"""The FP32 operator of orders 4, 5 and 6 on both sides of the element count up to which it takes a thread per
point (four, four and one elements per SM), single vectors and batches whose elements count together, ids
from the lattice and from a map, against the oracle."""
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

TOL = 2e-5     # that of the other FP32 operator tests


def solver(L, v, order, boxed):
    kw = dict(orders=(order, 1), prec="mixed", lmax=[1.0])
    if boxed:
        return cm.Solver("sem", verts=v, **kw)
    return cm.Solver("sem_mesh", coords=L.coords.reshape(L.E, -1, 3), gid=L.gid.reshape(L.E, -1), n=L.n,
                     dirichlet=L.dirichlet.copy(), **kw)


@pytest.mark.parametrize("order,mesh", [(4, (19, 8, 4)), (4, (29, 7, 3)), (5, (19, 8, 4)), (5, (29, 7, 3)),
                                        (6, (19, 4, 2)), (6, (17, 3, 3))])      # on 152 SMs
@pytest.mark.parametrize("boxed", [True, False])
def test_single(order, mesh, boxed):
    v = W.sem_box_vertices(*mesh)
    L = SemLevel(v, order)
    s = solver(L, v, order, boxed)
    x = np.random.default_rng(order).uniform(-1, 1, L.n)
    y = torch.full((L.n,), 3.0, dtype=torch.float32, device="cuda")
    cm.chebmg_apply_A(s.ctx, 0, cm.CHEBMG_F32, T(x, torch.float32), y)
    assert relerr(N(y), L.apply_A(x)) < TOL
    s.close()


@pytest.mark.parametrize("order", [4, 5, 6])
@pytest.mark.parametrize("mesh,nb", [((2, 1, 1), 3), ((3, 2, 3), 40)])      # 6 and 720 elements together
@pytest.mark.parametrize("boxed", [True, False])
def test_batch(order, mesh, nb, boxed):
    v = W.sem_box_vertices(*mesh)
    L = SemLevel(v, order)
    s = solver(L, v, order, boxed)
    X = np.random.default_rng(order).uniform(-1, 1, (nb, L.n))
    Y = torch.full((nb, L.n), 3.0, dtype=torch.float32, device="cuda")
    cm.chebmg_apply_A_batched(s.ctx, 0, cm.CHEBMG_F32, T(X, torch.float32), Y)
    for q in (0, nb // 2, nb - 1):
        assert relerr(N(Y[q]), L.apply_A(X[q])) < TOL
    s.close()
