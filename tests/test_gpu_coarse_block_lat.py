"""The batched coarse CG on box lattices (one block per right-hand side, interior rows alone): one row
per thread, several rows per thread, thin boxes and boxes without a free node, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import multigrid as M
from oracle import problems as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2210_03179_gb300 as cm  # noqa: E402
from gpu_util import N, T, relerr  # noqa: E402


@pytest.mark.parametrize("mesh", [(2, 2, 2), (3, 2, 5), (30, 3, 2), (10, 10, 10), (13, 12, 11)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-8), ("mixed", 1e-5)])     # coarse solve 1e-10; FP32 cycle
def test_cycle_of_a_batch(mesh, prec, tol):
    v = W.sem_box_vertices(*mesh)
    H = P.sem_hierarchy(v, (2, 1), kind="4th", k=1, sided="symmetric", lmax=[2.2])
    s = cm.Solver("sem", verts=v, orders=(2, 1), kind="4th", order=1, sided="symmetric", prec=prec, lmax=[2.2])
    L = H.levels[0]
    R = np.random.default_rng(sum(mesh)).uniform(-1, 1, (3, L.n)) * ~L.dirichlet
    R[1] = 0.0                                   # a zero right-hand side among the others
    Z = torch.full((3, L.n), 7.0, dtype=torch.float64, device="cuda")
    cm.chebmg_vcycle_batched(s.ctx, T(R), Z)
    assert relerr(N(Z), np.stack([M.vcycle(H, r) for r in R])) < tol
    s.close()


def test_no_free_coarse_node():
    # one element across: the coarse level has boundary nodes alone, the finer one has free nodes
    v = W.sem_box_vertices(1, 2, 2)
    H = P.sem_hierarchy(v, (2, 1), kind="4th", k=1, sided="symmetric", lmax=[2.2])
    s = cm.Solver("sem", verts=v, orders=(2, 1), kind="4th", order=1, sided="symmetric", lmax=[2.2])
    L = H.levels[0]
    R = np.random.default_rng(1).uniform(-1, 1, (2, L.n)) * ~L.dirichlet
    Z = torch.empty((2, L.n), dtype=torch.float64, device="cuda")
    cm.chebmg_vcycle_batched(s.ctx, T(R), Z)
    z = np.zeros_like(R)
    for q in range(2):                           # smoothing alone: twice order 1
        x = M.smooth(L, R[q], 1, "4th", L.lmax)
        z[q] = M.smooth(L, R[q], 1, "4th", L.lmax, x0=x)
    assert relerr(N(Z), z) < 1e-12
    s.close()
