"""The lattice form of the grid-wide coarse CG (vector staged in shared memory) on boxes whose row
counts leave ragged last blocks, thin and long ones, and one without a free node, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import krylov as K
from oracle.sem import SemLevel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2210_03179_gb300 as cm  # noqa: E402
from gpu_util import N, T, relerr  # noqa: E402


@pytest.mark.parametrize("mesh", [(2, 2, 2), (5, 4, 3), (40, 3, 2), (2, 9, 17), (11, 10, 12), (17, 16, 15)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("degree", [1, 5, 16])
def test_solve(mesh, prec, degree):
    v = W.sem_box_vertices(*mesh)
    L = SemLevel(v, 1)
    L.invD = L.inv_diagonal()
    s = cm.Solver("sem", verts=v, orders=(3, 1), prec=prec, lmax=[2.4])
    cm.chebmg_set_coarse_kernel(s.ctx, cm.CHEBMG_COARSE_GRID)
    cm.chebmg_set_coarse_degree(s.ctx, degree)
    _, lmax = cm.chebmg_coarse_info(s.ctx)
    kern, blocks, rows = cm.chebmg_coarse_shape(s.ctx)
    assert kern == cm.CHEBMG_COARSE_GRID and (blocks - 1) * rows < L.n <= blocks * rows
    for seed in (1, 2, 3):         # several launches: tags move on
        b = np.random.default_rng(seed).uniform(-1, 1, L.n)
        z = torch.empty(L.n, dtype=torch.float64, device="cuda")
        it = cm.chebmg_coarse_solve(s.ctx, T(b), z)
        ref, it_ref = K.pcg_cheb4(L.apply_A, L.invD, np.where(L.dirichlet, 0.0, b), lmax, degree, 1e-10)
        assert abs(it - it_ref) <= 1
        assert relerr(N(z), ref) < 1e-8          # both stop at 1e-10
    s.close()


def test_no_free_node():
    s = cm.Solver("sem", verts=W.sem_box_vertices(1, 3, 2), orders=(3, 1), lmax=[2.4])
    n = s.size(1)
    z = torch.full((n,), 3.0, dtype=torch.float64, device="cuda")
    cm.chebmg_coarse_solve(s.ctx, torch.ones(n, dtype=torch.float64, device="cuda"), z)
    assert float(z.abs().max()) == 0.0
    s.close()
