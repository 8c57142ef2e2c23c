"""The order 5 <-> 3 box transfers in FP64 at element counts where a block takes one, five and seven elements,
single vectors and a batch's cycle, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import multigrid as M
from oracle import problems as P
from oracle.sem import SemLevel, SemTransfer

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2210_03179_gb300 as cm  # noqa: E402
from gpu_util import N, T  # noqa: E402


# one element a block up to 456 elements of 152 SMs, five on 512, 567 and 1,188, seven on 1,001
@pytest.mark.parametrize("mesh", [(1, 1, 2), (5, 3, 7), (9, 8, 6), (8, 8, 8), (9, 9, 7), (13, 11, 7), (12, 11, 9)])
def test_transfers(mesh):
    v = W.sem_box_vertices(*mesh)
    F, C = SemLevel(v, 5), SemLevel(v, 3)
    tr = SemTransfer(F, C)
    s = cm.Solver("sem", verts=v, orders=(5, 3, 1), lmax=[1.0, 1.0])
    rng = np.random.default_rng(4)
    r, z, base = rng.uniform(-1, 1, F.n), rng.uniform(-1, 1, C.n), rng.uniform(-1, 1, F.n)
    base[F.dirichlet] = 0.0
    rc = torch.full((C.n,), 5.0, dtype=torch.float64, device="cuda")
    cm.chebmg_restrict(s.ctx, 0, cm.CHEBMG_F64, T(r), rc)
    ref = tr.restrict(np.where(F.dirichlet, 0.0, r))
    assert np.abs(N(rc) - ref).max() <= 1e-12 * np.abs(ref).max()
    zf = torch.full((F.n,), 5.0, dtype=torch.float64, device="cuda")
    cm.chebmg_prolong(s.ctx, 0, cm.CHEBMG_F64, T(z), zf)
    ref = tr.prolong(np.where(C.dirichlet, 0.0, z))
    assert np.abs(N(zf) - ref).max() <= 1e-12 and np.all(N(zf)[F.dirichlet] == 0.0)
    zf = T(base)
    cm.chebmg_prolong(s.ctx, 0, cm.CHEBMG_F64, T(z), zf, accumulate=True)
    assert np.abs(N(zf) - (base + ref)).max() <= 1e-12
    s.close()


@pytest.mark.parametrize("nb", [3, 24])      # 3 x 24 and 24 x 24 elements
def test_batched_cycle(nb):
    v = W.sem_box_vertices(4, 3, 2)
    H = P.sem_hierarchy(v, (5, 3, 1), kind="opt4th", k=2, sided="one-sided")
    s = cm.Solver("sem", verts=v, orders=(5, 3, 1), kind="opt4th", order=2, sided="one-sided",
                  lmax=[L.lmax for L in H.levels[:-1]])
    R = np.random.default_rng(5).uniform(-1, 1, (nb, H.levels[0].n))
    R[:, H.levels[0].dirichlet] = 0.0
    Z = torch.empty(nb, H.levels[0].n, dtype=torch.float64, device="cuda")
    cm.chebmg_vcycle_batched(s.ctx, T(R), Z)
    for q in (0, nb - 1):
        ref = M.vcycle(H, R[q])
        assert np.abs(N(Z[q]) - ref).max() <= 1e-8 * np.abs(ref).max()     # coarse solves stop at 1e-10
    s.close()
