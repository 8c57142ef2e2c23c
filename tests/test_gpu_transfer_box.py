"""The box transfers of every supported order pair on boxes one element thick, ragged last blocks and
batches, both precisions, with boundary entries that must be ignored on input and written zero."""
import numpy as np
import pytest

import workloads as W
from oracle.sem import SemLevel, SemTransfer

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2210_03179_gb300 as cm  # noqa: E402
from gpu_util import N, T  # noqa: E402

TOL = {cm.CHEBMG_F64: 1e-12, cm.CHEBMG_F32: 2e-5}


@pytest.mark.parametrize("orders", [(7, 3), (3, 1), (7, 5), (5, 3)])
@pytest.mark.parametrize("mesh", [(2, 1, 1), (1, 3, 2), (5, 3, 3)])
def test_pair(orders, mesh):
    v = W.sem_box_vertices(*mesh)
    F, C = SemLevel(v, orders[0]), SemLevel(v, orders[1])
    Tr = SemTransfer(F, C)
    # a level below the pair, so that both of its levels carry FP32 data
    full = orders if orders[1] == 1 else orders + (1,)
    s = cm.Solver("sem", verts=v, orders=full, prec="mixed", lmax=[1.0] * (len(full) - 1))
    rng = np.random.default_rng(sum(mesh))
    rf, zc, base = rng.uniform(-1, 1, F.n), rng.uniform(-1, 1, C.n), rng.uniform(-1, 1, F.n)
    base[F.dirichlet] = 0.0
    for dt, ty in ((cm.CHEBMG_F64, torch.float64), (cm.CHEBMG_F32, torch.float32)):
        rc = torch.full((C.n,), 5.0, dtype=ty, device="cuda")
        cm.chebmg_restrict(s.ctx, 0, dt, T(rf, ty), rc)
        ref = Tr.restrict(np.where(F.dirichlet, 0.0, rf))
        assert np.abs(N(rc) - ref).max() <= TOL[dt] * max(np.abs(ref).max(), 1.0)
        zf = torch.full((F.n,), 5.0, dtype=ty, device="cuda")
        cm.chebmg_prolong(s.ctx, 0, dt, T(zc, ty), zf)
        ref = Tr.prolong(np.where(C.dirichlet, 0.0, zc))
        assert np.abs(N(zf) - ref).max() <= TOL[dt] and np.all(N(zf)[F.dirichlet] == 0.0)
        zf = T(base, ty)
        cm.chebmg_prolong(s.ctx, 0, dt, T(zc, ty), zf, accumulate=True)
        assert np.abs(N(zf) - (base + ref)).max() <= TOL[dt]
    s.close()
