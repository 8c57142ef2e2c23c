"""Single operator and restriction calls on both sides of the sizes at which they become dependent launch
chains: the route by its launches (a chain zeroes by a kernel, an ordinary call by a memset), and the
results against the oracle."""
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

F32, F64 = cm.CHEBMG_F32, cm.CHEBMG_F64
TYPE = {F32: torch.float32, F64: torch.float64}
TOL = {F32: 2e-5, F64: 1e-12}


def launches(f):
    n0 = cm.chebmg_launch_count()
    f()
    return cm.chebmg_launch_count() - n0


@pytest.mark.parametrize("dt", [F32, F64])
@pytest.mark.parametrize("mesh", [(2, 2, 2), (3, 3, 3), (4, 3, 4)])     # 343, 1,000 and 1,690 nodes at order 3
def test_operator(mesh, dt):
    v = W.sem_box_vertices(*mesh)
    L = SemLevel(v, 3)
    s = cm.Solver("sem", verts=v, orders=(3, 1), prec="mixed", lmax=[1.0])
    x = np.random.default_rng(1).uniform(-1, 1, L.n)
    y = torch.full((L.n,), 3.0, dtype=TYPE[dt], device="cuda")
    xt = T(x, TYPE[dt])
    got = launches(lambda: cm.chebmg_apply_A(s.ctx, 0, dt, xt, y))
    assert got == (2 if dt == F64 or L.n >= 1200 else 1)
    ref = L.apply_A(x)
    assert np.abs(N(y) - ref).max() <= TOL[dt] * np.abs(ref).max()
    s.close()


@pytest.mark.parametrize("dt", [F32, F64])
@pytest.mark.parametrize("mesh", [(2, 2, 2), (4, 4, 4), (5, 4, 4)])     # 3,375, 24,389 and 30,276 nodes at order 7
def test_transfers(mesh, dt):
    v = W.sem_box_vertices(*mesh)
    F, C = SemLevel(v, 7), SemLevel(v, 3)
    tr = SemTransfer(F, C)
    s = cm.Solver("sem", verts=v, orders=(7, 3, 1), prec="mixed", lmax=[1.0, 1.0])
    rng = np.random.default_rng(2)
    r, z = rng.uniform(-1, 1, F.n), rng.uniform(-1, 1, C.n)
    rc = torch.full((C.n,), 3.0, dtype=TYPE[dt], device="cuda")
    zf = torch.full((F.n,), 3.0, dtype=TYPE[dt], device="cuda")
    rt, zt = T(r, TYPE[dt]), T(z, TYPE[dt])
    got = launches(lambda: cm.chebmg_restrict(s.ctx, 0, dt, rt, rc))
    assert got == (2 if F.n >= (5000 if dt == F64 else 25000) else 1)
    ref = tr.restrict(np.where(F.dirichlet, 0.0, r))
    assert np.abs(N(rc) - ref).max() <= TOL[dt] * np.abs(ref).max()
    assert launches(lambda: cm.chebmg_prolong(s.ctx, 0, dt, zt, zf)) == 1
    ref = tr.prolong(np.where(C.dirichlet, 0.0, z))
    assert np.abs(N(zf) - ref).max() <= TOL[dt] * np.abs(ref).max()
    s.close()


def test_level_out_of_range():
    s = cm.Solver("sem", verts=W.sem_box_vertices(2, 2, 2), orders=(3, 1), lmax=[1.0])
    x, c = torch.zeros(343, dtype=torch.float64, device="cuda"), torch.zeros(27, dtype=torch.float64, device="cuda")
    L = cm.lib()
    for level in (-1, 1, 2):
        assert L.chebmg_restrict(s.ctx, level, F64, x.data_ptr(), c.data_ptr()) == cm.CHEBMG_EINVAL
        assert L.chebmg_prolong(s.ctx, level, F64, c.data_ptr(), x.data_ptr(), 0) == cm.CHEBMG_EINVAL
    for level in (-1, 2):
        assert L.chebmg_apply_A(s.ctx, level, F64, x.data_ptr(), x.data_ptr()) == cm.CHEBMG_EINVAL
    s.close()
