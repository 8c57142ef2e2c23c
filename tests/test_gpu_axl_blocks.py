"""The order-5 FP64 operator at element counts and batches where a block takes four, five and seven elements,
ragged last blocks among them, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle.sem import SemLevel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2210_03179_gb300 as cm  # noqa: E402
from gpu_util import N, T  # noqa: E402


# 612, 704, 1001, 1188 and 1430 elements: with blocks of four the busiest of 152 SMs has 10, 10, 10, 10 and 15 warps,
# of five 6, 6, 12, 12 and 12, of seven 8, 8, 8, 16 and 16, of one 10, 10, 14, 16 and 20
@pytest.mark.parametrize("mesh", [(17, 9, 4), (11, 8, 8), (13, 11, 7), (12, 11, 9), (13, 11, 10)])
def test_single(mesh):
    v = W.sem_box_vertices(*mesh)
    L = SemLevel(v, 5)
    s = cm.Solver("sem", verts=v, orders=(5, 1), lmax=[1.0])
    x = np.random.default_rng(7).uniform(-1, 1, L.n)
    y = torch.full((L.n,), 3.0, dtype=torch.float64, device="cuda")
    cm.chebmg_apply_A(s.ctx, 0, cm.CHEBMG_F64, T(x), y)
    ref = L.apply_A(x)
    assert np.abs(N(y) - ref).max() <= 1e-12 * np.abs(ref).max()
    s.close()


@pytest.mark.parametrize("mesh,nb", [((3, 4, 6), 9), ((4, 4, 5), 14), ((3, 2, 2), 60)])
def test_batch(mesh, nb):
    v = W.sem_box_vertices(*mesh)
    L = SemLevel(v, 5)
    s = cm.Solver("sem", verts=v, orders=(5, 1), lmax=[1.0])
    X = np.random.default_rng(8).uniform(-1, 1, (nb, L.n))
    Y = torch.full((nb, L.n), 3.0, dtype=torch.float64, device="cuda")
    cm.chebmg_apply_A_batched(s.ctx, 0, cm.CHEBMG_F64, T(X), Y)
    for q in (0, nb // 2, nb - 1):
        ref = L.apply_A(X[q])
        assert np.abs(N(Y[q]) - ref).max() <= 1e-12 * np.abs(ref).max()
    s.close()
