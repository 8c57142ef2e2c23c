"""The adjoint step kernels on FD levels where their branches change: orders 1 to 10 (more than one group
of dots), the one-sided cycle, grids that are not multiples of a tile, one and several errors, against
the oracle's forward-mode gradient."""
import numpy as np
import pytest

import workloads as W
from oracle import problems as P
from oracle import sensitivity as SE

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2210_03179_gb300 as cm  # noqa: E402
from gpu_util import T  # noqa: E402


@pytest.mark.parametrize("m,k,sided,nrhs,steps", [
    (15, 1, "symmetric", 1, 1), (31, 1, "one-sided", 3, 2), (47, 3, "symmetric", 2, 2), (65, 2, "symmetric", 1, 1),
    (31, 5, "one-sided", 2, 1),
])
def test_gradient(m, k, sided, nrhs, steps):
    coarsest = {65: 32}.get(m, 7)
    H = P.fd_hierarchy(m, kind="4th", k=k, sided=sided, coarsest=coarsest)
    s = cm.Solver("fd2d", m=m, kind="4th", order=k, sided=sided, coarsest=coarsest,
                  lmax=[L.lmax for L in H.levels[:-1]])
    order = 2 * k if sided == "one-sided" else k
    betas = 1.0 + 0.1 * np.random.default_rng(k).uniform(-1, 1, order)
    E0 = W.random_vectors(m * m, nrhs, seed=m)
    f, gb, gs, _ = cm.chebmg_cycle_error_grad(s.ctx, T(E0), betas, 1.03, steps)
    f_ref, g_ref = SE.error_ratio_and_gradient(H, E0, betas, 1.03, steps)
    assert f == pytest.approx(f_ref, rel=1e-10)
    g, g_ref = np.array(gb + [gs]), np.asarray(g_ref)
    assert np.abs(g - g_ref).max() < 1e-8 * np.abs(g_ref).max()      # as the existing gradient test
    s.close()
