"""The grid-wide coarse CG at every block size of its lattice form and in its general form on a lattice,
selected by hand: against the oracle on small boxes (a compact one, and a long one whose bands take
more loads per thread), and by the residual on boxes so large that only the big blocks fit."""
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


def vertices(mesh):
    """The perturbed box; long ones with elements of one size instead of a unit box."""
    if max(mesh) <= 3 * min(mesh):
        return W.sem_box_vertices(*mesh)
    return np.ascontiguousarray(W.sem_box_vertices(*mesh, amplitude=0.0) * np.array(mesh) / min(mesh))


def solver(mesh, prec, rows):
    s = cm.Solver("sem", verts=vertices(mesh), orders=(2, 1), prec=prec, lmax=[2.25])
    cm.chebmg_set_coarse_lattice(s.ctx, rows)
    assert cm.chebmg_coarse_lattice(s.ctx) == rows
    kern, blocks, per = cm.chebmg_coarse_shape(s.ctx)
    n = s.size(1)
    assert kern == cm.CHEBMG_COARSE_GRID and (blocks - 1) * per < n <= blocks * per and (rows == 0 or per == rows)
    return s, n


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("mesh,rows", [((11, 10, 12), r) for r in (0, 64, 128, 256, 512, 1024)]
                         + [((300, 3, 2), r) for r in (0, 512, 1024)] + [((150, 3, 2), 256), ((2, 3, 160), 64)])
def test_against_the_oracle(mesh, rows, prec):
    s, n = solver(mesh, prec, rows)
    L = SemLevel(vertices(mesh), 1)
    L.invD = L.inv_diagonal()
    _, lmax = cm.chebmg_coarse_info(s.ctx)
    for degree in (1, 6):
        cm.chebmg_set_coarse_degree(s.ctx, degree)
        b = np.random.default_rng(degree).uniform(-1, 1, n)
        z = torch.empty(n, dtype=torch.float64, device="cuda")
        it = cm.chebmg_coarse_solve(s.ctx, T(b), z)
        ref, it_ref = K.pcg_cheb4(L.apply_A, L.invD, np.where(L.dirichlet, 0.0, b), lmax, degree, 1e-10)
        assert abs(it - it_ref) <= 1
        assert relerr(N(z), ref) < 1e-8          # both stop at 1e-10
    s.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("mesh,rows", [((31, 32, 30), 256), ((36, 36, 36), 512), ((36, 36, 36), 0), ((45, 45, 45), 1024),
                                       ((45, 45, 45), 0), ((54, 54, 54), 0)])
def test_residual_of_large_boxes(mesh, rows, prec):
    s, n = solver(mesh, prec, rows)
    free = torch.zeros(n, dtype=torch.float64, device="cuda")
    cm.chebmg_inv_diagonal(s.ctx, 1, cm.CHEBMG_F64, free)
    free = (free != 0).double()
    for seed, degree in ((1, 1), (2, 12)):
        cm.chebmg_set_coarse_degree(s.ctx, degree)
        b = T(np.random.default_rng(seed).uniform(-1, 1, n))
        z, Az = torch.full_like(b, 7.0), torch.empty_like(b)
        cm.chebmg_coarse_solve(s.ctx, b, z)
        cm.chebmg_apply_A(s.ctx, 1, cm.CHEBMG_F64, z, Az)
        assert float((z * (1 - free)).abs().max()) == 0.0
        # the CG stops at 1e-10 of its recurrence; that and the true residual differ by rounding alone, some
        # hundred iterations at a condition number of a few thousand: below 1e-10 again
        assert float(((b - Az) * free).norm() / (b * free).norm()) < 2e-10
    s.close()


def test_block_sizes_that_cannot_run():
    s, n = solver((300, 3, 2), "mixed", 512)
    for rows in (64, 256, 96, 2048, -1):       # bands of more loads than a thread keeps; no such sizes
        with pytest.raises(cm.ChebmgError):
            cm.chebmg_set_coarse_lattice(s.ctx, rows)
    assert cm.chebmg_coarse_lattice(s.ctx) == 512
    s.close()
    f = cm.Solver("fd2d", m=31, coarsening=2, coarsest=7)
    with pytest.raises(cm.ChebmgError):
        cm.chebmg_set_coarse_lattice(f.ctx, 0)
    assert cm.chebmg_coarse_lattice(f.ctx) == 0
    f.close()


def test_long_boxes_keep_the_general_form():
    """Where only lattice blocks larger than the general form's fit, setup chooses the general form
    (300 x 10 x 3 elements: 243 us a solve against 372 us in blocks of 512)."""
    for mesh in ((300, 3, 2), (400, 2, 2)):
        s = cm.Solver("sem", verts=vertices(mesh), orders=(2, 1), prec="fp64", lmax=[2.25])
        assert cm.chebmg_coarse_lattice(s.ctx) == 0
        kern, _, rows = cm.chebmg_coarse_shape(s.ctx)
        assert kern == cm.CHEBMG_COARSE_GRID and rows % 256 == 0
        s.close()
    for mesh in ((16, 16, 16), (36, 36, 36)):
        s = cm.Solver("sem", verts=vertices(mesh), orders=(2, 1), prec="fp64", lmax=[2.25])
        assert cm.chebmg_coarse_lattice(s.ctx) in (64, 128, 512)
        s.close()
