"""GMRES on the coarsest grid, run by a cluster of 16 blocks per grid: the
residual of a single coarse solve at the sizes where the split of the cells over
the blocks can go wrong -- fewer cells than blocks, a last block with fewer
cells, the largest grid (32768 cells: every block and thread full) -- and every
boundary mix.  The solve checks its own residual in FP64 before it returns, so
the residual evaluated here may exceed the tolerance by rounding only (1e-3 of
it: the tolerance is six orders above the rounding of the operands)."""
import numpy as np
import pytest

from paper_1410_8568_gb300 import gbmg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,bc,forced", [
    ((8, 8, 8), (0, 0, 0), True),          # 2^3: 8 cells, 16 blocks
    ((24, 24, 24), (1, 0, 1), True),       # 3^3 = 27: 2 cells per block, the last blocks empty
    ((36, 28, 44), (0, 1, 0), False),      # 9 x 7 x 11
    ((50, 50, 50), (1, 1, 0), False),      # 25^3 = 15625: 977 cells per block, the last 970
    ((2, 128, 128), (0, 1, 1), False),     # 32768: 2048 cells per block, 8 per thread
    ((31, 31, 31), (0, 0, 0), False),      # one level of 29791 cells
])
def test_residual_of_one_coarse_solve(shape, bc, forced):
    rng = np.random.default_rng(sum(shape))
    cells = (shape[2], shape[1], shape[0])
    rho = torch.from_numpy(np.exp(rng.uniform(0.0, np.log(100.0), size=cells))).cuda()
    tol = 1e-8
    with gbmg.Solver(shape, bc, rho=rho, precision=gbmg.FP64, coarse_tol=tol, coarse_max_iters=20000,
                     coarse_solver=gbmg.COARSE_GMRES if forced else gbmg.COARSE_AUTO) as S:
        lvl = S.num_levels() - 1
        nx, ny, nz = S.level_shape(lvl)
        r = torch.from_numpy(rng.standard_normal((nz, ny, nx))).cuda()
        e, ae = torch.empty_like(r), torch.empty_like(r)
        S.coarse_solve(r, e, prec=gbmg.FP64)
        S.apply(lvl, e, ae, prec=gbmg.FP64)
        b = r - r.mean()
        assert abs(float(e.mean())) <= 1e-12 * float(e.abs().max())
        assert float((b - ae).norm()) <= tol * (1 + 1e-3) * float(b.norm())
        again = torch.empty_like(e)
        S.coarse_solve(r, again, prec=gbmg.FP64)
        assert torch.equal(e, again)
