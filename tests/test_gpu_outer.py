"""The FP64 outer kernels at the sizes where their split of the cells can go
wrong: planes smaller and larger than a block's pairs, rows of an odd number of
cells, an odd number of cells, ragged z pieces, every wrap.  The starting
residual's norm of a nonzero iterate against the oracle's (FP64 handles: both
round at 2^-53 of a sum of 13 terms a cell, 1e-12 of the norm is far above it;
mixed handles add up the FP32 residuals, 1e-6), the residual a solve
reports against the oracle's operator, and a right-hand side that is only 8-byte aligned."""
import numpy as np
import pytest

import oracle
from paper_1410_8568_gb300 import gbmg
from paper_1410_8568_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [((2, 2, 2), (0, 1, 0)), ((6, 10, 4), (1, 0, 1)), ((5, 7, 9), (0, 0, 0)), ((7, 8, 8), (1, 1, 0)),
          ((18, 4, 50), (0, 1, 1)), ((130, 6, 10), (1, 0, 0)), ((64, 64, 40), (1, 1, 0)), ((96, 48, 72), (0, 0, 1))]


def problem(shape, seed):
    rng = np.random.default_rng(seed)
    cells = (shape[2], shape[1], shape[0])
    rho = np.exp(rng.uniform(0.0, np.log(50.0), size=cells))
    b, p = rng.standard_normal(cells), rng.standard_normal(cells)
    return rho, b - b.mean(), p


@pytest.mark.parametrize("shape,bc", SHAPES)
@pytest.mark.parametrize("prec,outer,tol", [(gbmg.FP64, gbmg.OUTER_FP64, 1e-12), (gbmg.MIXED, gbmg.OUTER_FP64, 1e-6)])
@pytest.mark.parametrize("solver", [gbmg.SOLVER_MG, gbmg.SOLVER_PCG])
def test_starting_residual(shape, bc, prec, outer, tol, solver):
    rho, b, p0 = problem(shape, sum(shape))
    faces = oracle.faces_from_density(shape, bc, rho)
    want = np.linalg.norm(b - oracle.apply(shape, bc, faces, p0))
    with gbmg.Solver(shape, bc, rho=torch.from_numpy(rho).cuda(), precision=prec, outer=outer, solver=solver,
                     max_iters=1) as S:
        st = S.solve(torch.from_numpy(b).cuda(), torch.from_numpy(p0).cuda(), tol=1e-15)
        assert abs(st.res0 - want) <= tol * want


@pytest.mark.parametrize("shape,bc", SHAPES[1:])
@pytest.mark.parametrize("solver", [gbmg.SOLVER_MG, gbmg.SOLVER_PCG])
def test_solve_and_unaligned_rhs(shape, bc, solver):
    rho, b, _ = problem(shape, 3 * sum(shape))
    faces = oracle.faces_from_density(shape, bc, rho)
    with gbmg.Solver(shape, bc, rho=torch.from_numpy(rho).cuda(), solver=solver, max_iters=400) as S:
        rhs = torch.from_numpy(b).cuda()
        p = torch.zeros_like(rhs)
        st = S.solve(rhs, p, tol=1e-10)
        # the reported residual (a sum of FP32 residuals: 1e-5) against the oracle's
        # operator; both round their terms w (p_nb - p_c) at 2^-53 each.  (Plain
        # cycles do not converge on the longest cells, 130 x 6 x 10 of a cube.)
        x = p.cpu().numpy()
        r = np.linalg.norm(b - oracle.apply(shape, bc, faces, x)) / np.linalg.norm(b)
        terms = 2 * sum(np.abs(a).max() * n * n for a, n in zip(faces, shape)) * np.abs(x).max() * np.sqrt(x.size)
        assert abs(st.rel_res - r) <= 1e-5 * r + 4 * 2.0 ** -53 * terms / np.linalg.norm(b)
        assert st.status == gbmg.OK or (st.status == gbmg.ENOTCONV and shape[0] == 130)
        shifted = torch.empty(rhs.numel() + 1, dtype=torch.float64, device="cuda")[1:].view(rhs.shape)
        shifted.copy_(rhs)
        assert shifted.data_ptr() % 16 == 8
        q = torch.zeros_like(rhs)
        S.solve(shifted, q, tol=1e-10)
        assert torch.equal(p, q)
