"""The coarsest grid's dense inverse: one block up to 31 cells, a cluster of 16
blocks above, one warp per row in the solve.  Checked below and above the edges of
the set-ups (31 cells, 285 cells, 512 cells: the largest) by the residual of one
solve, against the bound for a matrix inverted by elimination without pivoting
(symmetric positive definite): 8 n u cond(S) |b|, u = 2^-53, S = -A + c 1 1^T
with the set-up's c (mean diagonal / n)."""
import numpy as np
import pytest

from paper_1410_8568_gb300 import gbmg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,bc", [
    ((2, 3, 3), (0, 0, 0)),      # 18
    ((5, 3, 2), (1, 1, 1)),      # 30; a two-cell periodic axis
    ((3, 3, 5), (1, 0, 1)),      # 45
    ((31, 2, 2), (0, 0, 1)),     # 124
    ((11, 13, 2), (0, 1, 0)),    # 286
    ((5, 7, 11), (0, 0, 0)),     # 385
    ((2, 2, 128), (1, 0, 1)),    # 512
])
def test_coarse_solve_residual(shape, bc):
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    cells = shape[::-1]
    rho = torch.from_numpy(np.exp(rng.uniform(0.0, np.log(100.0), size=cells))).cuda()
    with gbmg.Solver(shape, bc, rho=rho, precision=gbmg.FP64, coarse_solver=gbmg.COARSE_AUTO) as S:
        assert S.num_levels() == 1 and S.level_shape(0) == tuple(shape)
        A = torch.empty((n, n), dtype=torch.float64, device="cuda")
        unit = torch.zeros(cells, dtype=torch.float64, device="cuda")
        for c in range(n):
            unit.view(-1)[c] = 1.0
            S.apply(0, unit, A[c].view(cells), prec=gbmg.FP64)
            unit.view(-1)[c] = 0.0
        M = -A.cpu().numpy().T
        kappa = np.linalg.cond(M + np.trace(M) / n / n)
        r = torch.from_numpy(rng.standard_normal(cells)).cuda()
        b = r - r.mean()
        e = torch.empty_like(r)
        S.coarse_solve(b, e, prec=gbmg.FP64)
        res = b.cpu().numpy().ravel() + M @ e.cpu().numpy().ravel()
        assert np.linalg.norm(res) <= 8 * n * 2.0 ** -53 * kappa * float(b.norm())
        again = torch.empty_like(e)
        S.set_density(rho)
        S.coarse_solve(b, again, prec=gbmg.FP64)
        assert torch.equal(e, again)


@pytest.mark.parametrize("shape", [
    (56, 40, 40),   # 175 coarsest cells: the bottom of the cycle in one block
    (40, 40, 72),   # 225: a launch per level and the solve by its own launch
    (56, 56, 36),   # 14 x 14 x 9: GMRES
    (40, 56, 88),   # 385
])
def test_solve_alone_and_in_a_batch(shape):
    """Converged (the solver's own FP64 residual) and the same bits next to a grid
    that keeps the one-block bottom."""
    rng = np.random.default_rng(shape[0] + shape[2])
    probs = []
    for sh in (shape, (32, 32, 32)):
        rho = torch.from_numpy(np.exp(rng.uniform(0.0, np.log(10.0), size=sh[::-1]))).cuda()
        b = torch.from_numpy(rng.standard_normal(sh[::-1])).cuda()
        probs.append((sh, rho, b - b.mean()))
    alone = []
    for sh, rho, b in probs:
        with gbmg.Solver(sh, (0, 0, 0), rho=rho, max_iters=100) as S:
            p = torch.zeros_like(b)
            st = S.solve(b, p, tol=1e-10)
            assert st.rel_res <= 1e-10
            alone.append(p)
    solvers = [gbmg.Solver(sh, (0, 0, 0), rho=rho, max_iters=100) for sh, rho, _ in probs]
    ps = [torch.zeros_like(b) for _, _, b in probs]
    B = gbmg.Batch(solvers)
    B.solve([b for _, _, b in probs], ps, tol=1e-10)
    for p, q in zip(ps, alone):
        assert torch.equal(p, q)
