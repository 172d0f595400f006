"""FP64 restriction with a lane per fine row (tables of at most 300 000 coarse
cells): the same bits as the row tiles in whole solves, below and above that line,
with few items (less than a warp's 8, not a multiple of them) and with wraps; and in
a batch whose grids share the launch."""
import numpy as np
import pytest

from paper_1410_8568_gb300 import gbmg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def fields(shape):
    rng = np.random.default_rng(sum(shape))
    rho = torch.from_numpy(np.exp(rng.uniform(0.0, np.log(10.0), size=shape[::-1]))).cuda()
    b = torch.from_numpy(rng.standard_normal(shape[::-1])).cuda()
    return rho, b - b.mean()


def solver(shape, bc, rho, tiles):
    return gbmg.Solver(shape, bc, rho=rho, precision=gbmg.FP64, tiles=tiles, max_iters=6)


@pytest.mark.parametrize("shape,bc", [
    ((4, 4, 4), (1, 1, 1)),        # one item of a lane group per coarse row
    ((12, 20, 4), (0, 1, 0)),      # 3 items per coarse row
    ((36, 28, 44), (1, 0, 0)),
    ((128, 128, 144), (1, 1, 0)),  # 294 912 coarse cells
    ((128, 128, 160), (0, 0, 1)),  # 327 680: the next level's is the first
])
def test_solve_bits(shape, bc):
    rho, b = fields(shape)
    got = []
    for tiles in (0, gbmg.TILES_AUTO):
        p = torch.zeros_like(b)
        with solver(shape, bc, rho, tiles) as S:
            S.solve(b, p, tol=1e-30, raise_on_error=False)
        got.append(p)
    assert torch.equal(*got)


def test_batch_bits():
    shapes = [(32, 32, 32), (48, 24, 16), (64, 32, 48)]
    data = [fields(s) for s in shapes]
    alone = []
    for s, (rho, b) in zip(shapes, data):
        p = torch.zeros_like(b)
        with solver(s, (0, 0, 0), rho, 0) as S:
            S.solve(b, p, tol=1e-30, raise_on_error=False)
        alone.append(p)
    solvers = [solver(s, (0, 0, 0), rho, gbmg.TILES_AUTO) for s, (rho, _) in zip(shapes, data)]
    ps = [torch.zeros_like(b) for _, b in data]
    B = gbmg.Batch(solvers)
    B.solve([b for _, b in data], ps, tol=1e-30)
    B.close()
    for p, q in zip(ps, alone):
        assert torch.equal(p, q)
    for S in solvers:
        S.close()
