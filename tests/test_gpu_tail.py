"""The bottom of the V-cycle in one launch (FP32 cycles): whole solves whose
first tail level is the largest (2048 pairs of cells, four per thread), the
smallest, or ragged, with small (one value per lane) and larger coarsest
inverses, every boundary mix, against the oracle's p*; and as many cycles as the
FP64 handle, whose cycles run the same levels as separate launches.  With one
cycle per refinement step FP32 rounding changes the residual after a cycle by
about 1e-6 of its size, so the counts differ by at most one (a residual that
ends next to the tolerance)."""
import numpy as np
import pytest

import oracle
from paper_1410_8568_gb300 import gbmg
from paper_1410_8568_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [
    ((32, 32, 32), (0, 0, 0)),   # 16^3: 2048 items; 2^3 coarsest
    ((32, 32, 32), (1, 1, 1)),
    ((64, 16, 32), (1, 0, 0)),   # 32 x 8 x 16: rows of 16 items
    ((8, 8, 8), (0, 1, 0)),      # one relaxed tail level, 4^3
    ((24, 16, 12), (1, 1, 0)),   # 12 x 8 x 6, 72 coarsest cells (a warp per row)
    ((12, 12, 20), (0, 0, 1)),   # 6 x 6 x 10: rows that are not whole quads, 45 coarsest cells
    ((24, 24, 24), (0, 0, 0)),   # 12^3, 6^3, 27 coarsest cells (two rows per warp)
]


@pytest.mark.parametrize("shape,bc", SHAPES)
@pytest.mark.parametrize("kw", [{}, {"nu1": 1, "nu2": 2, "omega": 1.1}, {"nu1": 3, "nu2": 0},
                                {"prolongation": gbmg.PROLONG_FLUX}])
def test_tail_solves(shape, bc, kw):
    rng = np.random.default_rng(sum(shape) + 7 * sum(bc))
    rho = I.density_field(shape, None, [(tuple(rng.uniform(0.3, 0.7, 3)), 0.2)], 100.0)
    b = rng.standard_normal((shape[2], shape[1], shape[0]))
    b -= b.mean()
    faces = oracle.faces_from_density(shape, bc, rho)
    want = oracle.solve_exact(shape, bc, faces, b).x
    iters = {}
    for prec in (gbmg.MIXED, gbmg.FP64):
        with gbmg.Solver(shape, bc, rho=torch.from_numpy(rho).cuda(), precision=prec, inner_cycles=1, **kw) as S:
            rhs, p = torch.from_numpy(b).cuda(), torch.zeros(b.shape, dtype=torch.float64, device="cuda")
            st = S.solve(rhs, p, tol=1e-10)
            assert st.status == gbmg.OK
            iters[prec] = st.iters
            err = np.linalg.norm(p.cpu().numpy() - want) / np.linalg.norm(want)
            assert err <= 1e-8, (prec, err)
    assert abs(iters[gbmg.MIXED] - iters[gbmg.FP64]) <= 1, iters
