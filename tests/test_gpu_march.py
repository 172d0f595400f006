"""The marching one-pass red-black sweep that handles choose by rule (FP32
cycles): bitwise the half-sweep launches at the sizes where its tiles, rows,
strips and chunks can go wrong -- rows cut into unequal tiles, several rows per
warp, idle lanes, ragged strips and chunks, every kind of wrap -- and whole
solves, alone, on coarser levels and in a batch whose grids share the launch."""
import numpy as np
import pytest

from paper_1410_8568_gb300 import gbmg
from paper_1410_8568_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,bc", [
    ((320, 256, 256), (1, 1, 0)),   # 80 quads: tiles of 27, 27, 26
    ((320, 256, 256), (0, 0, 1)),
    ((192, 192, 192), (0, 1, 1)),   # two tiles of 24 quads
    ((64, 512, 512), (1, 0, 0)),    # two rows per warp
    ((48, 528, 496), (1, 0, 1)),    # two rows of 12 quads per warp, 8 idle lanes; ragged strips and chunks
    ((16, 512, 1024), (0, 1, 0)),   # 8 rows per warp
    ((128, 128, 128), (1, 1, 1)),   # a tile per row
])
@pytest.mark.parametrize("omega", [1.0, 1.2])
def test_chosen_sweep_equals_half_sweeps(shape, bc, omega):
    gen = torch.Generator(device="cuda").manual_seed(sum(shape))
    cells = (shape[2], shape[1], shape[0])
    rho = torch.exp(torch.rand(cells, generator=gen, dtype=torch.float64, device="cuda") * np.log(1000.0))
    b = torch.randn(cells, generator=gen, device="cuda")
    x0 = torch.randn(cells, generator=gen, device="cuda")
    with gbmg.Solver(shape, bc, rho=rho, omega=omega) as S:
        assert gbmg.sweep_shape(S.tile_choice(gbmg.TILE_SWEEP, 0))[2], "the rule picks the marching sweep here"
        for sweeps in (1, 2):
            want, x, work = x0.clone(), x0.clone(), torch.full_like(x0, float("nan"))
            S.smooth(0, b, want, sweeps, prec=gbmg.MIXED)
            S.smooth_onepass(0, b, x, work, sweeps, prec=gbmg.MIXED)
            assert torch.equal(x if sweeps % 2 == 0 else work, want)


def solve(P, sweep, outer=gbmg.OUTER_FP64, **kw):
    with gbmg.Solver(P.shape, P.bc, rho=torch.from_numpy(P.rho).cuda(), sweep=sweep, outer=outer, **kw) as S:
        rhs, p = torch.from_numpy(P.rhs).cuda(), torch.zeros(P.rhs.shape, dtype=torch.float64, device="cuda")
        st = S.solve(rhs, p, tol=1e-10)
        assert st.status == gbmg.OK
        return p, st.iters


@pytest.mark.parametrize("n,kw", [(128, {}), (128, {"outer": gbmg.OUTER_XP}), (128, {"nu1": 4, "use_graph": False}),
                                  (256, {})])  # 256^3: the 128^3 level marches too
def test_solves_are_bitwise_the_half_sweep_solves(n, kw):
    P = I.config2(n)
    want, it = solve(P, gbmg.SWEEP_HALF, **kw)
    got, it2 = solve(P, gbmg.SWEEP_AUTO, **kw)
    assert it == it2 and torch.equal(want, got)


def test_batch_shares_the_launch():
    probs = [I.config2(128), I.config1(48), I.config1(96, ratio=10.0), I.config2(128, ratio=100.0)]
    alone = [solve(P, gbmg.SWEEP_HALF) for P in probs]
    solvers = [gbmg.Solver(P.shape, P.bc, rho=torch.from_numpy(P.rho).cuda()) for P in probs]
    B = gbmg.Batch(solvers)
    rhs = [torch.from_numpy(P.rhs).cuda() for P in probs]
    ps = [torch.zeros_like(r) for r in rhs]
    for (p, it), q, st in zip(alone, ps, B.solve(rhs, ps, tol=1e-10)):
        assert st.status == gbmg.OK and st.iters == it and torch.equal(p, q)
    B.close()
    for S in solvers:
        S.close()


@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e30])
def test_outer_iterate_at_any_scale(scale):
    """The last sweep of a step adds the correction times a power of 2 to the
    caller's iterate, on the bits of the correction: the same bits as by
    multiply-adds."""
    P = I.config2(128)
    rhs = torch.from_numpy(P.rhs).cuda() * scale
    got = []
    for sweep in (gbmg.SWEEP_HALF, gbmg.SWEEP_AUTO):
        p = torch.zeros_like(rhs)
        with gbmg.Solver(P.shape, P.bc, rho=torch.from_numpy(P.rho).cuda(), sweep=sweep) as S:
            assert S.solve(rhs, p, tol=1e-10).status == gbmg.OK
        got.append(p)
    assert torch.equal(*got)
