"""FP32 cycles whose diagonals are subnormal floats (below 1.2e-38): relaxed as
any positive diagonal is, by every kernel that relaxes.

Single sweeps against the relaxation in FP64 of the kernel's own FP32 faces: a
residual of 6 products and its sum round at 2^-24 of their sizes, or at half the
smallest float, 2^-150; the quotient is within 2 ulp, the update rounds once.
Solves of a problem and of the same one with its coefficients times 2^-127: FP32
holds both (powers of 2), so every level does the same arithmetic and the iterates
agree but for the last bits of the coarsest inverse.  The right-hand side is a
checkerboard plus a small random part, so that no scaled correction overflows."""
import numpy as np
import pytest

from paper_1410_8568_gb300 import gbmg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def colours(shape):
    k, j, i = np.indices((shape[2], shape[1], shape[0]))
    return (i + j + k) & 1


def relaxed(x, b, w, bc, omega):
    """Relaxation of every cell in FP64, and the bound on an FP32 one's error."""
    num, size, d = np.zeros_like(x), np.abs(b), np.zeros_like(x)
    for ax in range(3):
        a = 2 - ax
        lo, hi = w[ax], np.roll(w[ax], -1, a)  # (a wall's low face is 0: the roll brings that 0 to the high wall)
        dl, dh = np.roll(x, 1, a) - x, np.roll(x, -1, a) - x
        num += lo * dl + hi * dh
        size += lo * np.abs(dl) + hi * np.abs(dh)
        d += lo + hi
    q = (num - b) / d
    err = (8 * 2.0 ** -24 * size + 8 * 2.0 ** -150) / d * (1 + 2.0 ** -20) + np.abs(q) * (4 * 2.0 ** -23 + 6 * 2.0 ** -150 / d)
    return x + omega * q, omega * err + 2.0 ** -23 * (np.abs(x) + omega * np.abs(q))


SWEEPS = [((16, 12, 8), (1, 0, 1), (1, 2)), ((128, 16, 8), (1, 1, 0), (1, 7, 10)), ((7, 6, 5), (0, 0, 0), ()),
          ((64, 64, 64), (0, 1, 1), (2,))]


@pytest.mark.parametrize("shape,bc,onepass", SWEEPS)
@pytest.mark.parametrize("scale", [3e-38, 2e-39, 1e-41])
@pytest.mark.parametrize("omega", [1.0, 1.3])
def test_sweep(shape, bc, onepass, scale, omega):
    rng = np.random.default_rng(sum(shape))
    cells = (shape[2], shape[1], shape[0])
    faces = []
    for ax in range(3):
        f = scale * rng.uniform(0.5, 1.5, size=cells)
        if bc[ax] == gbmg.NEUMANN:
            np.moveaxis(f, 2 - ax, 0)[0] = 0.0
        faces.append(torch.from_numpy(f).cuda())
    x0 = rng.standard_normal(cells).astype(np.float32)
    b = (scale * rng.standard_normal(cells)).astype(np.float32)
    with gbmg.Solver(shape, bc, faces=faces, omega=omega, length=tuple(float(n) for n in shape)) as S:
        w = [a.double().cpu().numpy() for a in S.level_faces32(0)]
        x, db = torch.from_numpy(x0).cuda(), torch.from_numpy(b).cuda()
        S.smooth(0, db, x, 1, prec=gbmg.MIXED)
        got = x.double().cpu().numpy()
        old, red = x0.astype(np.float64), colours(shape) == 0
        want, err = relaxed(old, b.astype(np.float64), w, bc, omega)
        assert (np.abs(got - want) <= err)[red].all()
        old[red] = got[red]
        want, err = relaxed(old, b.astype(np.float64), w, bc, omega)
        assert (np.abs(got - want) <= err)[~red].all()
        for v in onepass:
            y, work = torch.from_numpy(x0).cuda(), torch.zeros_like(x)
            S.smooth_onepass(0, db, y, work, 1, prec=gbmg.MIXED, variant=v)
            assert torch.equal(work, x), v


@pytest.mark.parametrize("n,small", [(32, 2.0 ** -14), (128, 2.0 ** -20)])
def test_solve_of_scaled_coefficients(n, small):
    shape = (n, n, n)
    rng = np.random.default_rng(n)
    sign = rng.permutation(np.repeat([1.0, -1.0], n ** 3 // 2)).reshape(shape)
    b = torch.from_numpy((1.0 - 2.0 * colours(shape)) + small * sign).cuda()
    out = []
    for scale in (1.0, 2.0 ** -127):
        faces = [torch.full(shape, scale, dtype=torch.float64, device="cuda")] * 3
        with gbmg.Solver(shape, (gbmg.PERIODIC,) * 3, faces=faces, length=(float(n),) * 3) as S:
            p = torch.zeros_like(b)
            st = S.solve(b, p, tol=1e-10)
            out.append((st.iters, p * scale))
    assert out[0][0] == out[1][0]
    assert float((out[0][1] - out[1][1]).norm() / out[0][1].norm()) <= 1e-9
