"""Level-0 face coefficients from a density, against extended precision.

A harmonic face is 2 / (h^2 (rho_l + rho_c)).  The sum, the reciprocal and the
product with 1 / h^2 round once each (the reciprocal by 0.5 ulp of FP32 pieces, or
by Newton steps outside [2^-60, 2^61)): three times 2^-53, and a quarter for what
is below a rounding; the host's h, h^2 and 1 / h^2 add four more.  An arithmetic
face is half the sum of two reciprocals: the same count.  Sizes: short axes, ragged,
more cells than one pass of the grid's threads."""
import numpy as np
import pytest

from paper_1410_8568_gb300 import gbmg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def density(shape, kind, rng):
    cells = shape[::-1]
    if kind == "ratio_1000":
        return np.exp(rng.uniform(0.0, np.log(1000.0), size=cells))
    if kind == "whole":  # sums that are short, powers of two among them
        return rng.integers(1, 9, size=cells).astype(np.float64)
    if kind == "wide":  # over the edges of the FP32 expansion's range
        return np.ldexp(rng.uniform(1.0, 2.0, size=cells), rng.integers(-66, 66, size=cells))
    return np.ldexp(rng.uniform(1.0, 2.0, size=cells), rng.integers(-400, 400, size=cells))


@pytest.mark.parametrize("shape", [(2, 3, 5), (33, 17, 9), (160, 128, 64)])
@pytest.mark.parametrize("kind", ["ratio_1000", "whole", "wide", "beyond"])
@pytest.mark.parametrize("mode,length", [(gbmg.HARMONIC, 1.0), (gbmg.HARMONIC, 0.37), (gbmg.ARITHMETIC, 1.0)])
def test_faces(shape, kind, mode, length):
    rng = np.random.default_rng(sum(shape))
    bc = (1, 0, 1)
    rho = density(shape, kind, rng)
    faces = [torch.empty(shape[::-1], dtype=torch.float64, device="cuda") for _ in range(3)]
    gbmg.faces_from_density(shape, bc, torch.from_numpy(rho).cuda(), *faces, mode=mode)
    scaled = None
    if kind in ("ratio_1000", "whole"):
        with gbmg.Solver(shape, bc, rho=torch.from_numpy(rho).cuda(), face_mode=mode,
                         length=(length,) * 3) as S:
            scaled = [w.cpu().numpy() for w in S.level_faces(0)]
            S.set_density(torch.from_numpy(rho).cuda(), mode)
            for w, v in zip(scaled, S.level_faces(0)):
                assert np.array_equal(w, v.cpu().numpy())
    r = rho.astype(np.longdouble)
    for d in range(3):
        ax = 2 - d
        low = np.roll(r, 1, axis=ax)
        want = 2 / (r + low) if mode == gbmg.HARMONIC else (1 / r + 1 / low) / 2
        if not bc[d]:
            want[(slice(None),) * ax + (0,)] = 0
        got = faces[d].cpu().numpy()
        assert np.all(np.abs(got - want) <= np.longdouble(3.25 * 2.0 ** -53) * want)
        if scaled is not None:
            h = np.longdouble(length) / shape[d]
            want = want / (h * h)
            assert np.all(np.abs(scaled[d] - want) <= np.longdouble(7.25 * 2.0 ** -53) * want)
