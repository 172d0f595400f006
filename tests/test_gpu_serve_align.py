"""A served request's iterate at any double: the outer kernels move the caller's
array as 16-byte pairs, which an array at an odd element of its allocation does
not have.  First off the sources (such an access would fault the GPU), then
served requests at an odd element, in every outer iteration, on rows of an even
and an odd number of cells and on levels with and without the marching sweep."""
import glob
import os
import re

import numpy as np
import pytest

import oracle
from paper_1410_8568_gb300 import gbmg

torch = pytest.importorskip("torch")
CSRC = os.path.join(os.path.dirname(gbmg.__file__), "csrc")


def test_pairs_of_the_callers_iterate_move_behind_the_alignment_test():
    helpers, marches = 0, 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        # vector accesses of O.p / po.p: in the two helpers that take the test's outcome
        vec = [m.start() for m in re.finditer(r"ld2\(O\.p\b|double2 \*>\(O\.p\b", src)]
        for at in vec:
            assert "pairs" in src[at - 60:at], (path, src[at:at + 40])
            helpers += 1
        for m in re.finditer(r"\(double2 \*\)po\.p", src):
            body = src[src.rfind("outer_out(", 0, m.start()):m.start()]
            assert "(size_t)po.p & 15" in body, path
        # the march over p runs where there are items, and an unaligned p has none
        for m in re.finditer(r"march_pairs\(\s*O, O\.p\b", src):
            assert "O.mitems" in src[src.rfind("if (", 0, m.start()):m.start()], path
            marches += 1
    assert helpers == 2 and marches == 1
    api = open(os.path.join(CSRC, "mg_api.cu")).read()
    assert len(re.findall(r"\bmitems\b", api)) == 1
    assert re.search(r"mitems = \(\(uintptr_t\)p & 15\) == 0 \? v\.mall : 0;", api)
    assert len(re.findall(r"\bv\.p = p;", api)) == 1 and "ov_h[g].p" not in api, "p is bound in one place"


def problem(shape, seed):
    rng = np.random.default_rng(seed)
    cells = (shape[2], shape[1], shape[0])
    rho = np.exp(rng.uniform(0.0, np.log(20.0), size=cells))
    b = rng.standard_normal(cells)
    return rho, b - b.mean()


MODES = {"mixed": {}, "fp64": dict(precision=gbmg.FP64), "xp": dict(outer=gbmg.OUTER_XP),
         "pcg": dict(solver=gbmg.SOLVER_PCG)}


@pytest.mark.gpu
@pytest.mark.parametrize("mode", MODES)
def test_served_iterate_at_an_odd_element(mode):
    tol = 1e-9
    asks = []
    srv = gbmg.Server(4 << 30, max_slots=4, **MODES[mode])
    try:
        for shape, bc in [((5, 7, 9), (0, 0, 0)), ((32, 24, 16), (1, 0, 1)), ((128, 128, 96), (1, 1, 0))]:
            rho, b = problem(shape, sum(shape))
            faces = oracle.faces_from_density(shape, bc, rho)
            rhs = torch.from_numpy(b).cuda()
            whole = torch.full((b.size + 2,), 7.0, dtype=torch.float64, device="cuda")
            p = whole[1:-1].view(rhs.shape)
            p.copy_(torch.linspace(-1.0, 1.0, b.size, dtype=torch.float64, device="cuda").view(rhs.shape))  # warm start
            assert p.data_ptr() % 16 == 8
            dev = [torch.from_numpy(f).cuda() for f in faces]
            torch.cuda.synchronize()
            asks.append((shape, bc, faces, b, whole, p, srv.submit(shape, bc, dev, rhs, p, tol=tol)))
        assert srv.drain() == gbmg.OK
        for shape, bc, faces, b, whole, p, ticket in asks:
            rc, st = srv.poll(ticket)
            assert rc == gbmg.OK and st.rel_res <= tol
            x = p.cpu().numpy()
            # the reported residual may be a sum of FP32 ones (1e-5 of it); both sides
            # round their terms w (p_nb - p_c) at 2^-53 each
            r = np.linalg.norm(b - oracle.apply(shape, bc, faces, x)) / np.linalg.norm(b)
            terms = 2 * sum(np.abs(a).max() * n * n for a, n in zip(faces, shape)) * np.abs(x).max() * np.sqrt(x.size)
            assert r <= tol * (1.0 + 1e-5) + 4 * 2.0 ** -53 * terms / np.linalg.norm(b)
            assert abs(x.mean()) <= 2.0 ** -53 * 4 * np.abs(x).max() * np.sqrt(x.size)
            assert float(whole[0]) == 7.0 and float(whole[-1]) == 7.0
    finally:
        srv.close()
