"""What bench.py says of the kernels is what their sources do (CPU)."""
import os
import re

import bench
from paper_1410_8568_gb300 import gbmg

CSRC = os.path.join(os.path.dirname(gbmg.__file__), "csrc")


def test_fp64_operations_of_the_residual():
    src = open(os.path.join(CSRC, "mg_outer.cuh")).read()
    march = src[src.index("void march_pairs("):]
    loop = march[march.index("for (int k = k0; k < k1; k++)"):march.index("f(c, s0, s1, xc);")]
    fmas = len(re.findall(r"\bfma\(", loop))
    value = r"x[a-z]+\d?(?:\.[xy])?"
    differences = set(re.findall(r"(%s - %s)" % (value, value), loop))
    # fma, fma: operations of the two cells of a pair
    assert bench.RES_FP64_OPS == (fmas + len(differences)) / 2


def test_kernel_label_names_the_threads_of_a_block():
    src = open(os.path.join(CSRC, "mg_march.cu")).read()
    warps = int(re.search(r"constexpr int W = (\d+);", src).group(1))
    marching = [v for v in range(1, gbmg.SWEEP_VARIANTS) if gbmg.sweep_shape(v)[2]]
    for v in marching:
        assert "%d threads" % (32 * warps) in bench.finest_kernel(v, 0)
        assert "544" not in bench.finest_kernel(v, 0)
    assert "1024 threads" in bench.finest_kernel(1, 0)
    assert "half-sweep" in bench.finest_kernel(0, 1)
