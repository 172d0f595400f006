"""Kernels that run as thread-block clusters touch another block's shared memory
only between two cluster barriers: before the first one a block of the cluster
may not have started, after the last one it may have left.  Read from the
sources: such an access on the GPU would be undefined."""
import glob
import os
import re

import pytest

from paper_1410_8568_gb300 import gbmg

CSRC = os.path.join(os.path.dirname(gbmg.__file__), "csrc")
BARRIER = re.compile(r"\bcluster_(?:sync|wait)\s*\(")
ACCESS = r"\b(?:ld|st)_cluster\s*\("


def code(path):
    src = open(path).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/|__launch_bounds__\([^)]*\)", "", src, flags=re.S)


def bodies(src, head):
    """(name, body) of every function whose signature matches `head`."""
    for m in re.finditer(head + r"[^;{}]*?\b(\w+)\s*\([^;{}]*\)\s*\{", src):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        yield m.group(1), src[m.end():i]


def cluster_kernels():
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = code(path)
        # helpers of the file that reach into other blocks count as accesses
        remote = {n for n, b in bodies(src, r"__device__") if re.search(ACCESS, b)}
        access = re.compile("|".join([ACCESS] + [r"\b%s\s*\(" % n for n in remote]))
        for name, body in bodies(src, r"__global__"):
            if access.search(body):
                out.append((os.path.basename(path), name, body, access))
    return out


KERNELS = cluster_kernels()


def test_the_cluster_kernels_are_found():
    assert {k[1] for k in KERNELS} >= {"k_coarse_gmres", "k_coarse_setup"}


@pytest.mark.parametrize("kernel", KERNELS, ids=[k[1] for k in KERNELS])
def test_remote_accesses_lie_between_cluster_barriers(kernel):
    _, _, body, access = kernel
    used = [m.start() for m in access.finditer(body)]
    held = [m.start() for m in BARRIER.finditer(body)]
    assert held and held[0] < used[0], "a remote access before every block is known to have started"
    assert held[-1] > used[-1], "no barrier between the last remote access and the end"
