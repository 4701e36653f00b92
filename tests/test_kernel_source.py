"""What a kernel's source must hold for its lanes not to race, where running a
kernel could not show it reliably (and a race is not provoked on a GPU)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_06984_gb300", "csrc")


def kernel_body(name, file):
    """Text of a __global__ function, comments removed."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, file)).read())
    at = src.index("{", re.search(r"\b%s\s*\(const" % name, src).end())
    depth = 0
    for k in range(at, len(src)):
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        if depth == 0:
            return src[at:k + 1]
    raise AssertionError("unbalanced braces")


def test_ghost_adjoints_are_read_by_the_whole_group_before_any_is_cleared():
    """k_adj_gff: all 2^d lanes of a group read the Q adjoints of their ghost,
    and each clears its share.  Shuffles do not order memory accesses, so a
    warp barrier that every lane reaches lies between."""
    body = kernel_body("k_adj_gff", "adjoint.cuh")
    reads = [m.end() for m in re.finditer(r"=\s*lam_c\[", body)]
    clears = [m.start() for m in re.finditer(r"lam_c\[[^;]*\]\s*=\s*R\(0\)", body)]
    assert reads and clears
    between = body[max(reads):min(clears)]
    assert "__syncwarp()" in between
    # before the lanes without a ghost leave the iteration
    assert between.index("__syncwarp()") < between.index("if (!active) continue")
