"""Graphs of several coarse steps: the same results as the steps one by one,
no graph of a size beyond its use, and a graph that cannot be made leaves the
shorter ones in use."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1601_06984_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def deep2d(levels, n=32):
    """Nested 2D boxes of n x n cells, `levels` deep."""
    boxes, lo, hi = [], (0, 0), (n, n)
    for _ in range(levels - 1):
        w = [b - a for a, b in zip(lo, hi)]
        lo, hi = tuple(2 * (a + k // 4) for a, k in zip(lo, w)), tuple(2 * (b - k // 4) for b, k in zip(hi, w))
        boxes.append((lo, hi))
    return W.nested_boxes(2, (n - 1).bit_length(), (n, n), boxes, (W.BC_PERIODIC,) * 4)


# levels, time mode, stencil: below and at the most instants a long graph takes (16), and beyond
@pytest.mark.parametrize("levels,mode,precision", [(2, 0, 0), (2, 1, 1), (2, 2, 2), (3, 2, 0), (5, 0, 1), (6, 0, 1)])
def test_long_graphs_equal_level_by_level(levels, mode, precision):
    from paper_1601_06984_gb300 import lbm
    m = deep2d(levels)
    om = 1.6 if mode == 2 else W.omega_coarse_from_finest(1.6, levels)
    sims = []
    for timing in (0, 1):
        s = lbm.Sim(m, 9, om, precision=precision, time_mode=mode)
        s.init(*W.uniform_fields(m, 1.0, (0.02, 0.01)), W.pdf_perturbation(m, 9, 1e-3))
        s.timing_enable(timing)
        for n in (64, 16, 17, 33):  # long graphs from both parities, with short ones after them
            s.step(n)
        sims.append(s)
    a, b = sims
    assert np.array_equal(a.get_state(), b.get_state())
    assert np.array_equal(a.ghosts()[1], b.ghosts()[1])


# cudaGraphInstantiate in front of the runtime's: refuses graphs of more than
# MAX_NODES nodes and writes down the most that were asked for
SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>
typedef int (*inst_t)(void**, void*, unsigned long long);
typedef int (*nodes_t)(void*, void*, size_t*);
int cudaGraphInstantiate(void** exec, void* graph, unsigned long long flags) {
  static size_t most = 0;
  size_t n = 0;
  ((nodes_t)dlsym(RTLD_NEXT, "cudaGraphGetNodes"))(graph, 0, &n);
  if (n > most) most = n;
  FILE* f = fopen(getenv("NODES_FILE"), "w");
  fprintf(f, "%zu", most);
  fclose(f);
  if (n > (size_t)atol(getenv("MAX_NODES"))) return 2; /* cudaErrorMemoryAllocation */
  return ((inst_t)dlsym(RTLD_NEXT, "cudaGraphInstantiate"))(exec, graph, flags);
}
"""
CHILD = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
from test_gpu_long_graphs import deep2d
from paper_1601_06984_gb300 import lbm, workloads as W
m = deep2d({levels})
s = lbm.Sim(m, 9, {omega}, time_mode={mode})
s.init(*W.uniform_fields(m, 1.0, (0.02, 0.01)))
s.step(64)
n = s.launches()
s.step(32)
print("launches", s.launches() - n)
"""


def run_child(tmp_path, levels, mode, max_nodes):
    """Launches of 32 coarse steps after 64 of them, and the largest graph asked for."""
    src, so, nodes = tmp_path / "shim.c", tmp_path / "shim.so", tmp_path / "nodes"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", str(src), "-o", str(so), "-ldl"], check=True)
    om = 1.6 if mode == 2 else W.omega_coarse_from_finest(1.6, levels)
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"), levels=levels, mode=mode, omega=repr(om))
    env = dict(os.environ, LD_PRELOAD=str(so), NODES_FILE=str(nodes), MAX_NODES=str(max_nodes))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return int(r.stdout.split("launches")[1]), int(nodes.read_text())


def test_long_graphs_stay_small(tmp_path):
    """Six levels of diffusive scaling advance at 1,024 instants a coarse step:
    the two-step graph is the largest that is made."""
    _, most = run_child(tmp_path, 6, 2, 10**9)
    assert most <= 2 * 1024 * 8  # at most eight nodes an instant


def test_a_long_graph_that_cannot_be_made_leaves_the_short_ones(tmp_path):
    """Two levels: 7 launches a replayed step (9 launched level by level)."""
    assert run_child(tmp_path, 2, 0, 10**9)[0] == 32 * 7
    launches, most = run_child(tmp_path, 2, 0, 40)
    assert most > 40  # a long graph was refused
    assert launches == 32 * 7
