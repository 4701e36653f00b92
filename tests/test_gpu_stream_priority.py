"""Priorities of the captured steps' kernels against the bound stream's."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# cudaGraphInstantiate in front of the runtime's: writes down whether the graph
# runs by its nodes' priorities, and the least and the greatest of its kernels
SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>
#include <cuda_runtime_api.h>
#define NEXT(f) ((__typeof__(&f))dlsym(RTLD_NEXT, #f))
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* exec, cudaGraph_t graph, unsigned long long flags) {
  size_t n = 0;
  NEXT(cudaGraphGetNodes)(graph, 0, &n);
  cudaGraphNode_t* v = malloc(n * sizeof *v);
  NEXT(cudaGraphGetNodes)(graph, v, &n);
  int lo = 1000, hi = -1000;
  for (size_t k = 0; k < n; ++k) {
    enum cudaGraphNodeType t;
    cudaLaunchAttributeValue a;
    NEXT(cudaGraphNodeGetType)(v[k], &t);
    if (t != cudaGraphNodeTypeKernel) continue;
    if (NEXT(cudaGraphKernelNodeGetAttribute)(v[k], cudaLaunchAttributePriority, &a) != cudaSuccess) abort();
    if (a.priority < lo) lo = a.priority;
    if (a.priority > hi) hi = a.priority;
  }
  free(v);
  FILE* f = fopen(getenv("PRIORITY_FILE"), "w");
  fprintf(f, "%d %d %d", (flags & cudaGraphInstantiateFlagUseNodePriority) != 0, hi, lo);
  fclose(f);
  return NEXT(cudaGraphInstantiate)(exec, graph, flags);
}
"""
CHILD = """
import sys
sys.path.insert(0, {root!r})
import torch
from paper_1601_06984_gb300 import lbm, workloads as W
m = W.config_tgv3d({n})
streams = [torch.cuda.ExternalStream(p) if p == 0 else torch.cuda.Stream(priority=p) for p in {priorities}]
s = lbm.Sim(m, 19, 1.6, precision=1, stream=streams[0])
for t in streams:  # bound again to each
    s.bind(stream=t)
    s.init(*W.tgv_fields(m, 0.01))
    s.step(2)
    torch.cuda.synchronize()
    print(open({out!r}).read())
"""


def graphs(tmp_path, n, priorities):
    """(nodes' priorities in force, least, greatest) of the step graph, per bound stream."""
    src, so, out = tmp_path / "shim.c", tmp_path / "shim.so", tmp_path / "priorities"
    src.write_text(SHIM)
    sys.path.insert(0, ROOT)
    from paper_1601_06984_gb300.build import _cuda_home
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-I" + os.path.join(_cuda_home(), "include"), str(src), "-o", str(so),
                    "-ldl"], check=True)
    code = CHILD.format(root=ROOT, n=n, priorities=list(priorities), out=str(out))
    env = dict(os.environ, LD_PRELOAD=str(so), PRIORITY_FILE=str(out))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return [tuple(int(x) for x in l.split()) for l in r.stdout.splitlines()]


def test_priorities_follow_the_bound_stream(tmp_path):
    """Bricks at the bound stream's, the chain one level above, also after
    binding to another stream (0 is the default stream's, the device's least)."""
    assert graphs(tmp_path, 32, (0, -1, -2, 0)) == [(1, 0, -1), (1, -1, -2), (1, -2, -3), (1, 0, -1)]


def test_large_meshes_run_at_the_bound_stream_priority(tmp_path):
    assert [g[0] for g in graphs(tmp_path, 128, (0, -1))] == [0, 0]
