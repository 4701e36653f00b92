"""Rules of the host code that need no GPU, compiled from its headers."""
import os
import subprocess

from paper_1601_06984_gb300 import build

CHECKS = r"""
#include <cstdio>
#include "lbm_internal.h"
int main() {
  int bad = 0;
  auto check = [&](bool ok, const char* what, long long a, long long b) {
    if (!ok) std::printf("%s: %lld %lld\n", what, a, b), ++bad;
  };
  // reverse ghost kernels: every block size has a thread for each of up to 2^18
  // items, and blocks for no more than the work
  for (int block : {32, 64, 128, 256})
    for (long long n : {0ll, 1ll, 31ll, 32ll, 33ll, 1000ll, 52288ll, (1ll << 18) - 1, 1ll << 18, 1ll << 24}) {
      const long long g = lbm::adj_grid(n, block), want = n < (1ll << 18) ? n : 1ll << 18;
      check(g >= 1 && g * block >= want, "adj_grid has too few threads", n, block);
      check(g == 1 || (g - 1) * block < want, "adj_grid has idle blocks", n, block);
    }
  return bad != 0;
}
"""


def test_rules(tmp_path):
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text(CHECKS)
    inc = [build.INCLUDE, build.CSRC, os.path.join(build._cuda_home(), "include")]
    subprocess.run(["g++", "-std=c++17", "-O1", *["-I" + i for i in inc], str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
