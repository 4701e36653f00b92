"""Rules of the host code that need no GPU, compiled from its headers or its
text."""
import os
import re
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

# touch_pages with the runtime's answer given: memory it may write holds a
# zeroed byte per page afterwards, other memory faults on a write
TOUCH = r"""
#include <sys/mman.h>
#include <unistd.h>
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstring>
enum { cudaSuccess = 0 };
enum { cudaMemoryTypeUnregistered = 0, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged };
struct cudaPointerAttributes { int type; };
static int answer_status, answer_type;
int cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  a->type = answer_type;
  return answer_status;
}
int cudaGetLastError() { return 0; }
%s
int main() {
  const size_t bytes = (8 << 20) + 123;
  const int none = PROT_NONE, both = PROT_READ | PROT_WRITE, flags = MAP_PRIVATE | MAP_ANONYMOUS;
  for (int type : {cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged}) {
    answer_type = type;
    touch_pages(mmap(nullptr, bytes, none, flags, -1, 0), bytes);
  }
  answer_type = cudaMemoryTypeUnregistered;
  answer_status = 1;  // the runtime cannot tell
  touch_pages(mmap(nullptr, bytes, none, flags, -1, 0), bytes);
  answer_status = cudaSuccess;
  touch_pages(nullptr, bytes);
  char* p = static_cast<char*>(mmap(nullptr, bytes, both, flags, -1, 0));
  std::memset(p, 1, bytes);
  touch_pages(p, bytes);
  const size_t page = std::max(4096l, sysconf(_SC_PAGESIZE));
  for (size_t k = 0; k < bytes; ++k)
    if (p[k] != (k %% page ? 1 : 0)) return 1;
  return 0;
}
"""


def test_pages_are_touched_in_unregistered_host_memory_only(tmp_path):
    text = open(os.path.join(build.CSRC, "api.cpp")).read()
    fn = re.search(r"^static void touch_pages\(.*?^}$", text, re.S | re.M).group(0)
    src, exe = tmp_path / "touch.cpp", tmp_path / "touch"
    src.write_text(TOUCH % fn)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fopenmp", str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_rules(tmp_path):
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text(CHECKS)
    inc = [build.INCLUDE, build.CSRC, os.path.join(build._cuda_home(), "include")]
    subprocess.run(["g++", "-std=c++17", "-O1", *["-I" + i for i in inc], str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
