"""Host check of the bisection queue's launch (no GPU): `bisect_lanes` (csrc/stein.cu, compiled here
verbatim) gives each queued eigenvalue 4 to 32 lanes, and every entry needs its lanes among the
launch's threads, on a GPU of any number of SMs (full parts, partitions, a failed query).  The
launch has 4 threads per eigenvalue of all problems, rounded up to its blocks, and at most
that many entries."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STEIN = os.path.join(ROOT, "paper_1402_4247_gb300", "csrc", "stein.cu")

DRIVER = r"""
#include <cstdio>
#define __host__
#define __device__
%(consts)s
%(lanes)s
int main() {
  long bad = 0, checked = 0;
  for (int sms = 0; sms <= 176; ++sms)
    // numbers of eigenvalues around the one from which the queue is used (4 lanes per warp lane)
    for (long cap = sms * 32 + 1; cap <= sms * 32 + 5000; cap = cap * 5 / 4 + 1) {
      const long threads = (cap * BQ_LANES + SZ_THREADS - 1) / SZ_THREADS * SZ_THREADS;
      for (long cnt = 1; cnt <= cap; cnt = cnt < 64 ? cnt + 1 : cnt * 9 / 8) {
        const int ln = bisect_lanes(cnt, threads, 4 * sms);
        ++checked;
        if (ln < BQ_LANES || ln > 32 || (ln & (ln - 1))) ++bad;
        if (cnt * ln > threads) ++bad;                                       // an entry without its lanes
        if (ln < 32 && 2 * cnt * ln <= threads && cnt * ln <= 64L * sms) ++bad;  // idle schedulers
      }
    }
  printf("%%ld %%ld\n", bad, checked);
  return 0;
}
"""


def test_every_queue_entry_has_its_lanes(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    text = open(STEIN).read()
    consts = "\n".join(re.search(rf"constexpr int {c} = [^;]+;", text).group(0) for c in ("BQ_LANES", "SZ_THREADS"))
    m = re.search(r"__host__ __device__ inline int bisect_lanes\(.*?\n}\n", text, re.S)
    assert m, "bisect_lanes"
    kernel = text[text.index("stebz_bisect_kernel(int n"):]
    assert "bisect_lanes(cnt, gridDim.x * blockDim.x, " in kernel[:kernel.index("\n}\n")]
    src = tmp_path / "drv.cpp"
    src.write_text(DRIVER % {"consts": consts, "lanes": m.group(0)})
    exe = tmp_path / "drv"
    subprocess.run([cxx, "-O2", "-std=c++17", "-o", str(exe), str(src)], check=True)
    bad, checked = (int(v) for v in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert checked > 10000
    assert bad == 0
