"""The marks that note in which epoch of the cell list a free-surface cell emptied
(host arithmetic, compiled from the library's header)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "lb_common.cuh"
using namespace lbgb;
template <class Real>
static int check() {
  // every epoch of a 32-bit step counter: no zero, no density, no two alike (the
  // marks fall strictly, so neighbours differ)
  const unsigned epochs = unsigned((1ull << 32) / FS_EPOCH);
  Real last = Real(0);
  for (unsigned e = 0; e < epochs; ++e) {
    const Real m = fs_mark(e, Real(0));
    if (!(m < last) || !(m > Real(-1e-3))) { std::printf("epoch %u\n", e); return 1; }
    last = m;
  }
  return 0;
}
int main() { return check<float>() || check<double>(); }
"""


def test_marks_of_all_epochs_differ(tmp_path):
    src, exe = tmp_path / "marks.cu", tmp_path / "marks"
    src.write_text(SOURCE)
    nvcc = "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc if os.path.exists(nvcc) else "nvcc", "-std=c++17", "-O2", "-I",
                    os.path.join(ROOT, "paper_0912_4230_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
