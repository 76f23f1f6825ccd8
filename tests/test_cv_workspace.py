"""The scratch of the control variate's training: rssri_cv_train sizes it once, for the larger
of its batch and its evaluation set, and uses it with both, so the size for m rows must cover
every smaller number of rows.  Host arithmetic only."""
import os
import subprocess

from paper_2005_12338_gb300 import build

CHECK = r"""
#include <cstdio>
#include "cv_mlp.cuh"
int main() {
  size_t need = 0;
  for (int m = 1; m <= 65536; ++m) {
    int ks, kc;
    rssri::cv_row_chunks(m, &ks, &kc);
    if (ks < 1 || kc < 1 || (long long)ks * kc < m || (long long)(ks - 1) * kc >= m) {
      std::printf("chunks of %d rows: %d of %d\n", m, ks, kc);
      return 1;
    }
    const size_t here = (size_t)ks * (rssri::CV_HIDDEN + rssri::CV_HIDDEN * rssri::CV_NFEAT) + 128;
    if (here > need) need = here;
    if (rssri::cv_sum_floats(m) < need) {
      std::printf("%d rows: %zu floats, %zu needed up to there\n", m, rssri::cv_sum_floats(m), need);
      return 1;
    }
  }
  return 0;
}
"""


def test_scratch_covers_every_smaller_batch(tmp_path):
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(CHECK)
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
