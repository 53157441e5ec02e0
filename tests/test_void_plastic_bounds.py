"""CPU check of vp_cluster (post_kernels.cuh), the look-up of a pixel's final
void-plastic cluster: it reads the scratch of the labelling at indices inside
the image only, whatever a labelling that gave up has left there (any label, any
target, any root), and returns a pixel of the image or -1.  The scratch lies in a
larger array whose margins hold values that would be returned or followed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda/include"

SRC = r"""
#include <cstdio>
#include <random>
#include <vector>
#include "post_kernels.cuh"
int main() {
  std::mt19937_64 g(1);
  const int64_t n = 64;
  const int32_t odd[] = {-2147483647 - 1, -65, -2, -1, 64, 65, 127, 2147483647};
  long bad = 0, found = 0;
  for (int k = 0; k < 200000; k++) {
    // reads outside [0, n) would meet the margins' 5, an index inside
    std::vector<int32_t> T(3 * n, 5), F(3 * n, 5);
    auto any = [&]() { return g() % 3 ? (int32_t)(g() % n) : odd[g() % 8]; };
    for (int i = 0; i < n; i++) T[n + i] = any(), F[n + i] = any();
    const int32_t r = any();
    const int32_t f = epfft::vp_cluster(r, T.data() + n, F.data() + n, n);
    // the same by the definition
    int32_t want = -1;
    if (r >= 0 && r < n && T[n + r] >= 0 && T[n + r] < n) want = F[n + T[n + r]];
    if (want < 0 || want >= n) want = -1;
    bad += f != want;
    found += f >= 0;
  }
  printf("%ld %ld\n", bad, found);
}
"""


def test_lookup_stays_inside_the_image(tmp_path):
    if not shutil.which("g++") or not os.path.isdir(CUDA):
        pytest.skip("needs g++ and the CUDA headers")
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=address,undefined", "-I",
                    os.path.join(ROOT, "paper_0802_2488_gb300", "csrc"), "-I", CUDA, str(tmp_path / "t.cpp"), "-o", exe],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert int(out[0]) == 0 and int(out[1]) > 10000


def test_the_relabelling_uses_it():
    src = open(os.path.join(ROOT, "paper_0802_2488_gb300", "csrc", "post_kernels.cu")).read()
    assert "vp.final_root[b + vp.target" not in src and "vp_cluster(lab[b + x]" in src
