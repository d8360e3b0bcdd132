"""The CG kernel's byte offsets into its field and the rule for their width, from the header that the
kernel includes, compiled for the host, against 64-bit arithmetic: fields around and above 4 GB (2^29
slots) included."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2303_00790_gb300", "csrc", "cg_offsets.cuh")
PROGRAM = r"""
#include "%s"
#include <cstdio>
#include <initializer_list>
template <int B, typename O> int check(int64_t n) {
  const int64_t B3 = B * B * B, bricks = n / B3;
  const int64_t stride[3] = {1, B, (int64_t)B * B};
  int bad = 0;
  const O zero = kscf::cg_zero<O>(n, 4096);
  bad += zero != 8ull * (uint64_t)(n + 2048);
  const int64_t at[] = {0, bricks / 2, bricks - 1};
  for (int64_t brick : at)
    for (int64_t li = 0; li < B3; li += 7) {
      bad += kscf::cg_own<O, B>((int)(brick * B3 + li)) != 8ull * (uint64_t)(brick * B3 + li + B3);
      for (int f = 0; f < 6; f++)   // the slot at distance 1 beyond the face, seen from the base
        for (int64_t m : {(int64_t)0, bricks - 1}) {
          const int64_t inside = m * B3 + li + ((f & 1) ? -B : B) * stride[f >> 1];
          bad += kscf::cg_face<O, B>((int)m, (int)li, f, zero) != 8ull * (uint64_t)(inside + B3);
          bad += kscf::cg_face<O, B>(-1, (int)li, f, zero) != zero + 8ull * (uint64_t)B3;
        }
    }
  return bad;
}
int main() {
  int bad = 0;
  for (int64_t n : {(int64_t)1 << 20, ((int64_t)1 << 29) - 16384, ((int64_t)1 << 29) + 4096, ((int64_t)1 << 31) - 4096})
    bad += (kscf::cg_wide(n, 4096, 8) ? check<8, uint64_t>(n) : check<8, uint32_t>(n)) +
           (kscf::cg_wide(n, 4096, 16) ? check<16, uint64_t>(n) : check<16, uint32_t>(n));
  std::printf("%%d\n", bad);
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_offsets_of_large_fields(tmp_path):
    src = tmp_path / "offsets.cpp"
    src.write_text(PROGRAM % HEADER)
    exe = str(tmp_path / "offsets")
    subprocess.run(["g++", "-std=c++17", "-O1", str(src), "-o", exe], check=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout.strip() == "0"
