"""Host-side comparison of tabulations (cvweno_internal.cuh, same_norms): decided by the members that
the batch reads, not by the padding behind them or by the cell size (compiled and run without a GPU)."""
import os
import subprocess

from paper_2601_16911_gb300 import build as B

SOURCE = r"""
#include <cstdio>
#include <cstring>
#include <new>
#include "cvweno_internal.cuh"
using namespace cvw;

template <int P>
int check() {
  using T = PackedTables<2, P>;
  alignas(T) static unsigned char mem[2][sizeof(T)];
  T* t[2];
  for (int k = 0; k < 2; ++k) {  // equal members over different bytes
    memset(mem[k], k ? 0xff : 0x00, sizeof(T));
    t[k] = reinterpret_cast<T*>(mem[k]);
    for (int my = 0; my < T::NY1; ++my)
      for (int p = 0; p < T::MP; ++p) t[k]->sigma2[my][p] = make_float2(1.0f + my, 0.5f * p);
    for (int e = 0; e < T::NR2; ++e) t[k]->R2[e] = make_float2(0.25f * e, -1.0f * e);
    for (int m = 0; m < T::ND; ++m) t[k]->tscale[m] = 3.0f * k + m;
  }
  int bad = same_norms(*t[0], *t[1]) ? 0 : 1;
  t[1]->R2[T::NR2 - 1].y += 1.0f;
  bad += same_norms(*t[0], *t[1]) ? 2 : 0;
  t[1]->R2[T::NR2 - 1] = t[0]->R2[T::NR2 - 1];
  t[1]->sigma2[0][0].x += 1.0f;
  bad += same_norms(*t[0], *t[1]) ? 4 : 0;
  printf("p = %d: %d\n", P, bad);
  return bad;
}

int main() { return check<1>() + check<2>() + check<3>() + check<4>(); }
"""


def test_same_norms_reads_members_only(tmp_path):
    src, exe = tmp_path / "norms.cu", tmp_path / "norms"
    src.write_text(SOURCE)
    cmd = [B._nvcc(), *B.ARCH, "-O0", "-std=c++17", "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"), str(src), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
