"""Gather and store forms of the tensor-core contraction (CPU, compiled with the host compiler):
wherever a plan takes vector accesses, the general offsets of the elements they cover are adjacent
and the first is aligned, over orders, sizes and strides of up to three dims a side."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_05285_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <algorithm>
#include "pv_batch.cuh"
using namespace pv;
static int off(int i, int n, const int* sz, const int* st) {
  int o = 0;
  for (int d = n - 1; d >= 0; --d) { o += (i % sz[d]) * st[d]; i /= sz[d]; }
  return o;
}
static int total(int n, const int* sz) { int t = 1; for (int d = 0; d < n; ++d) t *= sz[d]; return t; }
int main() {
  const int S[] = {2, 3, 4, 6, 16};
  long long seen[6] = {0, 0, 0, 0, 0, 0};
  for (int a : S) for (int b : S) for (int c : S) for (int e : S) {
    // a tensor of dims (a, b, c, e) in each order of its dims as rows (two) and contraction (two)
    int sz[4] = {a, b, c, e}, st[4] = {b * c * e, c * e, e, 1}, p[4] = {0, 1, 2, 3};
    do {
      TcSpec t = TcSpec();
      t.nr = 2; t.nk = 2; t.nc = 1;
      for (int d = 0; d < 2; ++d) {
        t.rs[d] = sz[p[d]]; t.rP[d] = st[p[d]];
        t.ks[d] = sz[p[2 + d]]; t.kP[d] = st[p[2 + d]]; t.kQ[d] = d == 1 ? 1 : t.ks[1];
      }
      t.cs[0] = 16; t.cQ[0] = total(2, t.ks); t.cC[0] = total(2, t.rs);
      t.rC[1] = 1; t.rC[0] = t.rs[1];
      const int R = total(2, t.rs), K = total(2, t.ks);
      tc_forms(t, true, true, true, true, true);
      ++seen[t.modeP];
      if (t.pairP) ++seen[3];
      for (int i = 0; i < R; ++i)
        for (int k = 0; k < K; ++k) {
          const int o = off(i, 2, t.rs, t.rP) + off(k, 2, t.ks, t.kP);
          if (t.modeP == TC_VEC_K && (K % 4 || (k % 4 == 0 ? o % 4 : o != 1 + off(i, 2, t.rs, t.rP) + off(k - 1, 2, t.ks, t.kP)))) return 1;
          if (t.modeP == TC_VEC_T && (R % 4 || (i % 4 == 0 ? o % 4 : o != 1 + off(i - 1, 2, t.rs, t.rP) + off(k, 2, t.ks, t.kP)))) return 2;
          if (t.pairP && (K % 2 || (k % 2 == 0 ? o % 2 : o != 1 + off(i, 2, t.rs, t.rP) + off(k - 1, 2, t.ks, t.kP)))) return 3;
        }
      // the same dims as rows and columns of C
      t.nc = 2;
      for (int d = 0; d < 2; ++d) {
        t.rC[d] = st[p[d]]; t.cs[d] = sz[p[2 + d]]; t.cC[d] = st[p[2 + d]]; t.cQ[d] = 1;
      }
      tc_forms(t, true, true, true, true, true);
      if (t.vecC) ++seen[4];
      if (t.vecC)
        for (int i = 0; i < R; ++i)
          for (int k = 0; k < K; ++k) {
            const int o = off(i, 2, t.rs, t.rC) + off(k, 2, t.cs, t.cC);
            if (K % 4 || (k % 4 == 0 ? o % 4 : o != 1 + off(i, 2, t.rs, t.rC) + off(k - 1, 2, t.cs, t.cC))) return 4;
          }
      tc_forms(t, false, false, false);
      if (t.modeP != TC_SCALAR || t.modeQ != TC_SCALAR || t.pairP || t.pairQ || t.vecC) return 5;
    } while (std::next_permutation(p, p + 4));
  }
  for (int k = 0; k < 5; ++k)
    if (!seen[k]) return 6;
  return 0;
}
"""


def test_vector_forms_cover_adjacent_aligned_elements(tmp_path):
    src, exe = tmp_path / "forms.cpp", tmp_path / "forms"
    src.write_text(SOURCE)
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    if r.returncode:
        pytest.fail(r.stderr[-2000:])
    assert subprocess.run([str(exe)]).returncode == 0
