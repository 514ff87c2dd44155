"""The descending order of singular values is a permutation for any input (CPU, host compiler):
a truncation with infinities or NaN among its entries must not leave an index of a kept vector
unset, since the kernels address shared memory with it."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_05285_gb300", "csrc")

SOURCE = r"""
#include <cmath>
#include <limits>
#include "pv_batch.cuh"
using namespace pv;
template <typename T>
int run() {
  const T inf = std::numeric_limits<T>::infinity(), nan = std::numeric_limits<T>::quiet_NaN();
  const T bad[] = {nan, inf, -inf, std::numeric_limits<T>::max(), 0};
  for (int tall = 0; tall < 2; ++tall)
    for (int nc = 1; nc <= 9; ++nc)
      for (int k = 0; k < 5; ++k)
        for (int at = -1; at < nc; ++at) {   // column `at` (-1: all of them) holds the value
          const int len = tall ? nc + 2 : 12, m = tall ? len : nc, kk = nc < 4 ? nc : 4;
          std::vector<T> Y(nc * len), U(m * kk), out(m * kk), work(4 * (nc + 1) * (len + 2) + 4 * (m + 1) * (m + 2)),
              sig(nc + 4), red(64);
          for (int i = 0; i < nc * len; ++i) Y[i] = (T)std::sin(1.0 + 3 * i);
          for (int j = 0; j < nc; ++j)
            if (at < 0 || at == j) Y[j * len + j % len] = bad[k];
          std::vector<int> order(nc + 4, nc);   // an index that no column has
          double ls = 0;
          unsigned long long sweeps = 0;
          int flag = 0;
          OpTrunc<T> op{Y.data(), (long long)Y.size(), tall != 0, nc, len, m, kk, U.data(), (long long)U.size(),
                        out.data(), (long long)out.size(), &ls, 1, (T)1e-6, 8, &sweeps, nullptr};
          op(0, red.data(), &flag, work.data(), (long long)work.size(), order.data(), sig.data());
          std::vector<int> seen(nc + 1, 0);
          for (int j = 0; j < nc; ++j)
            if (order[j] < 0 || order[j] >= nc || seen[order[j]]++) return 1 + tall;
          // numbers in descending order, ties by index, before what is not one
          for (int j = 0; j + 1 < nc; ++j) {
            const T a = sig[order[j]], b = sig[order[j + 1]];
            if (b == b && (!(a == a) || a < b || (a == b && order[j] > order[j + 1]))) return 3;
          }
        }
  return 0;
}
int main() { return run<float>() ? 1 : (run<double>() ? 2 : 0); }
"""


def test_ranks_are_a_permutation(tmp_path):
    src, exe = tmp_path / "order.cpp", tmp_path / "order"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
