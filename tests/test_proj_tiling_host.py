"""The tiling of the decoder stack's projections (csrc/proj_tiling.h) on the host: the
one of least cost among all numbers of tiles, as counting through every one of them
finds it, in a few evaluations at any number of rows; and the workspace query, which
asks for six of them, stays quick at the largest batches."""
import ctypes
import os
import subprocess
import time

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "proj_tiling.h"
using namespace jet;

// every number of tiles, in order; the first of least cost
static Tiling counted(int N, int O, int K, bool split, int pairs) {
  const int least = (N + 255) / 256;
  Tiling best{};
  long long best_cost = -1;
  for (int c = least; c <= 2 * least + 2; ++c) {
    Tiling t{};
    t.Nt = ((N + c - 1) / c + 15) / 16 * 16;
    t.n_tt = (N + t.Nt - 1) / t.Nt;
    t.otiles = (O + 127) / 128;
    t.groups = (t.otiles + 1) / 2;
    t.nkb = (K + 63) / 64;
    t.tail_group = t.groups;
    const int units = t.groups * t.n_tt;
    t.splits = 1;
    while (split && units * (t.splits + 1) <= pairs && t.nkb / (t.splits + 1) >= 8) ++t.splits;
    const long long all = (long long)units * t.splits;
    long long cost = (all + pairs - 1) / pairs * ((t.nkb + t.splits - 1) / t.splits) * (t.Nt + 80);
    if (best_cost < 0 || cost < best_cost) {
      best = t;
      best_cost = cost;
    }
    const int full = units / pairs, head = full * pairs / t.n_tt;
    if (t.splits > 1 || full == 0 || head == t.groups) continue;
    for (int ct = c + 1; ct <= 4 * c; ++ct) {
      Tiling u = t;
      u.tail_Nt = ((N + ct - 1) / ct + 15) / 16 * 16;
      u.tail_n_tt = (N + u.tail_Nt - 1) / u.tail_Nt;
      u.tail_group = head;
      const long long rest = (long long)(t.groups - head) * u.tail_n_tt;
      cost = (full * (t.Nt + 80) + (rest + pairs - 1) / pairs * (u.tail_Nt + 80)) * t.nkb;
      if (cost * 100 < best_cost * 97) {
        best = u;
        best_cost = cost;
      }
    }
  }
  return best;
}

int main() {
  std::srand(7);
  for (int it = 0; it < 20000; ++it) {
    const int N = it < 3000 ? it + 1 : 1 + std::rand() % (it % 50 ? 3000 : 20000);
    const int O = 16 * (1 + std::rand() % (it % 3 ? 200 : 2000));
    const int K = 16 * (1 + std::rand() % 800);
    const bool split = std::rand() % 4 != 0;
    const int pairs = it % 5 ? 76 : 1 + std::rand() % 100;
    const Tiling a = projection_tiling(N, O, K, split, pairs), b = counted(N, O, K, split, pairs);
    if (a.n_tt != b.n_tt || a.Nt != b.Nt || a.otiles != b.otiles || a.groups != b.groups ||
        a.nkb != b.nkb || a.splits != b.splits || a.tail_group != b.tail_group ||
        a.tail_n_tt != b.tail_n_tt || a.tail_Nt != b.tail_Nt) {
      std::printf("N %d O %d K %d split %d pairs %d: %d x %d, tail %d x %d; %d x %d, tail %d x %d\n",
                  N, O, K, split, pairs, a.n_tt, a.Nt, a.tail_n_tt, a.tail_Nt, b.n_tt, b.Nt,
                  b.tail_n_tt, b.tail_Nt);
      return 1;
    }
  }
  return 0;
}
"""


def test_tiling_is_the_counted_one(tmp_path, repo_root):
    src, exe = tmp_path / "tiling.cpp", tmp_path / "tiling"
    src.write_text(HARNESS)
    inc = os.path.join(repo_root, "paper_2609_33874_gb300", "csrc")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-Wall", "-Werror", "-I", inc,
                    str(src), "-o", str(exe)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout


def test_workspace_query_does_not_grow_with_the_rows(jet):
    # 500,000 rows: 1.1 s when every number of tiles was tried, well under 1 ms now
    n = jet.jet_sizes()
    for name, x in dict(R=1, C=1, N=500000, T=500000, V=8, total_prefix=8, max_prefix=8, min_cand=1,
                        max_cand=1, max_rows=500000, max_len=500000).items():
        setattr(n, name, x)
    dims = jet.make_dims(jet.DTYPE_BF16, Hq=4, Hkv=2, d=64, D=512, Hl=2, dk=128, dv=64)
    best = 1e9
    for _ in range(3):
        t = time.perf_counter()
        assert jet.library().jet_stack_workspace_bytes(ctypes.byref(n), ctypes.byref(dims), 2048) > 0
        best = min(best, time.perf_counter() - t)
    assert best < 0.1
