"""The attention kernel's work items (csrc/attend_items.h, plain arithmetic) on the
host: over random plans, and layouts that agree with their sizes or do not, every item
stays inside the batch and inside the partials the plan's workspace holds, and the
items of a request that fits cover each of its rows and keys once."""
import os
import subprocess

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "attend_items.h"
using namespace jet;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

static int rnd(int lo, int hi) { return lo + std::rand() % (hi - lo + 1); }

static int request(const ItemPlan& a, int Hq, int r, int n0, int nr, int p0, int P) {
  const RequestCut cut = request_cut(a, n0, nr, p0, P);
  const int nq = cut.nq, sp = cut.sp;
  CHECK(nq >= 1 && nq <= a.qgroups && sp >= 1 && sp <= a.splits);
  std::vector<int> seen(size_t(nr) * P, 0);
  for (int qb = 0; qb < nq; ++qb)
    for (int split = 0; split < sp; ++split) {
      const ItemGeo e = item_geo_at(a, r, a.Hkv - 1, qb, split, n0, nr, p0, P, cut);
      CHECK(e.ok && e.splits_r == sp);
      CHECK(e.nv >= 1 && e.n0 >= 0 && e.n0 + e.row0 + (e.nv + a.g - 1) / a.g <= a.N);
      CHECK(e.k_begin < e.k_end && e.p0 >= 0 && e.p0 + e.k_end <= a.total_prefix);
      // where the partial of the block's last vector goes
      const int gv = e.vbase + e.nv - 1;
      const long long at = ((long long)e.split * a.N + e.n0 + gv / a.g) * Hq + e.kh * a.g + gv % a.g;
      CHECK(at < (long long)a.splits * a.N * Hq);
      CHECK((e.nct > 0) == (split == sp - 1 && a.has_cand && nr > 1));
      for (int n = e.row0; n < e.row0 + e.nv / a.g; ++n)
        for (int k = e.k_begin; k < e.k_end; ++k) ++seen[size_t(n) * P + k];
    }
  for (int x : seen) CHECK(x == 1);
  // nothing past the items
  CHECK(!item_geo_at(a, r, 0, nq, 0, n0, nr, p0, P, cut).ok);
  CHECK(!item_geo_at(a, r, 0, 0, sp, n0, nr, p0, P, cut).ok);
  return 0;
}

static bool fits(const ItemPlan& a, int n0, int nr, int p0, int P) {
  return request_cut(a, n0, nr, p0, P).nq > 0;
}

int main() {
  int fit = 0, left_out = 0;
  for (int it = 0; it < 4000; ++it) {
    std::srand(it);
    ItemPlan a{};
    a.R = rnd(1, 4);
    a.Hkv = rnd(1, 3);
    a.g = rnd(1, 128);
    a.rb = 128 / a.g;
    a.has_cand = rnd(0, 1);
    const int Hq = a.g * a.Hkv;
    std::vector<int> P, nr;
    int maxP = 0, maxn = 0;
    for (int r = 0; r < a.R; ++r) {
      P.push_back(rnd(1, 700));
      nr.push_back(rnd(1, 12));
      a.total_prefix += P[r];
      a.N += nr[r];
      if (P[r] > maxP) maxP = P[r];
      if (nr[r] > maxn) maxn = nr[r];
    }
    a.chunk = 64 * rnd(1, 12);
    a.splits = (maxP + a.chunk - 1) / a.chunk;
    a.qgroups = (maxn + a.rb - 1) / a.rb;
    int n0 = 0, p0 = 0;
    for (int r = 0; r < a.R; ++r) {
      CHECK(fits(a, n0, nr[r], p0, P[r]));
      if (request(a, Hq, r, n0, nr[r], p0, P[r])) return 1;
      n0 += nr[r];
      p0 += P[r];
    }
    // another batch's words under this plan: what fits is in bounds, the rest left out
    for (int t = 0; t < 20; ++t) {
      const int x = rnd(-20, a.N + 20), n = rnd(-3, a.N + 3), y = rnd(-100, a.total_prefix + 100),
                p = rnd(-10, a.total_prefix + 10);
      if (fits(a, x, n, y, p)) {
        ++fit;
        if (request(a, Hq, 0, x, n, y, p)) return 1;
      } else {
        ++left_out;
        CHECK(!item_geo_at(a, 0, 0, 0, 0, x, n, y, p, request_cut(a, x, n, y, p)).ok);
      }
    }
    // a prefix longer than the plan's chunks, inside the batch
    if (a.splits * a.chunk < a.total_prefix) {
      ++left_out;
      CHECK(!fits(a, 0, 1, 0, a.splits * a.chunk + 1));
    }
  }
  CHECK(fit > 1000 && left_out > 1000);
  const int big = 2147483647;
  ItemPlan a{};
  a.R = a.Hkv = a.g = a.splits = a.qgroups = 1;
  a.rb = 128;
  a.N = 10;
  a.total_prefix = 100;
  a.chunk = 128;
  CHECK(!fits(a, 0, big, 0, 10) && !fits(a, big, 1, 0, 10));
  CHECK(!fits(a, 0, 1, 0, big) && !fits(a, 0, 1, big, 10));
  CHECK(!fits(a, -big, 1, 0, 10) && !fits(a, 0, 1, -big, 10));
  return 0;
}
"""


def test_items_stay_inside_the_plan(tmp_path, repo_root):
    src, exe = tmp_path / "items.cpp", tmp_path / "items"
    src.write_text(HARNESS)
    inc = os.path.join(repo_root, "paper_2609_33874_gb300", "csrc")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-Wall", "-Werror", "-I", inc,
                    str(src), "-o", str(exe)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
