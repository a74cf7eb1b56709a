// How a projection of the decoder stack (proj_tc.cu) is cut into units of work: plain
// arithmetic, for the launches, the workspace plan and host tests.
#pragma once

namespace jet {

constexpr int kProjRows = 128;   // weight rows per CTA
constexpr int kProjK = 64;       // elements of a K slice
constexpr int kProjMaxNt = 256;  // rows of a token tile, at most

struct Tiling {
  int n_tt, Nt, otiles, groups, nkb, splits;  // groups: 256-row weight slices
  int tail_group, tail_n_tt, tail_Nt;  // slices from tail_group on in narrower tiles
};

// Token tiles of at most 256 rows (a multiple of 16: each CTA of a pair holds
// half); units of 256 weight rows on CTA pairs; K split while the units still
// fit the 76 SM pairs once, keeping at least 8 K slices per unit. A function
// of the shapes only, so that the workspace planned for a call matches the
// launch.
// The number of tiles is the one of least cost: rounds of the SM pairs, times K
// slices a unit, times a slice's time, which goes as Nt + 80 (the weights' share of
// the bytes an SM takes in; 64 to 110 in place of 80 choose alike but for a few
// sizes). Always the fewest tiles left the last round half empty: four layers of
// D 4,096 and Dff 12,288 took 525 us of 178 rows, now 513; 643 of 355, now 634; 715
// of 444, now 691; 851 of 555, now 808; 1,802 of 2,800, now 1,688. Splits over more
// than one round gain up to 1 % there, but 355 rows take 1 - 2 % more.
// Where the weight slices past the full rounds would leave most pairs idle, they are
// a tail in narrower token tiles that all pairs share (the gate and up projection of
// 24,576 features: 76 slices, then 20 in three tiles each): the stack takes 496 us of
// 178 rows without it, 481 with; 618 of 355, now 601; 685 of 444, now 674.
// Tiles are evened out to multiples of 16 rows, so at most 16 widths come into
// question; `tiles_after` goes from one to the next (counting every number of tiles
// instead, the search grew with the square of the rows: 99,000 rows of three narrow
// layers, D 256, waited 57 ms for the host, where the GPU takes 5.1).
inline Tiling projection_tiling(int N, int O, int K, bool split, int pairs) {
  const int least = (N + kProjMaxNt - 1) / kProjMaxNt;
  auto tiles = [&](int c, int& nt, int& n_tt) {  // c tiles, or fewer once rounded
    nt = ((N + c - 1) / c + 15) / 16 * 16;
    n_tt = (N + nt - 1) / nt;
  };
  // the smallest number of tiles that makes them narrower than nt
  auto tiles_after = [&](int nt, int none) { return nt <= 16 ? none : (N + nt - 17) / (nt - 16); };
  auto rounds = [&](long long units) { return (units + pairs - 1) / pairs; };
  Tiling best{};
  long long best_cost = -1;
  const int most = 2 * least + 2;
  for (int c = least, next; c <= most; c = next) {
    Tiling t{};
    tiles(c, t.Nt, t.n_tt);
    next = tiles_after(t.Nt, most + 1);
    t.otiles = (O + kProjRows - 1) / kProjRows;
    t.groups = (t.otiles + 1) / 2;
    t.nkb = (K + kProjK - 1) / kProjK;
    t.tail_group = t.groups;
    const int units = t.groups * t.n_tt;
    t.splits = 1;
    while (split && units * (t.splits + 1) <= pairs && t.nkb / (t.splits + 1) >= 8) ++t.splits;
    const long long per_kb = (t.nkb + t.splits - 1) / t.splits;
    long long cost = rounds((long long)units * t.splits) * per_kb * (t.Nt + 80);
    if (best_cost < 0 || cost < best_cost) {
      best = t;
      best_cost = cost;
    }
    // the same, with the slices past its full rounds in narrower tiles, up to four
    // times the number that any c of this width stands for
    const int full = units / pairs, head = full * pairs / t.n_tt;
    if (t.splits > 1 || full == 0 || head == t.groups) continue;
    const int last = 4 * (next <= most ? next - 1 : most);
    for (int ct = c + 1; ct <= last;) {
      Tiling u = t;
      tiles(ct, u.tail_Nt, u.tail_n_tt);
      u.tail_group = head;
      cost = (full * (t.Nt + 80) +
              rounds((long long)(t.groups - head) * u.tail_n_tt) * (u.tail_Nt + 80)) * t.nkb;
      if (cost * 100 < best_cost * 97) {
        best = u;
        best_cost = cost;
      }
      ct = tiles_after(u.tail_Nt, last + 1);
    }
  }
  return best;
}

}  // namespace jet
