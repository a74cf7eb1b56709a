// The work items of the tensor-core attention kernel (attend_tc.cu): how a
// request's rows and prefix are cut into (kv head, query block, prefix chunk)
// items, and which requests of a device layout fit the plan that the workspace
// was sized for. Plain arithmetic, for the kernels and for host tests.
#pragma once

#ifdef __CUDACC__
#define JET_HD __host__ __device__ __forceinline__
#else
#define JET_HD inline
#endif

namespace jet {

constexpr int kItemTile = 64;  // keys per tile

// What the items of a launch are cut by.
struct ItemPlan {
  int R, N, total_prefix, Hkv;
  int g, rb;      // query heads per kv head; rows per query block
  int chunk;      // prefix keys per chunk
  int splits;     // chunks per request, at most
  int qgroups;    // query blocks per request, at most
  int has_cand;   // the batch has fed candidate tokens (F > 0)
};

// How a request is cut: nq query blocks of rb rows, and its P prefix keys in sp
// chunks of nearly equal length - `per` 64-key tiles each, at most ceil(P / chunk)
// of them, none empty (the last also takes the candidates' own keys). nq is 0 for a
// request that is left out.
struct RequestCut {
  int nq, sp, per;
};

// The cut of a request of rows [n0, n0 + nr) and prefix [p0, p0 + P), as a device
// layout gives it, if it lies in the batch and within the plan. The partials'
// workspace holds `splits` chunks of every row, so a request with more is not
// worked on at all. (Taken once a request: the divisions are what it costs.)
JET_HD RequestCut request_cut(const ItemPlan& a, int n0, int nr, int p0, int P) {
  RequestCut c{};
  if (nr < 1 || nr > a.N || n0 < 0 || n0 > a.N - nr) return c;
  if (P < 1 || P > a.total_prefix || p0 < 0 || p0 > a.total_prefix - P) return c;
  const int tiles = (P + kItemTile - 1) / kItemTile;
  const int s = P <= a.chunk ? 1 : (P + a.chunk - 1) / a.chunk;
  c.per = s == 1 ? tiles : (tiles + s - 1) / s;
  c.sp = s == 1 ? 1 : (tiles + c.per - 1) / c.per;
  const int nq = nr <= a.rb ? 1 : (nr + a.rb - 1) / a.rb;
  if (nq <= a.qgroups && c.sp <= a.splits) c.nq = nq;
  return c;
}

// Geometry of one work item (request r, key/value head kh, query block qb,
// prefix chunk split); every role derives it the same way from the item.
struct ItemGeo {
  int r, kh, n0, nr, p0, P, row0, vbase, nv, k_begin, k_end, npt, nct, ntiles, splits_r, f_begin;
  int split;
  bool ok;
};

// The item's geometry, from its request's rows, prefix and cut.
JET_HD ItemGeo item_geo_at(const ItemPlan& a, int r, int kh, int qb, int split, int n0, int nr,
                           int p0, int P, const RequestCut& cut) {
  ItemGeo e{};
  e.r = r;
  e.kh = kh;
  e.split = split;
  if (r < 0 || r >= a.R || kh < 0 || kh >= a.Hkv || qb < 0 || qb >= cut.nq || split < 0 ||
      split >= cut.sp)
    return e;
  e.n0 = n0;
  e.nr = nr;
  e.p0 = p0;
  e.P = P;
  e.row0 = qb * a.rb;
  e.vbase = e.row0 * a.g;
  const int left = e.nr - e.row0;
  e.nv = (left < a.rb ? left : a.rb) * a.g;
  e.splits_r = cut.sp;
  e.k_begin = e.split * cut.per * kItemTile;
  e.k_end = e.k_begin + cut.per * kItemTile;
  if (e.k_end > e.P) e.k_end = e.P;
  e.npt = (e.k_end - e.k_begin + kItemTile - 1) / kItemTile;
  // the request's last chunk also takes its candidates' own keys: the F_r fed
  // tokens, as extra 64-key tiles masked per row to the row's candidate and
  // position (Sec. 4.1: a candidate attends to its own earlier tokens only)
  e.f_begin = e.n0 - e.r;  // fed-token index of the request's first fed row
  const int F_r = e.nr - 1;
  e.nct = (e.split == e.splits_r - 1 && a.has_cand && F_r > 0) ? (F_r + kItemTile - 1) / kItemTile
                                                               : 0;
  e.ntiles = e.npt + e.nct;
  e.ok = true;
  return e;
}

}  // namespace jet
