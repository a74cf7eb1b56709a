// Prefix scan of a linear-attention layer's recurrent state in chunks on the
// 5th-generation tensor cores (Sec. 4.1: the prefix state is computed once and
// every candidate forks from it). The recurrence is the one of the fork:
//   S_t = a_t (S_{t-1} - b_t k_t (k_t^T S_{t-1})) + b_t k_t v_t^T,
//   o_t = S_t^T q_t / sqrt(dk)                    (gated delta rule)
// or S_t = a_t S_{t-1} + b_t k_t v_t^T (plain gated linear attention).
//
// Over a chunk of C = 64 tokens starting from S0, with the decay products
// g_r = a_0 ... a_r and G[r][i] = a_{i+1} ... a_r (i <= r), the state after
// token r is S_r = g_r S0 + sum_{i<=r} G[r][i] k_i d_i^T, where the d_i solve
//   d_r + b_r sum_{i<r} G[r][i] (k_r . k_i) d_i = b_r v_r - b_r g_r S0^T k_r
// (d_r = b_r v_r for gated linear attention). Writing the solution of
// (I + A) X = B with A[r][i] = b_r G[r][i] (k_r . k_i) (i < r) for
// B = diag(b) V and B = diag(b g) K as U and W gives d = U - W S0, so
//   O   = diag(g) Q S0 + (M o G) d,  M[r][i] = q_r . k_i (i <= r)
//   S_C = g_{C-1} S0 + K^T diag(G[C-1][.]) d.
// Per chunk: one MMA gives [K; Q] K^T (the k.k and q.k products, exact in
// float32 from bf16 inputs); T = (I + A)^{-1} is formed on the CUDA cores in
// 16 x 16 blocks (the diagonal blocks by substitution, the rest as small
// products, level by level); then, on the transposed state (TMEM lane = value
// column):
//   U^T = V^T (T diag(b))^T,  W^T = K^T (T diag(b g))^T
//   X   = S0^T [-W | g Q]         -> d^T - U^T and (g Q S0)^T
//   X  += d^T (M o G)^T           -> O^T (accumulated onto (g Q S0)^T)
//   Dst = g_{C-1} S0^T + (d G[C-1])^T K  -> the next S0^T
// Operands that are not bf16 (S0, T diag(.), W, g Q, d, M o G) enter the MMA
// as a sum of two bf16 numbers (hi + lo, hi = bf16(x), lo = bf16(x - hi)): the
// products hi.hi + hi.lo + lo.hi keep about 16 bits, so the state keeps
// float32-like accuracy over the whole prefix. Forming T costs 64^3 / 6 FMAs a
// chunk instead of the 64^2 / 2 per column of a substitution for all 256
// columns of U and W.
//
// One CTA per SM works through items (request, head), longest requests first, with
// two groups of eight warps. The solve group works
// one chunk ahead of the state: it forms A, M o G, T, T diag(b) and T diag(b g)
// of chunk j + 1 (none of which needs the state) and issues U and W, while the
// state group runs X, d, O and the new state of chunk j. Lane c of TMEM (value
// column c, and key column c of W) belongs to thread c of each warpgroup, which
// split the columns. What bounds it: the chain of the state group (X, d, O and
// S, the new operand: 5 to 6 us a chunk) and the instructions of the hi/lo
// splits (40 % of the issue slots); with one group doing both in turn a chunk
// took 11 us. 32 requests x 512 tokens x 16 heads: delta rule 338 -> 228 us, gated
// linear attention 199 -> 147 us; 3 x 2,000 - 4,000 tokens 595 -> 359 and 341 ->
// 222 us. The groups run on from one item into the next: a CTA per item fills and
// drains this chain every time, and its lengths come in no order (the above 228 ->
// 220 and 147 -> 141 us; 64 x 64 tokens 89 -> 62 and 64 -> 43 us; 24 x 100 - 4,000
// tokens 671 -> 500 and 416 -> 319 us). Where it was lost before: bank conflicts and
// address arithmetic in the inverse, one chunk's gates scanned inside its chain,
// outputs written before the next chunk's X (of gated linear attention: in the place
// of its state MMAs; 141 -> 138 us, 3 x 2,000 - 4,000 tokens 234 -> 213).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "jet_device.cuh"
#include "jet_internal.h"
#include "sm100_ptx.cuh"

namespace jet {
namespace {

using namespace sm100;

constexpr int kC = 64;         // tokens per chunk
constexpr int kD = 128;        // dk = dv handled by this kernel
constexpr int kGroup = 256;    // threads of one group (solve or state)
constexpr int kThreads = 2 * kGroup;
constexpr int kWalker = 160;   // the solve group's thread that steps through the chunks
constexpr uint64_t kDrainNs = 200000000ull;

// Shared memory (offsets from the 1024-byte aligned base). Operand tiles are
// K-major with 128-byte swizzling: 64 elements (128 bytes) per row, 8-row
// atoms of 1024 bytes, the 128-element dimension split into two slices.
// Each dk-slice of the token tiles holds [K0 | Q0 | K1 | Q1] (64 token rows
// each, buffer = chunk parity), so [K; Q] of a chunk is one 128-row operand.
constexpr uint32_t kKQSlice = 4 * 8192;
constexpr uint32_t kOffKQ = 0;
constexpr uint32_t kKQBuf = 16384;                  // from one parity's K to the other's
constexpr uint32_t kOffV = 2 * kKQSlice;            // V: 64 rows x 2 dv-slices
constexpr uint32_t kVSlice = 8192;
// [-W | g Q] hi, lo: MN-major (dk rows of 64 tokens), two N slices (-W, then
// g Q) of 128 rows; the first slices hold T diag(b) and T diag(b g) until W
constexpr uint32_t kOffWQh = 81920, kOffWQl = 114688;
constexpr uint32_t kWQSlice = 16384;
// (M o G) hi, lo: 64 rows (output token) x 64 tokens, one pair per chunk parity
constexpr uint32_t kOffM = 147456;
constexpr uint32_t kMBuf = 16384, kMLo = 8192;
// A of the solve and T = (I + A)^{-1}, the 16 x 16 blocks at and below the
// diagonal in f32 (blk)
constexpr uint32_t kBlk = 324, kPitch = 20;  // floats of a block and of its rows
constexpr uint32_t kOffA = 180224;
constexpr uint32_t kOffT = kOffA + 10 * kBlk * 4;
constexpr uint32_t kOffOut = kOffT + 10 * kBlk * 4;  // a chunk's outputs [64 tokens][kD] bf16
// the gates and their products of up to three chunks: a[64], b[64], in-warp
// products of a[64], g[64], G[C-1][64], g_{C-1}
constexpr uint32_t kVecFloats = 5 * 64 + 4;
constexpr uint32_t kOffVec = kOffOut + 16384;
constexpr uint32_t kOffBar = kOffVec + 3 * kVecFloats * 4;
// chunk descriptors {first token, end of the prefix, head, row of (request, head)}
// of eight chunks in turn; an empty one (no tokens) ends the CTA's sequence
constexpr uint32_t kOffRing = kOffBar + 128;
constexpr int kRing = 8;
constexpr uint32_t kOffWalk = kOffRing + kRing * 16;
constexpr uint32_t kSmemBytes = kOffWalk + 32 + 1024;
static_assert(kOffOut % 16 == 0 && kOffVec % 16 == 0 && kOffRing % 16 == 0, "alignment");
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");

// TMEM columns: [K; Q] K^T at 0 (64); U^T at 64 (64); X = [S0^T (-W) | O^T] at
// 128 (128), its first half W^T before; the state at 256 (128)
constexpr uint32_t kColGM = 0, kColU = 64, kColX = 128, kColO = 192, kColSt = 256;
// the state as the X MMA's A operand: bf16 pairs (dk elements 2k, 2k + 1 of
// lane c in column k), hi then lo (64 columns each); once X has read it, d^T and
// (d G[C-1])^T, hi and lo (pairs of tokens, 32 columns each), as the A operands
// of the last MMAs
constexpr uint32_t kColS0h = 384, kColS0l = 448;
constexpr uint32_t kColDh = 384, kColDl = 416, kColDGh = 448, kColDGl = 480;

// byte offset of element (row, k) in a 128-byte swizzled K-major tile
__device__ __forceinline__ uint32_t sw_off(int row, int k, uint32_t slice_bytes) {
  return uint32_t(k >> 6) * slice_bytes + uint32_t(row >> 3) * 1024u + uint32_t(row & 7) * 128u +
         (uint32_t(((k & 63) >> 3) ^ (row & 7)) << 4) + uint32_t(k & 7) * 2u;
}

// byte offset of the 16-byte chunk j (elements 8 j .. 8 j + 7) of a row
__device__ __forceinline__ uint32_t sw_chunk(int row, int j) {
  return uint32_t(row >> 3) * 1024u + uint32_t(row & 7) * 128u + (uint32_t(j ^ (row & 7)) << 4);
}

__device__ __forceinline__ float bf(const uint8_t* base, uint32_t off) {
  return __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(base + off));
}

// x = hi + lo with hi, lo bf16
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const float2 hf = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - hf.x, y - hf.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// 32 consecutive state values of this thread's lane (dk i0 .. i0 + 31) as hi
// and lo bf16 pairs in 16 TMEM columns each
__device__ __forceinline__ void put32_tmem(uint32_t hi_col, uint32_t lo_col, const float* x) {
  float h[16], l[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    uint32_t hh, ll;
    split2(x[2 * k], x[2 * k + 1], hh, ll);
    h[k] = __uint_as_float(hh);
    l[k] = __uint_as_float(ll);
  }
  tmem_st_16cols(hi_col, h);
  tmem_st_16cols(lo_col, l);
}

// eight consecutive values (chunk j of a 64-element slice row) as hi and lo
__device__ __forceinline__ void put8(uint8_t* hi_tile, uint8_t* lo_tile, int row, int j,
                                     const float* x) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) split2(x[2 * p], x[2 * p + 1], h[p], l[p]);
  const uint32_t off = sw_chunk(row, j);
  *reinterpret_cast<uint4*>(hi_tile + off) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4*>(lo_tile + off) = make_uint4(l[0], l[1], l[2], l[3]);
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int32_t x, int32_t y, int32_t z, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)),
      "l"(policy)
      : "memory");
}

// eight floats from a 16-byte aligned address
__device__ __forceinline__ void load8(float* x, const float* p) {
  *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(p);
  *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(p + 4);
}

// barrier of one group's 256 threads (id 1: solve, 2: state)
__device__ __forceinline__ void group_sync(uint32_t id) { named_bar_sync(id, kGroup); }

// the same, returning whether `ok` holds for every thread of the group
__device__ __forceinline__ bool group_and(uint32_t id, bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(uint32_t(ok)), "r"(id), "n"(kGroup)
      : "memory");
  return r != 0;
}

// Block (i, k), k <= i, of A or T: rows kPitch floats apart and blocks kBlk, so
// that eight rows of a 16-byte column, or the same place of two blocks, fall in
// different banks, and every offset inside a block is a constant.
__device__ __forceinline__ float* blk(float* base, int i, int k) {
  return base + (i * (i + 1) / 2 + k) * kBlk;
}

// x <- the solution of (I + A_bb) x = x for the 16 x 16 diagonal block b, column
// by column of A (right-looking: the 15 - i updates by x[i] are independent),
// four columns' rows loaded at a time
__device__ __forceinline__ void solve_unit_lower16(const float* __restrict__ A, float (&x)[16]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float4 a[16];
#pragma unroll
    for (int r = 4 * q + 1; r < 16; ++r)
      a[r] = *reinterpret_cast<const float4*>(A + r * kPitch + 4 * q);
#pragma unroll
    for (int r = 4 * q + 1; r < 16; ++r) x[r] = fmaf(-a[r].x, x[4 * q], x[r]);
#pragma unroll
    for (int r = 4 * q + 2; r < 16; ++r) x[r] = fmaf(-a[r].y, x[4 * q + 1], x[r]);
#pragma unroll
    for (int r = 4 * q + 3; r < 16; ++r) x[r] = fmaf(-a[r].z, x[4 * q + 2], x[r]);
#pragma unroll
    for (int r = 4 * q + 4; r < 16; ++r) x[r] = fmaf(-a[r].w, x[4 * q + 3], x[r]);
  }
}

// First step of T = (I + A)^{-1}: the diagonal blocks T_bb (threads 0 .. 63: a
// column each) and, on threads 64 .. 159, the products P_bk = T_bb A_bk (k < b)
// as the solutions of (I + A_bb) x = A_bk[:, col], in the place of A_bk.
__device__ __forceinline__ void invert_diagonal(float* A, float* T, int tid) {
  const int jj = tid & 15;
  float x[16];
  if (tid < 64) {
    const int b = tid >> 4;
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = r == jj ? 1.f : 0.f;
    solve_unit_lower16(blk(A, b, b), x);
    float* t = blk(T, b, b) + jj;
#pragma unroll
    for (int r = 0; r < 16; ++r) t[r * kPitch] = x[r];
  } else {
    const int task = (tid - 64) >> 4, b = task < 1 ? 1 : task < 3 ? 2 : 3;
    float* t = blk(A, b, task - b * (b - 1) / 2) + jj;
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = t[r * kPitch];
    solve_unit_lower16(blk(A, b, b), x);
#pragma unroll
    for (int r = 0; r < 16; ++r) t[r * kPitch] = x[r];
  }
}

// Then the blocks below the diagonal level by level (d = i - j = 1, 2, 3):
// T_ij = -sum_{k=j}^{i-1} P_ik T_kj, one barrier a level. A thread forms four
// outputs of one row for one block k (16 products each), and the d threads of
// an output add theirs: each level is one pass of 20 independent 16-byte loads.
// They sit in different half or quarter warps, so that the lanes served together
// read the same rows (no bank conflicts).
__device__ __forceinline__ void invert_levels(float* P, float* T, int tid) {
#pragma unroll
  for (int d = 1; d < 4; ++d) {
    const int lanes = d == 1 ? 32 : d == 2 ? 16 : 8;  // outputs of a warp
    const int sp = (tid & 31) / lanes, t = (tid >> 5) * lanes + tid % lanes;
    // task t: block (jb + d, jb), row r, columns 4 c4 .. 4 c4 + 3
    const int jb = t >> 6, ib = jb + d, r = (t >> 2) & 15, c4 = t & 3, kb = jb + sp;
    const bool on = t < (4 - d) * 64 && sp < d;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (on) {
      const float* pr = blk(P, ib, kb) + r * kPitch;
      const float* tr = blk(T, kb, jb) + 4 * c4;
#pragma unroll
      for (int k4 = 0; k4 < 4; ++k4) {
        const float4 p4 = *reinterpret_cast<const float4*>(pr + 4 * k4);
        const float pv[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float4 t4 = *reinterpret_cast<const float4*>(tr + (4 * k4 + e) * kPitch);
          acc.x = fmaf(pv[e], t4.x, acc.x);
          acc.y = fmaf(pv[e], t4.y, acc.y);
          acc.z = fmaf(pv[e], t4.z, acc.z);
          acc.w = fmaf(pv[e], t4.w, acc.w);
        }
      }
    }
#pragma unroll
    for (int o = lanes; o < 32; o <<= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
      acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
    }
    if (on && sp == 0)
      *reinterpret_cast<float4*>(blk(T, ib, jb) + r * kPitch + 4 * c4) =
          make_float4(-acc.x, -acc.y, -acc.z, -acc.w);
    group_sync(1);
  }
}

// The gates of a chunk and their decay products, by two warps (t = 0 .. 63):
// g_t = a_0 .. a_t and G[C-1][t] = a_{t+1} .. a_63 by scans, each warp
// multiplying in the other's half
__device__ __forceinline__ void decays(float* v, int t, int lane, float a, float a_other,
                                       float b) {
  float pre = a, suf = a, all = a_other;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const float x = __shfl_up_sync(0xffffffffu, pre, d);
    if (lane >= d) pre *= x;
    const float y = __shfl_down_sync(0xffffffffu, suf, d);
    if (lane + d < 32) suf *= y;
    all *= __shfl_xor_sync(0xffffffffu, all, d);
  }
  suf = __shfl_down_sync(0xffffffffu, suf, 1);  // a_{t+1} .. of this warp
  if (lane == 31) suf = 1.f;
  const float g = t >= 32 ? all * pre : pre;
  v[t] = a;
  v[64 + t] = b;
  v[128 + t] = pre;
  v[192 + t] = g;
  v[256 + t] = t < 32 ? suf * all : suf;
  if (t == kC - 1) v[320] = g;
}

// MANY: more items (request, head) than CTAs, so that a CTA works through several;
// otherwise CTA i has item i, its chunks are known from its prefix alone, and the
// walk through the items is left out (with it, one 1,000-token request takes 67.1 us
// instead of 65.7 under gated linear attention).
template <bool DELTA, bool MANY>
__global__ void __launch_bounds__(kThreads, 1)
scan_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
               const __grid_constant__ CUtensorMap tmV, const int32_t* __restrict__ prefix_offset,
               const int32_t* __restrict__ req_order, int R, int total, int Hl, const float* __restrict__ s_init,
               const float* __restrict__ alpha, const float* __restrict__ beta,
               __nv_bfloat16* __restrict__ o, float* __restrict__ s_out, int* status,
               uint64_t wait_ns, int hold_first) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                           ~uintptr_t(1023));
  float* const vec = reinterpret_cast<float*>(sm + kOffVec);  // chunk j's gates at (j % 3) kVecFloats
  float* const Am = reinterpret_cast<float*>(sm + kOffA);
  float* const Tm = reinterpret_cast<float*>(sm + kOffT);
  __nv_bfloat16* ost = reinterpret_cast<__nv_bfloat16*>(sm + kOffOut);
  uint64_t* bar_k = reinterpret_cast<uint64_t*>(sm + kOffBar);  // [2], by chunk parity
  uint64_t* bar_q = bar_k + 2;                                  // [2]
  uint64_t* bar_v = bar_k + 4;
  uint64_t* bar_g = bar_k + 5;    // [K; Q] K^T of a chunk is done
  uint64_t* bar_uw = bar_k + 6;   // U and W of a chunk are done
  uint64_t* bar_x = bar_k + 7;    // X of a chunk is done: [-W | g Q] may be replaced
  uint64_t* bar_so = bar_k + 8;   // the state and output MMAs of a chunk
  uint64_t* ready = bar_k + 9;    // the solve group is done with a chunk
  uint64_t* u_free = bar_k + 10;  // a chunk's U and X have been read
  uint64_t* drain = bar_k + 11;   // [2]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(drain + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int role = warp >> 3;             // 0: solve, 1: state
  const int tid = threadIdx.x & (kGroup - 1);  // within the group
  const int grp = tid >> 7;   // warpgroup of the group
  const int c = tid & 127;    // TMEM lane: value column c (and key column c of W)
  int4* const ring = reinterpret_cast<int4*>(sm + kOffRing);
  if (threadIdx.x == 0) {
    for (int b = 0; b < 9; ++b) mbar_init(bar_k + b, 1);
    mbar_init(ready, kGroup / 32);
    mbar_init(u_free, kGroup / 32);
    mbar_init(drain, 1);
    mbar_init(drain + 1, 1);
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  pdl_begin();
  // This CTA's items, (request, head): request by request in order of decreasing
  // length, dealt out back and forth (0 .. n-1, n-1 .. 0, ...). `walk` steps
  // through the chunks of the items that have any; one thread keeps it, in shared
  // memory (registers are short), with the next item's prefix already read.
  // R and Hl are at most 65,535, so items and the grid fit 32 bits
  const unsigned items = unsigned(R) * unsigned(Hl);
  auto item_at = [&](int u) {
    return unsigned(u) * gridDim.x + ((u & 1) ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
  };
  // the item's request and prefix ({-1, 0, 0} past the last item; an empty prefix
  // for a request the layout does not hold)
  auto read_item = [&](int u) {
    const unsigned it = item_at(u);
    if (it >= items) return make_int3(-1, 0, 0);
    const int r = MANY ? req_order[it / unsigned(Hl)] : int(it / unsigned(Hl));
    int a = -1, b = -1;
    if (r >= 0 && r < R) {
      a = prefix_offset[r];
      b = prefix_offset[r + 1];
    }
    return make_int3(r, a, b);
  };
  struct Walk {
    int4 cur;   // the chunk to hand out next
    int3 next;  // the prefix of item u
    int u;
  };
  Walk& walk = *reinterpret_cast<Walk*>(sm + kOffWalk);
  auto valid = [&](const int3& x) {
    return x.x >= 0 && x.x < R && x.y >= 0 && x.y <= x.z && x.z <= total;
  };
  auto start = [&](int u, int3 x) {  // item u's first chunk; false: it has no tokens
    if (!valid(x)) {
      flag(status, JET_ERR_DEVICE);
      return false;
    }
    const int h = int(item_at(u) % unsigned(Hl));
    walk.cur = make_int4(x.y, x.z, h, x.x * Hl + h);
    return x.y < x.z;
  };
  auto take = [&] {  // the next item that has tokens, or the empty chunk
    walk.cur = make_int4(0, 0, 0, 0);
    while (item_at(walk.u) < items) {
      const int u = walk.u;
      const int3 x = walk.next;
      walk.next = read_item(++walk.u);
      if (start(u, x)) return;
    }
  };
  auto hand_out = [&](int j) {
    ring[j & (kRing - 1)] = walk.cur;
    if (walk.cur.x + kC < walk.cur.y)
      walk.cur.x += kC;
    else if (walk.cur.x < walk.cur.y)
      take();
  };
  if (MANY && warp == 0) {
    const int3 x = read_item(lane & 1);  // the first two items at once
    const int3 x1 = make_int3(__shfl_sync(0xffffffffu, x.x, 1), __shfl_sync(0xffffffffu, x.y, 1),
                              __shfl_sync(0xffffffffu, x.z, 1));
    if (lane == 0) {
      walk.u = 1;
      walk.next = x1;
      if (!start(0, x)) take();
      for (int j = 0; j < 3; ++j) hand_out(j);
    }
    __syncwarp();
  }
  if (warp == 0) {
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  const uint32_t lane_off = uint32_t(32 * (warp & 3)) << 16;
  // chunk j of this CTA's sequence; the walk hands out chunk j + 3 during the solve of
  // chunk j, which is at most two chunks ahead of the state group
  // (without MANY: all of it from the item's prefix)
  int3 only{};
  if (!MANY) {
    only = read_item(0);
    if (!valid(only)) {
      if (threadIdx.x == 0) flag(status, JET_ERR_DEVICE);
      only.y = only.z = 0;
    }
  }
  auto chunk = [&](int j) {
    if (MANY) return ring[j & (kRing - 1)];
    return make_int4(only.y + j * kC, only.z, int(blockIdx.x % unsigned(Hl)), int(blockIdx.x));
  };
  auto has = [&](int j) {
    const int4 x = chunk(j);
    return x.x < x.y;
  };
  const uint64_t pol = policy_evict_first();

  // TMA copies of chunk j's K and Q (into the buffers of its parity) and V. The
  // first ones are issued by the solve group's thread 0, the later ones by the
  // thread 0 of the group that last read the buffer. `pend` / `par` remember the
  // barriers this thread armed (bits 0, 1: K, 2, 3: Q, 4: V) and the parity of
  // their last phase, for the wait after an abort.
  uint32_t pend = 0, par = 0;
  auto armed = [&](int bit, int phase) {
    pend |= 1u << bit;
    par = (par & ~(1u << bit)) | (uint32_t(phase & 1) << bit);
  };
  auto load = [&](const CUtensorMap* map, uint64_t* bar, uint32_t off, uint32_t slice, int j) {
    const int4 x = chunk(j);
    mbar_arrive_expect_tx(bar, 2 * 8192);
    for (int sl = 0; sl < 2; ++sl)
      tma_load_3d(sm + off + sl * slice, map, bar, sl * 64, x.z, x.x, pol);
  };
  auto load_k = [&](int j) {
    load(&tmK, bar_k + (j & 1), kOffKQ + (j & 1) * kKQBuf, kKQSlice, j);
    armed(j & 1, j >> 1);
  };
  auto load_q = [&](int j) {
    load(&tmQ, bar_q + (j & 1), kOffKQ + 8192 + (j & 1) * kKQBuf, kKQSlice, j);
    armed(2 + (j & 1), j >> 1);
  };
  auto load_v = [&](int j) {
    load(&tmV, bar_v, kOffV, kVSlice, j);
    armed(4, j);
  };
  bool ok = true;
  // g Q of chunk j as rows 64 .. 127 (the second N slice) of the MN-major
  // [-W | g Q] operand: thread c writes dk row c, each warpgroup half of the tokens
  auto write_gq = [&](int j) {
    const uint8_t* qt = sm + kOffKQ + 8192 + (j & 1) * kKQBuf;
    const float* vg = vec + (j % 3) * kVecFloats + 192;
#pragma unroll
    for (int j4 = 0; j4 < 4; ++j4) {
      const int jj = 4 * grp + j4;
      float x[8], gv[8];
      load8(gv, vg + 8 * jj);
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] = gv[e] * bf(qt, sw_off(8 * jj + e, c, kKQSlice));
      put8(sm + kOffWQh + kWQSlice, sm + kOffWQl + kWQSlice, c, jj, x);
    }
  };

  if (role == 0) {
    // ================================================================ solve
    if (tid == 0 && has(0) && !hold_first) {
      load_k(0);
      load_q(0);
      load_v(0);
      if (has(1)) {
        load_k(1);
        load_q(1);
      }
    }
    // a chunk's gates are read two chunks ahead and their products formed one
    // ahead, by the group's last two warps (token t of the chunk; 1 and 0 past
    // the prefix's end), beside the first step of the inverse
    const int gt = tid - (kGroup - kC);
    float ga = 1.f, go = 1.f, gb = 0.f;  // this token's, and a of the other warp's
    auto read_gates = [&](int j) {
      const int4 x = chunk(j);
      const int t = x.x + gt, u = x.x + (gt ^ 32);
      ga = t < x.y ? alpha[size_t(t) * Hl + x.z] : 1.f;
      gb = t < x.y ? beta[size_t(t) * Hl + x.z] : 0.f;
      go = u < x.y ? alpha[size_t(u) * Hl + x.z] : 1.f;
    };
    if (gt >= 0) {
      read_gates(0);
      decays(vec, gt, lane, ga, go, gb);
      read_gates(1);
    }
    // [K; Q] K^T of chunk j: k.k and q.k in float32 (one thread; false: its
    // operands did not come)
    auto issue_gm = [&](int j) {
      if (!mbar_wait(bar_k + (j & 1), (j >> 1) & 1, wait_ns, abort_flag) ||
          !mbar_wait(bar_q + (j & 1), (j >> 1) & 1, wait_ns, abort_flag))
        return false;
      tc_fence_after();
      const uint32_t kq = smem_u32(sm + kOffKQ + (j & 1) * kKQBuf);
#pragma unroll
      for (int st = 0; st < 8; ++st) {
        const uint32_t a = kq + (st >> 2) * kKQSlice + 32 * (st & 3);
        mma_f16(tmem + kColGM, desc_k_sw128(a), desc_k_sw128(a), idesc_bf16_f32(128, 64), st != 0);
      }
      mma_commit(bar_g);
      return true;
    };
    bool issued = true;  // this thread's loads and MMAs went out
    if (warp == 0 && has(0) && elect_one()) issued = issue_gm(0);
    __syncwarp();
    for (int j = 0; has(j); ++j) {
      const bool last = !has(j + 1);  // of the CTA's sequence
      const int odd = j & 1;
      uint8_t* const kt = sm + kOffKQ + odd * kKQBuf;  // this chunk's K (dk-slices kKQSlice apart)
      uint8_t* const mt = sm + kOffM + odd * kMBuf;    // this chunk's M o G
      float* const va = vec + (j % 3) * kVecFloats;  // this chunk's gates
      const float *vb = va + 64, *vh = va + 128, *vg = va + 192;
      bool okk = mbar_wait(bar_g, j & 1, wait_ns, abort_flag) && issued;
      ok = group_and(1, okk);  // and the gates are in
      if (!ok) break;
      tc_fence_after();
      float gr[32];
      tmem_ld_32cols(tmem + lane_off + kColGM + 32 * (1 - grp), gr);
      // ---- the solve's matrix A (k rows, lanes 0 .. 63) and M o G (q rows): the
      // first warpgroup columns 32 .. 63, the second columns 0 .. 31; the decay
      // G[rr][i] = a_{i+1} .. a_rr grows leftwards. This parity's M o G was last
      // read by the chunk before last, whose state MMAs this chunk's K (its load
      // came after them) has waited for.
      {
        const int rr = tid & 63, hf = 1 - grp;
        float av[32];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          *reinterpret_cast<float4*>(av + 4 * q) =
              *reinterpret_cast<const float4*>(va + 32 * hf + 4 * q);
        float g = hf == 0 && rr >= 32 ? vh[rr] : 1.f;
        const int top = rr - 32 * hf;  // the last column of this half up to rr
        tmem_wait_ld();
        if ((tid & 64) == 0) {
          if (DELTA) {
            // k row rr: A[rr][i] = b_rr G[rr][i] (k_rr . k_i), i < rr (what stands
            // from rr on is never read)
            g *= vb[rr];
#pragma unroll
            for (int i = 31; i >= 0; --i) {
              gr[i] *= g;
              if (i <= top) g *= av[i];
            }
            const int ib = rr >> 4;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const int kb = 2 * hf + (q >> 2);
              if (kb <= ib)
                *reinterpret_cast<float4*>(blk(Am, ib, kb) + (rr & 15) * kPitch + 4 * (q & 3)) =
                    make_float4(gr[4 * q], gr[4 * q + 1], gr[4 * q + 2], gr[4 * q + 3]);
            }
          }
        } else {
          // q row rr: (M o G)[rr][i] = (q_rr . k_i) G[rr][i], i <= rr
#pragma unroll
          for (int i = 31; i >= 0; --i) {
            gr[i] = i <= top ? gr[i] * g : 0.f;
            if (i <= top) g *= av[i];
          }
#pragma unroll
          for (int jj = 0; jj < 4; ++jj)
            put8(mt, mt + kMLo, rr, 4 * hf + jj, gr + 8 * jj);
        }
      }
      fence_proxy_async_shared();
      tc_fence_before();
      group_sync(1);
      if (DELTA) {
        // ---- T = (I + A)^{-1}, then T' = T diag(b) and T'' = T diag(b g) as
        // the hi/lo B operands (row r, 64 tokens i, K-major) of U = T' V and
        // W = T'' K, in the first N slice of the [-W | g Q] tiles, once the
        // previous chunk's X has read those
        if (tid < 64 + 6 * 16)
          invert_diagonal(Am, Tm, tid);
        else if (MANY && tid == kWalker)
          hand_out(j + 3);
        else if (gt >= 0 && !last) {
          decays(vec + (j + 1) % 3 * kVecFloats, gt, lane, ga, go, gb);
          read_gates(j + 2);
        }
        group_sync(1);
        invert_levels(Am, Tm, tid);
        okk = j == 0 || mbar_wait(bar_x, (j - 1) & 1, wait_ns, abort_flag);
        if (okk) {
          const int row = tid >> 2;
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2) {
            const int jj = 2 * (tid & 3) + h2;
            float x1[8], x2[8];
            float tv[8] = {}, bv[8], gv[8];
            if ((jj >> 1) <= (row >> 4))
              load8(tv, blk(Tm, row >> 4, jj >> 1) + (row & 15) * kPitch + 8 * (jj & 1));
            load8(bv, vb + 8 * jj);
            load8(gv, vg + 8 * jj);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              x1[e] = tv[e] * bv[e];  // T_ii is zero above the diagonal
              x2[e] = x1[e] * gv[e];
            }
            put8(sm + kOffWQh, sm + kOffWQl, row, jj, x1);
            put8(sm + kOffWQh + 8192, sm + kOffWQl + 8192, row, jj, x2);
          }
        }
        fence_proxy_async_shared();
        tc_fence_before();
        ok = group_and(1, okk);
        if (!ok) break;
        if (lane == 0) mbar_arrive(ready);
        // ---- U^T = V^T T'^T and W^T = K^T T''^T: V and K are MN-major A
        // operands (exact in bf16), T' and T'' enter as hi + lo; W^T takes the
        // first half of X, which (like U) the state group has read by then. The
        // next chunk's [K; Q] K^T follows at once.
        if (warp == 0 && elect_one()) {
          issued = mbar_wait(bar_v, j & 1, wait_ns, abort_flag) &&
                   (j == 0 || mbar_wait(u_free, (j - 1) & 1, wait_ns, abort_flag));
          if (issued) {
            tc_fence_after();
            const uint32_t idesc = idesc_bf16_f32(128, 64) | (1u << 15);
#pragma unroll
            for (int pass = 0; pass < 2; ++pass) {
              const uint32_t b = smem_u32(sm + (pass ? kOffWQl : kOffWQh));
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                mma_f16(tmem + kColU, desc_mn_sw128(smem_u32(sm + kOffV) + k * 2048, kVSlice),
                        desc_k_sw128(b + 32 * k), idesc, (pass | k) != 0);
                mma_f16(tmem + kColX, desc_mn_sw128(smem_u32(kt) + k * 2048, kKQSlice),
                        desc_k_sw128(b + 8192 + 32 * k), idesc, (pass | k) != 0);
              }
            }
            mma_commit(bar_uw);
            if (!last) issued = issue_gm(j + 1);
          }
        }
        __syncwarp();
      } else {
        // gated linear attention: U = diag(b) V straight into TMEM
        // (g Q as soon as the previous X has read its own, and the next chunk's
        // decays after this one is handed over: only U waits for d; with all of it
        // in the chain 3 x 2,000 - 4,000 tokens took 234 us instead of 225)
        okk = j == 0 || mbar_wait(bar_x, (j - 1) & 1, wait_ns, abort_flag);
        if (okk) write_gq(j);
        okk = okk && mbar_wait(bar_v, j & 1, wait_ns, abort_flag) &&
              (j == 0 || mbar_wait(u_free, (j - 1) & 1, wait_ns, abort_flag));
        if (okk) {
          tc_fence_after();
          const uint8_t* vt = sm + kOffV;
          float uv[32];
#pragma unroll
          for (int i = 0; i < 32; ++i)
            uv[i] = vb[32 * grp + i] * bf(vt, sw_off(32 * grp + i, c, kVSlice));
          tmem_st_32cols(tmem + lane_off + kColU + 32 * grp, uv);
          tmem_wait_st();
        }
        fence_proxy_async_shared();
        tc_fence_before();
        ok = group_and(1, okk);
        if (!ok) break;
        if (lane == 0) mbar_arrive(ready);
        if (gt >= 0 && !last) {
          decays(vec + (j + 1) % 3 * kVecFloats, gt, lane, ga, go, gb);
          read_gates(j + 2);
        }
        if (MANY && tid == kWalker) hand_out(j + 3);
        // neither V nor Q is read any more
        if (tid == 0 && !last) load_v(j + 1);
        if (tid == 0 && has(j + 2)) load_q(j + 2);
        __syncwarp();
        if (warp == 0 && !last && elect_one()) issued = issue_gm(j + 1);
        __syncwarp();
      }
    }
    ok = group_and(1, ok && issued);
  } else {
    // ================================================================ state
    // items without tokens: the state is the initial one (zeros without one); a warp
    // looks at 32 items at a time
    for (int u0 = 32 * (warp & 7); item_at(u0) < items; u0 += 32 * (kGroup / 32)) {
      const int3 x = read_item(u0 + lane);
      const bool empty = valid(x) && x.y == x.z;
      for (unsigned m = __ballot_sync(0xffffffffu, empty); m != 0; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const int r = __shfl_sync(0xffffffffu, x.x, src);
        const size_t head = (size_t(r) * Hl + size_t(item_at(u0 + src) % unsigned(Hl))) * kD * kD;
        for (int i = lane; i < kD * kD; i += 32) s_out[head + i] = s_init ? s_init[head + i] : 0.f;
      }
    }
    // an item's initial state, 32 of this warpgroup's 64 columns at a time: lane c
    // holds S0^T[c][.] = S0[.][c]
    auto read_init = [&](const int4& x, int i0, float (&v)[32]) {
      const float* s0 = s_init + (size_t(x.w) * kD + i0) * kD + c;
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = s_init ? s0[i * kD] : 0.f;
    };
    // the first item's: into TMEM and as the bf16 hi/lo operand of the first X
    if (has(0)) {
      for (int i0 = 64 * grp; i0 < 64 * grp + 64; i0 += 32) {
        float v[32];
        read_init(chunk(0), i0, v);
        tmem_st_32cols(tmem + lane_off + kColSt + i0, v);
        put32_tmem(tmem + lane_off + kColS0h + (i0 >> 1), tmem + lane_off + kColS0l + (i0 >> 1), v);
      }
    }
    tmem_wait_st();
    tc_fence_before();
    group_sync(2);
    const float rs = rsqrtf(float(kD));
    float ov[32];  // a chunk's outputs: value column c of this warpgroup's 32 tokens
    // chunk j's outputs from ov, through shared memory as they are stored ([token]
    // [value]): each token's 128 outputs are 256 contiguous bytes of o (the next
    // chunk's staging comes after several of this group's barriers)
    auto write_out = [&](int j) {
#pragma unroll
      for (int i = 0; i < 32; ++i) ost[(32 * grp + i) * kD + c] = __float2bfloat16_rn(ov[i] * rs);
      group_sync(2);
      const int4 x = chunk(j);
      const int n = min(kC, x.y - x.x);
      __nv_bfloat16* const od = o + (size_t(x.x + (tid >> 4)) * Hl + x.z) * kD + 8 * (tid & 15);
#pragma unroll
      for (int i = 0; i < kC * (kD / 8) / kGroup; ++i)
        if ((tid >> 4) + 16 * i < n)
          *reinterpret_cast<uint4*>(od + size_t(16 * i) * Hl * kD) =
              reinterpret_cast<const uint4*>(ost)[tid + kGroup * i];
    };
    bool pending = false;  // the previous chunk's outputs are still in ov
    for (int j = 0; has(j); ++j) {
      const int odd = j & 1;
      uint8_t* const kt = sm + kOffKQ + odd * kKQBuf;
      uint8_t* const mt = sm + kOffM + odd * kMBuf;
      bool okk = mbar_wait(ready, j & 1, wait_ns, abort_flag);
      const uint32_t scol = tmem + lane_off + kColSt + 64 * grp;
      if (DELTA) {
        if (okk) write_gq(j);  // while the tensor cores form U and W
        // -W as the first N slice: thread c writes key row c, each warpgroup half
        // of the tokens (T' and T'' have been read)
        okk = okk && mbar_wait(bar_uw, j & 1, wait_ns, abort_flag);
        tc_fence_after();
        if (okk) {
          float wv[32];
          tmem_ld_32cols(tmem + lane_off + kColX + 32 * grp, wv);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) wv[i] = -wv[i];
#pragma unroll
          for (int jj = 0; jj < 4; ++jj)
            put8(sm + kOffWQh, sm + kOffWQl, c, 4 * grp + jj, wv + 8 * jj);
        }
      }
      tmem_wait_st();  // the new state's operand, of the previous chunk
      fence_proxy_async_shared();
      tc_fence_before();
      ok = group_and(2, okk);
      if (!ok) break;
      if (DELTA && tid == 0) {  // this chunk's Q and V are no longer read
        if (has(j + 2)) load_q(j + 2);
        if (has(j + 1)) load_v(j + 1);
      }
      // ---- X = S0^T [-W | g Q] (delta rule) or O^T = S0^T (g Q) (gated linear
      // attention): three hi/lo passes; A (the state, K = dk) from TMEM, 8 packed
      // columns per K = 16 step; the B operand is MN-major (dk rows of 128 tokens)
      if (warp == 8 && elect_one()) {
        tc_fence_after();
#pragma unroll
        for (int pass = 0; pass < 3; ++pass) {
          const uint32_t a = tmem + (pass == 2 ? kColS0l : kColS0h);
          const uint32_t b = smem_u32(sm + (pass == 1 ? kOffWQl : kOffWQh));
#pragma unroll
          for (int st = 0; st < 8; ++st) {
            if (DELTA)
              mma_f16_ta(tmem + kColX, a + 8 * st, desc_mn_sw128(b + st * 2048, kWQSlice),
                         idesc_bf16_f32(128, 128) | (1u << 16), (pass | st) != 0);
            else
              mma_f16_ta(tmem + kColO, a + 8 * st, desc_mn_sw128(b + kWQSlice + st * 2048, kWQSlice),
                         idesc_bf16_f32(128, 64) | (1u << 16), (pass | st) != 0);
          }
        }
        mma_commit(bar_x);
      }
      __syncwarp();
      // while X runs: the previous chunk's outputs (delta rule), and this warpgroup's
      // 64 state columns scaled by g_{C-1} for the last MMA to accumulate onto (X
      // reads the hi/lo copy, not these)
      if (DELTA && pending) write_out(j - 1);
      {
        const float g = vec[(j % 3) * kVecFloats + 320];
        float s0[32];
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          tmem_ld_32cols(scol + 32 * hf, s0);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) s0[i] *= g;
          tmem_st_32cols(scol + 32 * hf, s0);
        }
      }
      const bool okx = mbar_wait(bar_x, j & 1, wait_ns, abort_flag);
      tc_fence_after();
      // ---- d = U + X (column c of d is row c of d^T): the first warpgroup
      // writes d^T, the second (d G[C-1])^T, as bf16 hi/lo A operands in TMEM
      // over the old state's (X has read it)
      if (okx) {
        const float* vgc = vec + (j % 3) * kVecFloats + 256;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          float dr[32];
          tmem_ld_32cols(tmem + lane_off + kColU + 32 * hf, dr);
          if (DELTA) {
            float xr[32];
            tmem_ld_32cols(tmem + lane_off + kColX + 32 * hf, xr);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) dr[i] += xr[i];
          } else {
            tmem_wait_ld();
          }
          if (grp == 1) {
#pragma unroll
            for (int i = 0; i < 32; ++i) dr[i] *= vgc[32 * hf + i];
          }
          put32_tmem(tmem + lane_off + (grp ? kColDGh : kColDh) + 16 * hf,
                     tmem + lane_off + (grp ? kColDGl : kColDl) + 16 * hf, dr);
        }
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(u_free);
      ok = group_and(2, okx);
      if (!ok) break;
      // ---- O^T += d^T (M o G)^T (three passes); state^T += (d G[C-1])^T K (two:
      // K is exact in bf16)
      if (warp == 8 && elect_one()) {
        tc_fence_after();
#pragma unroll
        for (int pass = 0; pass < 3; ++pass) {
          const uint32_t a = tmem + (pass == 2 ? kColDl : kColDh);
          const uint32_t b = smem_u32(mt + (pass == 1 ? kMLo : 0));
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_f16_ta(tmem + kColO, a + 8 * k, desc_k_sw128(b + 32 * k), idesc_bf16_f32(128, 64),
                       1u);
        }
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
          const uint32_t a = tmem + (pass == 1 ? kColDGl : kColDGh);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_f16_ta(tmem + kColSt, a + 8 * k,
                       desc_mn_sw128(smem_u32(kt) + k * 16 * 128, kKQSlice),
                       idesc_bf16_f32(128, 128) | (1u << 16), 1u);
        }
        mma_commit(bar_so);
      }
      __syncwarp();
      // gated linear attention's X is half as long and hides the scaling alone: the
      // outputs leave here (3 x 2,000 - 4,000 tokens 225 -> 213 us)
      if (!DELTA && pending) write_out(j - 1);
      ok = group_and(2, mbar_wait(bar_so, j & 1, wait_ns, abort_flag));
      if (!ok) break;
      tc_fence_after();
      // this chunk's K is no longer read: the chunk after next may land there
      if (tid == 0 && has(j + 2)) load_k(j + 2);
      // ---- the outputs (tokens 32 grp ..) into registers, and this warpgroup's 64
      // columns of the new state as the next chunk's operand
      tmem_ld_32cols(tmem + lane_off + kColO + 32 * grp, ov);
      {
        const int4 x = chunk(j);
        pending = x.x + kC < x.y;
      }
      if (pending) {
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          float s0[32];
          tmem_ld_32cols(scol + 32 * hf, s0);
          tmem_wait_ld();
          // packed columns 32 grp + 16 hf ..
          put32_tmem(tmem + lane_off + kColS0h + 32 * grp + 16 * hf,
                     tmem + lane_off + kColS0l + 32 * grp + 16 * hf, s0);
        }
      } else {
        // an item's last chunk: outputs and state leave, and the next item's initial
        // state takes the state's place
        tmem_wait_ld();
        write_out(j);
        const int4 x = chunk(j), nx = chunk(j + 1);
#pragma unroll 1
        for (int hf = 0; hf < 2; ++hf) {
          float s0[32];
          tmem_ld_32cols(scol + 32 * hf, s0);
          tmem_wait_ld();
          float* const so = s_out + (size_t(x.w) * kD + 64 * grp + 32 * hf) * kD + c;
#pragma unroll
          for (int i = 0; i < 32; ++i) so[i * kD] = s0[i];
          if (nx.x < nx.y) {
            read_init(nx, 64 * grp + 32 * hf, s0);
            tmem_st_32cols(scol + 32 * hf, s0);
            put32_tmem(tmem + lane_off + kColS0h + 32 * grp + 16 * hf,
                       tmem + lane_off + kColS0l + 32 * grp + 16 * hf, s0);
          }
        }
      }
    }
  }
  if (!ok) {
    // a wait ran out: let the copies and tensor-core work already issued
    // finish before the CTA frees its TMEM and ends
    *abort_flag = 1;
    if (tid == 0) {
      flag(status, JET_ERR_TIMEOUT);
      for (int b = 0; b < 5; ++b)
        if (pend & (1u << b)) mbar_wait(bar_k + b, (par >> b) & 1u, kDrainNs, nullptr);
    }
    __syncwarp();
    if ((warp & 7) == 0 && elect_one()) {
      mma_commit(drain + role);
      mbar_wait(drain + role, 0, kDrainNs, nullptr);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// [tokens, Hl, 128] bf16: boxes of 64 elements x 1 head x 64 tokens, 128-byte swizzle
bool encode_tokens(CUtensorMap* map, const void* base, int tokens, int Hl) {
  auto fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {cuuint64_t(kD), cuuint64_t(Hl), cuuint64_t(tokens)};
  const cuuint64_t strides[2] = {cuuint64_t(kD) * 2, cuuint64_t(Hl) * kD * 2};
  const cuuint32_t box[3] = {64, 1, cuuint32_t(kC)};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool scan_tc_supported(const jet_dims& d) {
  return d.dtype == JET_DTYPE_BF16 && d.dk == kD && d.dv == kD;
}

cudaError_t launch_scan_tc(const jet_layout& lay, const jet_dims& d, int rule,
                           const float* s_init, const void* q, const void* k, const void* v,
                           const float* alpha, const float* beta, void* o, float* s_out,
                           int* status, cudaStream_t st) {
  const jet_sizes& n = lay.n;
  CUtensorMap tmQ, tmK, tmV;
  if (!encode_tokens(&tmQ, q, n.total_prefix, d.Hl) ||
      !encode_tokens(&tmK, k, n.total_prefix, d.Hl) ||
      !encode_tokens(&tmV, v, n.total_prefix, d.Hl))
    return cudaErrorInvalidValue;
  const long long items = (long long)n.R * d.Hl;
  const int sms = std::max(1, sm_count());  // one CTA per SM
  const bool gla = rule == JET_RECUR_GLA, many = items > sms;
  auto kern = gla ? (many ? scan_tc_kernel<false, true> : scan_tc_kernel<false, false>)
                  : (many ? scan_tc_kernel<true, true> : scan_tc_kernel<true, false>);
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemBytes));
  if (e != cudaSuccess) return e;
  const unsigned grid = unsigned(many ? sms : items);
  return launch_pdl(kern, dim3(grid), dim3(kThreads), kSmemBytes, st, tmQ, tmK, tmV,
                    lay.prefix_offset, lay.req_order, n.R, n.total_prefix, d.Hl, s_init, alpha,
                    beta, static_cast<__nv_bfloat16*>(o), s_out, status, wait_budget_ns(),
                    test_stall());
}

}  // namespace jet
