// Per-candidate fork of a linear-attention recurrent state (Sec. 4.1).
//
// The paper keeps one stored prefix state and restores it before each
// candidate, evaluating candidates one after another. Here one CTA per
// (32-column slice, head, request) reads the prefix state slice once into
// registers and the request's fed tokens once into shared memory; every
// candidate then starts from an unmodified register copy of the slice,
// applies its fed tokens and writes its own final state, so the state
// writes of one candidate overlap the arithmetic of the next. Each fed token
// applies the gated delta rule
//   S <- alpha (S - beta k (k^T S)) + beta k v^T,   o = S^T q / sqrt(dk)
// (the paper does not state its recurrence; this is the reading used).
// The update is column-separable: column j of S needs only k, v_j and the
// column's own u_j = k^T S[:, j], so a CTA owns a 32-column slice of one
// head. The kernel is bound by the writes of the forked states. The plain
// gated linear-attention variant S <- alpha S + beta k v^T is the same update
// with u = 0 (the DELTA = false instantiation skips that reduction).
#include "jet_device.cuh"
#include "jet_internal.h"

namespace jet {
namespace {

constexpr int kDK = 128;        // key dimension handled (rows of S)
constexpr int kCols = 32;       // value columns per CTA
constexpr int kThreads = 128;   // 4 warps x 32 rows
constexpr int kWin = 16;        // fed tokens staged in shared memory at a time
constexpr int kMeta = 64;       // candidates whose lengths are staged at a time

__device__ __forceinline__ float4 f4_fma(float a, float4 x, float4 y) {
  return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}

// Reduce a per-thread float4 over the 128 rows of the slice; every thread
// receives the 4 column sums of its column quad. `red` holds 4 x 32 floats.
__device__ __forceinline__ float4 rows_sum(float4 v, float* red, int warp, int lane) {
#pragma unroll
  for (int o = 8; o <= 16; o <<= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    v.z += __shfl_xor_sync(0xffffffffu, v.z, o);
    v.w += __shfl_xor_sync(0xffffffffu, v.w, o);
  }
  const int jq = lane & 7;
  if (lane < 8) reinterpret_cast<float4*>(red)[warp * 8 + jq] = v;
  __syncthreads();
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    const float4 t = reinterpret_cast<const float4*>(red)[w * 8 + jq];
    s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
  }
  __syncthreads();
  return s;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// Stage fed tokens [w0, w0 + nt) (nt <= kWin) into shared memory as they are
// stored: their k and q rows, this slice's v columns and the gates. The
// copies are asynchronous and all in flight at once, so a window costs one
// memory latency and no registers; the caller synchronises the block.
template <typename T>
__device__ __forceinline__ void stage_window(const T* __restrict__ q, const T* __restrict__ k,
                                             const T* __restrict__ v,
                                             const float* __restrict__ alpha,
                                             const float* __restrict__ beta, int Hl, int dv,
                                             int h, int j0, int w0, int nt, int tid,
                                             T (*wk)[kDK], T (*wq)[kDK], T (*wv)[kCols],
                                             float* wa, float* wb) {
  constexpr int VE = 16 / int(sizeof(T));  // elements per 16-byte piece
  constexpr int KP = kDK / VE;             // pieces of a k (or q) row
  constexpr int VP = kCols / VE;           // pieces of a v slice row
  for (int e = tid; e < nt * KP; e += kThreads) {
    const int tok = e / KP, pc = e % KP;
    const size_t src = (size_t(w0 + tok) * Hl + h) * kDK + pc * VE;
    cp_async16(&wk[tok][pc * VE], k + src);
    cp_async16(&wq[tok][pc * VE], q + src);
  }
  for (int e = tid; e < nt * VP; e += kThreads) {
    const int tok = e / VP, pc = e % VP;
    cp_async16(&wv[tok][pc * VE], v + (size_t(w0 + tok) * Hl + h) * dv + j0 + pc * VE);
  }
  if (tid < nt) {
    cp_async4(&wa[tid], alpha + size_t(w0 + tid) * Hl + h);
    cp_async4(&wb[tid], beta + size_t(w0 + tid) * Hl + h);
  }
  cp_async_wait_all();
}

__device__ __forceinline__ int wt_of(int f, int w0) { return f - w0; }

// One token of the recurrence on this thread's part of the slice (rows
// 32 w + rg + 4 ii, columns 4 jq .. + 3), token wt of the staged window:
// S = alpha S + beta k (v - alpha u), u = k^T S (u = 0 for gated linear
// attention). Returns the slice's output columns o = S^T q (unscaled), the
// same in every thread of a column quad.
template <typename T, bool DELTA>
__device__ __forceinline__ float4 token_step(float4 (&S)[8], int wt, const T (*wk)[kDK],
                                             const T (*wq)[kDK], const T (*wv)[kCols],
                                             const float* wa, const float* wb, float* red,
                                             int warp, int lane) {
  const int rg = lane >> 3, jq = lane & 7;
  float kk[8], qq[8];
#pragma unroll
  for (int ii = 0; ii < 8; ++ii) {
    const int i = 32 * warp + rg + 4 * ii;
    kk[ii] = to_f32(wk[wt][i]);
    qq[ii] = to_f32(wq[wt][i]);
  }
  const float a = wa[wt], b = wb[wt];
  const float4 vv = make_float4(to_f32(wv[wt][4 * jq]), to_f32(wv[wt][4 * jq + 1]),
                                to_f32(wv[wt][4 * jq + 2]), to_f32(wv[wt][4 * jq + 3]));
  // u = k^T S for this column quad (the delta rule's erase term)
  float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
  if (DELTA) {
#pragma unroll
    for (int ii = 0; ii < 8; ++ii) u = f4_fma(kk[ii], S[ii], u);
    u = rows_sum(u, red, warp, lane);
  }
  const float4 w = make_float4(b * (vv.x - a * u.x), b * (vv.y - a * u.y), b * (vv.z - a * u.z),
                               b * (vv.w - a * u.w));
  float4 op = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int ii = 0; ii < 8; ++ii) {
    float4 s = S[ii];
    s = make_float4(fmaf(kk[ii], w.x, a * s.x), fmaf(kk[ii], w.y, a * s.y),
                    fmaf(kk[ii], w.z, a * s.z), fmaf(kk[ii], w.w, a * s.w));
    S[ii] = s;
    op = f4_fma(qq[ii], s, op);
  }
  return rows_sum(op, red, warp, lane);
}

// grid (dv / 32, Hl, R); thread (warp w, lane = 8 * rg + jq) owns rows
// 32 w + rg + 4 ii (ii < 8) and columns j0 + 4 jq .. + 3 of the slice.
// q_rows (optional, [N, Hl, dk]): every row's q; the request's shared row then
// reads the prefix state, o = S_r^T q / sqrt(dk), and o holds all N rows
// (fed token f at row f + r + 1) instead of the fed tokens alone.
// bf16: 72 registers and 28 KB of shared memory, so that seven CTAs share an
// SM (a (32 requests x 16 heads x 4 slices) grid then fills 1.93 waves of
// 1,064 CTAs instead of 2.25 waves of 912)
template <typename T, bool DELTA>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 2 ? 7 : 3)
fork_kernel(const int32_t* __restrict__ cand_offset, const int32_t* __restrict__ cand_row_offset,
            const int32_t* __restrict__ tgt_offset, const int32_t* __restrict__ row_offset,
            int R, int C, int F, int Hl, int dv, const float* __restrict__ s_prefix,
            const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
            const float* __restrict__ alpha, const float* __restrict__ beta,
            const T* __restrict__ q_rows, T* __restrict__ o, float* __restrict__ s_fork,
            int* status) {
  pdl_begin();
  __shared__ __align__(16) float red[4 * kCols];
  // a window of the request's fed tokens as stored: k, q (all rows), v (this
  // slice), gates
  __shared__ __align__(16) T wk[kWin][kDK];
  __shared__ __align__(16) T wq[kWin][kDK];
  __shared__ __align__(16) T wv[kWin][kCols];
  __shared__ __align__(16) float wa[kWin], wb[kWin];
  // the (length, first fed token) of up to kMeta candidates at a time
  __shared__ int cm[kMeta], cf[kMeta];
  // the prefix state slice, each thread's own 8 float4 at [ii][tid]
  __shared__ __align__(16) float4 ssp[8 * kThreads];
  __shared__ float qsh[kDK];  // the shared row's q (with q_rows)
  const int r = blockIdx.z, h = blockIdx.y, j0 = blockIdx.x * kCols;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rg = lane >> 3, jq = lane & 7;
  const int col = j0 + 4 * jq;
  if (r >= R) return;
  const int c0 = cand_offset[r], c1 = cand_offset[r + 1];
  const int f_begin = row_offset[r] - r;                   // the request's first fed token
  const int f_end = f_begin + row_offset[r + 1] - row_offset[r] - 1;
  if (c0 < 0 || c1 < c0 || c1 > C || f_begin < 0 || f_end < f_begin || f_end > F) {
    if (tid == 0) flag(status, JET_ERR_DEVICE);
    return;
  }

  // the prefix state slice (read once, kept in shared memory for every
  // candidate) and the first window of fed tokens load at once
  const float rs = rsqrtf(float(kDK));
  {
    float4 sp[8];
    const size_t head = (size_t(r) * Hl + h) * kDK;
    if (q_rows && tid < kDK)
      qsh[tid] = to_f32(q_rows[(size_t(row_offset[r]) * Hl + h) * kDK + tid]);
#pragma unroll
    for (int ii = 0; ii < 8; ++ii) {
      const int i = 32 * warp + rg + 4 * ii;
      sp[ii] = *reinterpret_cast<const float4*>(s_prefix + (head + i) * dv + col);
    }
#pragma unroll
    for (int ii = 0; ii < 8; ++ii) ssp[ii * kThreads + tid] = sp[ii];
    if (q_rows) {
      // the shared row: o = S_r^T q / sqrt(dk), from the prefix state itself
      __syncthreads();  // qsh is in
      float4 op = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int ii = 0; ii < 8; ++ii) op = f4_fma(qsh[32 * warp + rg + 4 * ii], sp[ii], op);
      op = rows_sum(op, red, warp, lane);
      if (warp == 0 && rg == 0) {
        T* dst = o + (size_t(row_offset[r]) * Hl + h) * dv + col;
        dst[0] = from_f32<T>(op.x * rs);
        dst[1] = from_f32<T>(op.y * rs);
        dst[2] = from_f32<T>(op.z * rs);
        dst[3] = from_f32<T>(op.w * rs);
      }
    }
  }
  // with q_rows, fed token f is written at row f + r + 1
  const size_t o_shift = q_rows ? size_t(r) + 1 : 0;
  int w0 = f_begin, w1 = min(f_begin + kWin, f_end);  // fed tokens [w0, w1) are staged
  if (w1 > w0)
    stage_window(q, k, v, alpha, beta, Hl, dv, h, j0, w0, w1 - w0, tid, wk, wq, wv, wa, wb);

  for (int cb = c0; cb < c1; cb += kMeta) {
    const int nb = min(kMeta, c1 - cb);
    __syncthreads();  // the previous batch's lengths are no longer read
    for (int e = tid; e < nb; e += kThreads) {
      cm[e] = tgt_offset[cb + e + 1] - tgt_offset[cb + e];
      cf[e] = cand_row_offset[cb + e] - r - 1;  // fed-token index of y_{c,1}
    }
    __syncthreads();
    for (int e = 0; e < nb; ++e) {
      const int c = cb + e;
      const int m = cm[e], f0 = cf[e];
      if (m < 1 || f0 < f_begin || f0 + m - 1 > f_end) {
        if (tid == 0) flag(status, JET_ERR_DEVICE);
        continue;
      }
      float4 S[8];
#pragma unroll
      for (int ii = 0; ii < 8; ++ii) S[ii] = ssp[ii * kThreads + tid];  // the prefix state
      for (int t = 0; t < m - 1; ++t) {
        const int f = f0 + t;
        if (f < w0 || f >= w1) {
          // stage the window of fed tokens starting at f
          __syncthreads();
          w0 = f;
          w1 = min(f + kWin, f_end);
          stage_window(q, k, v, alpha, beta, Hl, dv, h, j0, w0, w1 - w0, tid, wk, wq, wv, wa, wb);
          __syncthreads();
        }
        const float4 op = token_step<T, DELTA>(S, wt_of(f, w0), wk, wq, wv, wa, wb, red, warp,
                                               lane);
        if (warp == 0 && rg == 0) {
          T* dst = o + ((size_t(f) + o_shift) * Hl + h) * dv + col;
          dst[0] = from_f32<T>(op.x * rs);
          dst[1] = from_f32<T>(op.y * rs);
          dst[2] = from_f32<T>(op.z * rs);
          dst[3] = from_f32<T>(op.w * rs);
        }
      }
      if (s_fork) {
        // streaming stores: the forked states are not read again in the step,
        // so they should not displace its working set in L2 (3 us less here)
        const size_t fhead = (size_t(c) * Hl + h) * kDK;
#pragma unroll
        for (int ii = 0; ii < 8; ++ii) {
          const int i = 32 * warp + rg + 4 * ii;
          __stcs(reinterpret_cast<float4*>(s_fork + (fhead + i) * dv + col), S[ii]);
        }
      }
    }
  }
}

// The fork's outputs alone (no forked state written: a decoder stack's linear
// layers, or a step that does not keep the states), bf16, for candidates of at
// most kRowTok fed tokens. With no state to write, the prefix state is only
// read through products: with g_t = a_1 ... a_t and G(i, t) = a_{i+1} ... a_t
// over a candidate's tokens,
//   u_t = S_{t-1}^T k_t = g_{t-1} S0^T k_t + sum_{i<t} G(i, t-1) (k_i . k_t) w_i
//   w_t = b_t (v_t - a_t u_t)              (u = 0 for gated linear attention)
//   o_t = g_t S0^T q_t + sum_{i<=t} G(i, t) (k_i . q_t) w_i
// so one pass over S0 serves the k and q of kRowTok tokens at a time (any
// number of whole candidates), and what is left is a scalar recurrence per
// column. Stepping a state per candidate instead costs two block-wide
// reductions and four barriers a token, one token after another (48 us for 355
// rows of 32 requests x 16 heads, against 5 us of HBM time for the 33.5 MB of
// prefix states); the products on the CUDA cores took 44 us, bound by
// instruction issue and shared-memory latency. Here they run as warp-level MMAs
// (a 16-column tile of S0 per warp: too small a tile for a TMEM accumulator to
// pay): S0 enters as the exact sum of three bf16 numbers, k and q are bf16, so
// every product is exact and the sums are float32: 23 us for those rows (two
// CTAs an SM, 512 CTAs: two rounds of about 10 us, bound by their chains of
// loads), the four-layer stack around it 713 -> 646 us.
// A CTA owns 128 value columns of one head of one request. Infinite inputs
// give non-finite outputs, where the stepped form may give an infinity instead
// of a NaN.
constexpr int kRowTok = 16;         // fed tokens of a batch
constexpr int kRowCols = 128;       // value columns per CTA
constexpr int kRowThreads = 256;
constexpr int kXW = kDK / 2 + 4;    // row stride of the staged k and q (32-bit words)
constexpr int kUW = kRowCols + 8;   // row stride of the products (floats)

struct RowSmem {
  uint32_t xk[kRowTok][kXW];                // bf16 pairs
  uint32_t xq[kRowTok + 8][kXW];            // row kRowTok: the shared row's q, then zeros
  float up[2 * kRowTok + 1][kUW];           // S0^T k, S0^T q, S0^T (the shared row's q)
  float w[kRowTok][kRowCols];
  __nv_bfloat16 xv[kRowTok][kRowCols];
  float kk[kRowTok][kRowTok + 1], kq[kRowTok][kRowTok + 1];  // [t][i]
  float a[kRowTok], b[kRowTok];
  int tok[kRowTok], first[kRowTok];  // fed token of a slot; its candidate's first slot
  int count, next;                   // tokens of the batch; the next batch's candidate
};

// D += A B: A 16 x 16 (row-major fragments), B 16 x 8, bf16 in, float32 out
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                          uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// the upper halves of two float32 as a bf16 pair (x in the low half)
__device__ __forceinline__ uint32_t upper_pair(float x, float y) {
  return __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
}

// what is left of x below its upper half (exact; 0 for an infinity)
__device__ __forceinline__ float below_upper(float x) {
  const float hi = __uint_as_float(__float_as_uint(x) & 0xffff0000u);
  return x == hi ? 0.f : x - hi;
}

template <bool DELTA>
__global__ void __launch_bounds__(kRowThreads, 2)
fork_rows_kernel(const int32_t* __restrict__ cand_offset,
                 const int32_t* __restrict__ cand_row_offset,
                 const int32_t* __restrict__ tgt_offset, const int32_t* __restrict__ row_offset,
                 int R, int C, int F, int Hl, int dv, const float* __restrict__ s_prefix,
                 const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k,
                 const __nv_bfloat16* __restrict__ v, const float* __restrict__ alpha,
                 const float* __restrict__ beta, const __nv_bfloat16* __restrict__ q_rows,
                 __nv_bfloat16* __restrict__ o, int* status) {
  pdl_begin();
  extern __shared__ __align__(16) uint8_t row_smem[];
  RowSmem& sm = *reinterpret_cast<RowSmem*>(row_smem);
  const int r = blockIdx.z, h = blockIdx.y, j0 = blockIdx.x * kRowCols;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g4 = lane >> 2, t4 = lane & 3;
  if (r >= R) return;
  const int c0 = cand_offset[r], c1 = cand_offset[r + 1];
  const int n0 = row_offset[r];
  const int f_begin = n0 - r;  // the request's first fed token
  const int f_end = f_begin + row_offset[r + 1] - n0 - 1;
  if (c0 < 0 || c1 < c0 || c1 > C || f_begin < 0 || f_end < f_begin || f_end > F) {
    if (tid == 0) flag(status, JET_ERR_DEVICE);
    return;
  }
  // this warp's 16 columns of the prefix state in the order of the MMA's A
  // fragments, float32: A rows g4 and g4 + 8 are columns 2 g4 and 2 g4 + 1 (one
  // 8-byte load, 64 contiguous bytes per row of S0), A columns the rows of S0.
  // The layout reads above go first: the staging below waits on them, not on S0.
  float2 S[8][4];
  {
    const float* sp = s_prefix + (size_t(r) * Hl + h) * kDK * size_t(dv) + j0 + 16 * warp + 2 * g4;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int kr = 16 * ks + 2 * t4 + (e & 1) + 4 * (e & 2);
        S[ks][e] = *reinterpret_cast<const float2*>(sp + size_t(kr) * dv);
      }
  }
  const float rs = rsqrtf(float(kDK));
  // with q_rows, fed token f is written at row f + r + 1
  const size_t o_shift = q_rows ? size_t(r) + 1 : 0;
  bool shared_row = q_rows != nullptr;
  for (int c = c0; c < c1 || shared_row;) {
    // ---- the batch: whole candidates from c on, at most kRowTok tokens
    if (warp == 0) {
      const int cc = c + lane;
      int cnt = 0, f0 = 0;
      if (cc < c1) {
        cnt = tgt_offset[cc + 1] - tgt_offset[cc] - 1;
        f0 = cand_row_offset[cc] - r - 1;  // fed-token index of y_{c,1}
        if (cnt < 0 || cnt > kRowTok || f0 < f_begin || f0 + cnt > f_end) {
          flag(status, JET_ERR_DEVICE);
          cnt = 0;
        }
      }
      int inc = cnt;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += y;
      }
      const unsigned in = __ballot_sync(0xffffffffu, cc < c1 && inc <= kRowTok);
      if (in & (1u << lane)) {
        for (int i = 0; i < cnt; ++i) {
          sm.tok[inc - cnt + i] = f0 + i;
          sm.first[inc - cnt + i] = inc - cnt;
        }
      }
      const int taken = __popc(in);  // the inclusive sums grow: a prefix of the lanes
      const int total = __shfl_sync(0xffffffffu, inc, taken > 0 ? taken - 1 : 0);
      if (lane == 0) {
        sm.count = taken > 0 ? total : 0;
        sm.next = c + taken;
      }
    }
    __syncthreads();
    const int nt = sm.count;
    c = sm.next;
    // ---- stage k, q, this slice's v and the gates: one 16-byte piece of each
    // per thread (16 tokens x 16 pieces); rows past the batch's are zeros, so
    // that no stale value enters the MMAs
    {
      const int s = tid >> 4, pc = tid & 15;
      uint4 pk = make_uint4(0, 0, 0, 0), pq = pk, pv = pk, pr = pk;
      float ga = 0.f, gb = 0.f;
      if (s < nt) {
        const size_t row = size_t(sm.tok[s]) * Hl + h;
        pk = *reinterpret_cast<const uint4*>(k + row * kDK + 8 * pc);
        pq = *reinterpret_cast<const uint4*>(q + row * kDK + 8 * pc);
        pv = *reinterpret_cast<const uint4*>(v + row * dv + j0 + 8 * pc);
        if (pc == 0) {
          ga = alpha[row];
          gb = beta[row];
        }
      }
      if (shared_row && s == 0)
        pr = *reinterpret_cast<const uint4*>(q_rows + (size_t(n0) * Hl + h) * kDK + 8 * pc);
      *reinterpret_cast<uint4*>(&sm.xk[s][4 * pc]) = pk;
      *reinterpret_cast<uint4*>(&sm.xq[s][4 * pc]) = pq;
      *reinterpret_cast<uint4*>(&sm.xv[s][8 * pc]) = pv;
      if (s < 8) *reinterpret_cast<uint4*>(&sm.xq[kRowTok + s][4 * pc]) = pr;
      if (pc == 0) {
        sm.a[s] = ga;
        sm.b[s] = gb;
      }
    }
    __syncthreads();
    // ---- S0^T k and S0^T q: this warp's 16 columns x (two tiles of 8 tokens of
    // each, and the shared row's)
    {
      float acc[5][4];
#pragma unroll
      for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        uint32_t bf[5][2];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
          const uint32_t* x = i < 2 ? sm.xk[8 * i + g4] : sm.xq[8 * (i - 2) + g4];
          bf[i][0] = x[8 * ks + t4];
          bf[i][1] = x[8 * ks + t4 + 4];
        }
        float2 rest[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) rest[e] = S[ks][e];
        // S0 = the sum of its upper 8, middle 8 and last 8 significand bits
#pragma unroll
        for (int p = 0; p < 3; ++p) {
          const uint32_t af[4] = {upper_pair(rest[0].x, rest[1].x), upper_pair(rest[0].y, rest[1].y),
                                  upper_pair(rest[2].x, rest[3].x), upper_pair(rest[2].y, rest[3].y)};
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            const bool live = i == 4 ? shared_row : (i & 1) ? nt > 8 : nt > 0;
            if (live && (DELTA || i >= 2)) mma_16816(acc[i], af, bf[i][0], bf[i][1]);
          }
          if (p < 2) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              rest[e] = make_float2(below_upper(rest[e].x), below_upper(rest[e].y));
          }
        }
      }
      // acc[i]: columns 2 g4 (0, 1) and 2 g4 + 1 (2, 3) of the warp, tokens 2 t4
      // and 2 t4 + 1 of the tile
      const int col = 16 * warp + 2 * g4;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int u = 8 * i + 2 * t4;
        *reinterpret_cast<float2*>(&sm.up[u][col]) = make_float2(acc[i][0], acc[i][2]);
        *reinterpret_cast<float2*>(&sm.up[u + 1][col]) = make_float2(acc[i][1], acc[i][3]);
      }
      if (t4 == 0)
        *reinterpret_cast<float2*>(&sm.up[2 * kRowTok][col]) = make_float2(acc[4][0], acc[4][2]);
    }
    // ---- k_i . k_t (warp 0) and k_i . q_t (warp 1) of all the batch's tokens
    if (warp < 2 && (DELTA || warp == 1)) {
      const uint32_t(*xa)[kXW] = warp == 0 ? sm.xk : sm.xq;
      float acc[2][4];
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[0][e] = acc[1][e] = 0.f;
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        const int x = 8 * ks + t4;
        const uint32_t af[4] = {xa[g4][x], xa[g4 + 8][x], xa[g4][x + 4], xa[g4 + 8][x + 4]};
        mma_16816(acc[0], af, sm.xk[g4][x], sm.xk[g4][x + 4]);
        mma_16816(acc[1], af, sm.xk[g4 + 8][x], sm.xk[g4 + 8][x + 4]);
      }
      float(*dst)[kRowTok + 1] = warp == 0 ? sm.kk : sm.kq;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        dst[g4][8 * i + 2 * t4] = acc[i][0];
        dst[g4][8 * i + 2 * t4 + 1] = acc[i][1];
        dst[g4 + 8][8 * i + 2 * t4] = acc[i][2];
        dst[g4 + 8][8 * i + 2 * t4 + 1] = acc[i][3];
      }
    }
    __syncthreads();
    // ---- the recurrence of this thread's column: the block's halves take the
    // batch's candidates in turn
    const int col = tid & (kRowCols - 1), half = tid >> 7;
    int turn = 0;
    for (int s0 = 0; s0 < nt;) {
      int s1 = s0 + 1;
      while (s1 < nt && sm.first[s1] == s0) ++s1;
      if ((turn++ & 1) == half) {
        for (int t = s0; t < s1; ++t) {
          const float a = sm.a[t];
          float u = 0.f;
          if (DELTA) {
            float g = 1.f;
            for (int i = t - 1; i >= s0; --i) {
              u = fmaf(g * sm.kk[t][i], sm.w[i][col], u);
              g *= sm.a[i];
            }
            u = fmaf(g, sm.up[t][col], u);
          }
          const float w = sm.b[t] * (__bfloat162float(sm.xv[t][col]) - a * u);
          float acc = sm.kq[t][t] * w, g = a;
          for (int i = t - 1; i >= s0; --i) {
            acc = fmaf(g * sm.kq[t][i], sm.w[i][col], acc);
            g *= sm.a[i];
          }
          acc = fmaf(g, sm.up[kRowTok + t][col], acc);
          sm.w[t][col] = w;  // read by this thread alone
          o[((size_t(sm.tok[t]) + o_shift) * Hl + h) * dv + j0 + col] =
              __float2bfloat16_rn(acc * rs);
        }
      }
      s0 = s1;
    }
    if (shared_row && half == 1)
      o[(size_t(n0) * Hl + h) * dv + j0 + col] =
          __float2bfloat16_rn(sm.up[2 * kRowTok][col] * rs);
    shared_row = false;
    __syncthreads();  // the next batch refills the staging buffers
  }
}

}  // namespace

namespace {

template <bool DELTA>
cudaError_t launch_rows(const jet_layout& lay, const jet_dims& d, const float* s_prefix,
                        const void* q, const void* k, const void* v, const float* alpha,
                        const float* beta, const void* q_rows, void* o, int* status,
                        cudaStream_t st) {
  const jet_sizes& n = lay.n;
  auto kern = fork_rows_kernel<DELTA>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             int(sizeof(RowSmem)));
  if (e != cudaSuccess) return e;
  dim3 grid(unsigned(d.dv / kRowCols), unsigned(d.Hl), unsigned(n.R));
  return launch_pdl(kern, grid, dim3(kRowThreads), sizeof(RowSmem), st, lay.cand_offset,
                    lay.cand_row_offset, lay.tgt_offset, lay.row_offset, n.R, n.C, n.N - n.R, d.Hl,
                    d.dv, s_prefix, static_cast<const __nv_bfloat16*>(q),
                    static_cast<const __nv_bfloat16*>(k), static_cast<const __nv_bfloat16*>(v),
                    alpha, beta, static_cast<const __nv_bfloat16*>(q_rows),
                    static_cast<__nv_bfloat16*>(o), status);
}

template <bool DELTA>
cudaError_t launch_rule(const jet_layout& lay, const jet_dims& d, const float* s_prefix,
                        const void* q, const void* k, const void* v, const float* alpha,
                        const float* beta, const void* q_rows, void* o, float* s_fork,
                        int* status, cudaStream_t st) {
  const jet_sizes& n = lay.n;
  dim3 grid(unsigned(d.dv / kCols), unsigned(d.Hl), unsigned(n.R));
  const int F = n.N - n.R;
  // No states to write: the prefix state is read once for 16 fed tokens at a
  // time (23 us against 48 at 355 rows of 32 requests x 16 heads), as long as no
  // candidate is longer than such a batch, the value width fills its columns, and
  // there are tokens to share the read. With few fed tokens a request stepping is
  // faster: its CTAs read S0 in quarters, seven an SM (16 heads; 64 requests, one token
  // a request 17.3 us against 24.5 by products, 1.9 22.4 and 26.1, 3.0 30.4 and 27.0;
  // 256 requests, 2.1 tokens 87 and 107, 3.0 110 and 110; 32 requests of 2.4 tokens,
  // some 15 long, 21.5 and 16.4). So it is with up to five tokens and few CTAs (three
  // linear layers and a full one of D 4,096, one request of four tokens x 4 heads, 16
  // CTAs: 358 us against 366 by products; two requests, 32 CTAs: 362 and 367; 16 heads,
  // 64 CTAs: 394 and 383), and with candidates of more than 12 while it leaves SMs
  // unfilled, since the products' recurrence goes with the square of a candidate (8
  // requests x 4 heads, up to 13 a candidate, 128 CTAs: 17.3 us and 21.2; 256 CTAs 21.2
  // and 22.1, 512 25.5 and 23.2; of 11 a candidate 128 CTAs 16.3 and 16.4).
  const long long steppers = (long long)n.R * d.Hl * (d.dv / kCols);
  const bool step_states = 10LL * F <= 23LL * n.R || (F <= 5LL * n.R && steppers <= 32) ||
                          (n.max_len - 1 > 12 && steppers <= 256);
  if (!s_fork && d.dtype == JET_DTYPE_BF16 && n.max_len - 1 <= kRowTok && d.dv % kRowCols == 0 &&
      !step_states)
    return launch_rows<DELTA>(lay, d, s_prefix, q, k, v, alpha, beta, q_rows, o, status, st);
  if (d.dtype == JET_DTYPE_F32) {
    return launch_pdl(fork_kernel<float, DELTA>, grid, dim3(kThreads), 0, st, lay.cand_offset,
                      lay.cand_row_offset, lay.tgt_offset, lay.row_offset, n.R, n.C, F, d.Hl,
                      d.dv, s_prefix, static_cast<const float*>(q), static_cast<const float*>(k),
                      static_cast<const float*>(v), alpha, beta,
                      static_cast<const float*>(q_rows), static_cast<float*>(o), s_fork, status);
  }
  return launch_pdl(fork_kernel<__nv_bfloat16, DELTA>, grid, dim3(kThreads), 0, st,
                    lay.cand_offset, lay.cand_row_offset, lay.tgt_offset, lay.row_offset, n.R,
                    n.C, F, d.Hl, d.dv, s_prefix, static_cast<const __nv_bfloat16*>(q),
                    static_cast<const __nv_bfloat16*>(k), static_cast<const __nv_bfloat16*>(v),
                    alpha, beta, static_cast<const __nv_bfloat16*>(q_rows),
                    static_cast<__nv_bfloat16*>(o), s_fork, status);
}

}  // namespace


cudaError_t launch_fork_state(const jet_layout& lay, const jet_dims& d, int rule,
                              const float* s_prefix, const void* q, const void* k, const void* v,
                              const float* alpha, const float* beta, void* o, float* s_fork,
                              int* status, cudaStream_t st, const void* q_rows) {
  if (rule == JET_RECUR_GLA)
    return launch_rule<false>(lay, d, s_prefix, q, k, v, alpha, beta, q_rows, o, s_fork, status,
                              st);
  return launch_rule<true>(lay, d, s_prefix, q, k, v, alpha, beta, q_rows, o, s_fork, status, st);
}

}  // namespace jet
