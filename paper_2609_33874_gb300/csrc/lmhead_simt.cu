// LM head with on-chip log-sum-exp partials, float32 FMA path (Eq. 1, Eq. 2).
//
// z_{n,v} = hidden[n] . w_lm[v] for a tile of MR rows x 128 vocabulary
// entries; the tile's logits are reduced on chip to one (max, sum of exp) pair
// per row and the logits of the targets that fall in the tile are kept
// (Sec. 4.2: only the needed log-probabilities leave the GPU). float32 inputs
// take this path: the tensor cores would round them to tf32. bf16 inputs take
// the tcgen05 kernel instead.
//
// What bounds it: small batches are bound by the weights' stream through few
// SMs (one CTA per 128 vocabulary entries), larger ones by float32 FMA. So the
// operands arrive by asynchronous 16-byte copies, kStages K slices in flight
// (about 100 KB an SM), and a thread forms 4 vocabulary entries x MR rows from
// 16-byte shared-memory loads: the eight warps split every 32-element K slice
// (four elements each) instead of the tile, so that a row's float4 is one
// broadcast and a weight float4 is used MR times. The warps' partial sums are
// added at the end (eight chains of D / 8 terms: shorter than one of D).
// With few tiles two CTAs split a tile's K slices. 7 rows x 512 x 8192 (16.8 MB of
// weights): 9.9 us, 11.2 with one CTA a tile; a 32-row tile filled by 4-byte loads,
// one K slice at a time, took 73.6 us.
#include "jet_device.cuh"
#include "jet_internal.h"
#include "sm100_ptx.cuh"

namespace jet {
namespace {

constexpr int kBV = kVocabTile;  // vocabulary entries per tile (128)
constexpr int kBK = 32;          // hidden elements per stage: 128 bytes, 4 per warp
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kStages = 6;

// one stage: 128 weight rows, then MR hidden rows, of 128 bytes each
template <int MR>
constexpr int stage_floats() { return (kBV + MR) * kBK; }
template <int MR>
constexpr size_t smem_bytes() {
  const size_t ring = size_t(kStages) * stage_floats<MR>() * sizeof(float);
  const size_t red = size_t(kWarps) * MR * kBV * sizeof(float);  // reuses the ring
  return ring > red ? ring : red;
}

// 16 bytes, or zeros when `ok` is false (nothing is read then)
__device__ __forceinline__ void copy16(float* dst, const float* src, bool ok) {
  const uint32_t n = ok ? 16u : 0u;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src), "r"(n)
               : "memory");
}

// 16-byte chunk c of row r of a stage, permuted by the row so that the rows a
// warp reads at one chunk fall in different banks
__device__ __forceinline__ int chunk_at(int r, int c) { return r * kBK + ((c ^ (r & 7)) << 2); }

// PAIR: the two CTAs of a cluster take half of the K slices each, and the even one
// adds the odd one's sums to its own.
template <int MR, bool PAIR>
__global__ void __launch_bounds__(kThreads)
lmhead_simt_kernel(const int32_t* __restrict__ target_ids, const int32_t* __restrict__ row_tgt_offset,
                   const int32_t* __restrict__ row_tgt_index, int N, int T_, int V, int D,
                   const float* __restrict__ hidden, const float* __restrict__ w_lm,
                   float2* __restrict__ part, float* __restrict__ z_tgt, int* status) {
  pdl_begin();
  extern __shared__ __align__(16) float ring[];
  const int row0 = int(PAIR ? blockIdx.x >> 1 : blockIdx.x) * MR;
  const bool odd = PAIR && (blockIdx.x & 1);
  const int vt = blockIdx.y;
  const int v0 = vt * kBV;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // this CTA's K slices [k0, k0 + nkb)
  const int all = (D + kBK - 1) / kBK;
  const int k0 = odd ? all / 2 : 0;
  const int nkb = !PAIR ? all : odd ? all - all / 2 : all / 2;

  // K slice k0 + kb into its stage: the rows past N and V and the elements past D
  // (a multiple of 8) are zeros
  auto load = [&](int kb) {
    float* st = ring + (kb % kStages) * stage_floats<MR>();
#pragma unroll
    for (int i = 0; i < kBV * 8 / kThreads; ++i) {
      const int e = tid + i * kThreads, r = e >> 3, c = e & 7;
      const int kx = (k0 + kb) * kBK + 4 * c;
      const bool ok = v0 + r < V && kx < D;
      copy16(st + chunk_at(r, c), w_lm + (ok ? size_t(v0 + r) * D + kx : 0), ok);
    }
    if (tid < MR * 8) {
      const int r = tid >> 3, c = tid & 7;
      const int kx = (k0 + kb) * kBK + 4 * c;
      const bool ok = row0 + r < N && kx < D;
      copy16(st + kBV * kBK + r * kBK + 4 * c, hidden + (ok ? size_t(row0 + r) * D + kx : 0), ok);
    }
  };
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) {
    if (s < nkb) load(s);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }

  // the targets predicted by this warp's rows (row0 + warp + 8 i), one a lane,
  // read while the first slices are on their way (rows with more than 32
  // targets read the rest at the end)
  constexpr int RW = MR / kWarps;
  int tj[RW], tv[RW], t0[RW], t1[RW];
#pragma unroll
  for (int i = 0; i < RW; ++i) {
    const int n = row0 + warp + kWarps * i;
    t0[i] = n < N ? row_tgt_offset[n] : 0;
    t1[i] = n < N ? row_tgt_offset[n + 1] : 0;
    tj[i] = t0[i] + lane < t1[i] ? row_tgt_index[t0[i] + lane] : -1;
  }
#pragma unroll
  for (int i = 0; i < RW; ++i) {
    const bool in = t0[i] + lane < t1[i];
    if (in && (tj[i] < 0 || tj[i] >= T_)) flag(status, JET_ERR_DEVICE);
    tv[i] = in && tj[i] >= 0 && tj[i] < T_ ? target_ids[tj[i]] - v0 : -1;
  }

  float acc[4][MR];
#pragma unroll
  for (int b = 0; b < 4; ++b)
#pragma unroll
    for (int a = 0; a < MR; ++a) acc[b][a] = 0.f;
  for (int kb = 0; kb < nkb; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();  // slice kb is in, and nobody reads the stage refilled next
    if (kb + kStages - 1 < nkb) load(kb + kStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* st = ring + (kb % kStages) * stage_floats<MR>();
    float4 w[4];
#pragma unroll
    for (int b = 0; b < 4; ++b)
      w[b] = *reinterpret_cast<const float4*>(st + chunk_at(lane + 32 * b, warp));
#pragma unroll
    for (int a = 0; a < MR; ++a) {
      const float4 h = *reinterpret_cast<const float4*>(st + kBV * kBK + a * kBK + 4 * warp);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        acc[b][a] = fmaf(h.x, w[b].x, acc[b][a]);
        acc[b][a] = fmaf(h.y, w[b].y, acc[b][a]);
        acc[b][a] = fmaf(h.z, w[b].z, acc[b][a]);
        acc[b][a] = fmaf(h.w, w[b].w, acc[b][a]);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  float* red = ring;  // [warp][row][vocabulary entry]
#pragma unroll
  for (int a = 0; a < MR; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) red[(warp * MR + a) * kBV + lane + 32 * b] = acc[b][a];
  __syncthreads();
  if (PAIR) {
    if (odd) {
      for (int e = tid; e < MR * kBV; e += kThreads) {
        float z = red[e];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) z += red[w * MR * kBV + e];
        red[e] = z;  // read and written by this thread alone
      }
    }
    sm100::cluster_sync();
  }

  // epilogue: warp w takes rows w, w + 8 ..: base-2 (max, sum) over the tile's
  // vocabulary, target gather
#pragma unroll
  for (int i = 0; i < RW; ++i) {
    const int a = warp + kWarps * i, n = row0 + a;
    if (n >= N || odd) break;
    constexpr float kLog2e = 1.4426950408889634f;
    float z[4], mx = -INFINITY;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      z[b] = 0.f;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) z[b] += red[(w * MR + a) * kBV + lane + 32 * b];
      if (PAIR) z[b] += sm100::ld_shared_remote(red + a * kBV + lane + 32 * b, 1);
      if (v0 + lane + 32 * b < V) mx = fmaxf(mx, z[b] * kLog2e);
    }
    mx = warp_max(mx);
    float s = 0.f;
#pragma unroll
    for (int b = 0; b < 4; ++b)
      if (v0 + lane + 32 * b < V) s += exp2f(z[b] * kLog2e - mx);
    s = warp_sum(s);
    if (lane == 0) part[size_t(n) * gridDim.y + vt] = make_float2(mx, s);
    for (int t = t0[i]; t < t1[i]; t += 32) {
      int j = tj[i], off = tv[i];
      if (t > t0[i]) {
        j = t + lane < t1[i] ? row_tgt_index[t + lane] : -1;
        const bool in = j >= 0 && j < T_;
        if (t + lane < t1[i] && !in) flag(status, JET_ERR_DEVICE);
        off = in ? target_ids[j] - v0 : -1;
      }
      unsigned hit = __ballot_sync(0xffffffffu, off >= 0 && off < kBV);
      for (; hit; hit &= hit - 1) {
        const int src = __ffs(hit) - 1;
        const int jj = __shfl_sync(0xffffffffu, j, src), o = __shfl_sync(0xffffffffu, off, src);
        if ((o & 31) == lane) {
          const int b = o >> 5;
          z_tgt[jj] = b == 0 ? z[0] : b == 1 ? z[1] : b == 2 ? z[2] : z[3];
        }
      }
    }
  }
  if (PAIR) sm100::cluster_sync();  // the odd CTA's sums stay until they are read
}

template <int MR>
cudaError_t launch_mr(const jet_layout& lay, const jet_dims& d, const ScorePlan& plan,
                      const void* hidden, const void* w_lm, void* ws, int* status,
                      cudaStream_t st) {
  const jet_sizes& n = lay.n;
  char* base = static_cast<char*>(ws);
  float2* part = reinterpret_cast<float2*>(base + plan.part_off);
  float* z_tgt = reinterpret_cast<float*>(base + plan.ztgt_off);
  const size_t smem = smem_bytes<MR>();
  // pairs while both CTAs of every tile find an SM of their own: a
  // one-request step of 7 rows and 8,192 entries takes 36.8 us of D 1,024 without
  // them, 28.7 with, 67.6 and 45.8 of D 2,560, 23.4 both ways of D 512 and below
  // (its launches); past that the halves would queue
  const long long row_tiles = (n.N + MR - 1) / MR;
  const bool pair = 2 * row_tiles * plan.vtiles <= sm_count();
  const auto kern = pair ? lmhead_simt_kernel<MR, true> : lmhead_simt_kernel<MR, false>;
  const cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  const dim3 grid(unsigned(pair ? 2 * row_tiles : row_tiles), unsigned(plan.vtiles));
  auto launch = [&](auto how) {
    return how(kern, grid, dim3(kThreads), smem, st, lay.target_ids, lay.row_tgt_offset,
               lay.row_tgt_index, n.N, n.T, n.V, d.D, static_cast<const float*>(hidden),
               static_cast<const float*>(w_lm), part, z_tgt, status);
  };
  return pair ? launch([](auto... x) { return launch_pdl_pairs(x...); })
              : launch([](auto... x) { return launch_pdl(x...); });
}

}  // namespace

cudaError_t launch_lmhead_simt(const jet_layout& lay, const jet_dims& d, const ScorePlan& plan,
                               const void* hidden, const void* w_lm, void* ws, int* status,
                               cudaStream_t st) {
  // one small row tile for up to 8 rows (half the accumulators and epilogue of
  // the 16-row tile, 64 more registers free); more rows take 16 at a time, which
  // halves the weight reads from L2 per row
  if (lay.n.N <= 8) return launch_mr<8>(lay, d, plan, hidden, w_lm, ws, status, st);
  return launch_mr<16>(lay, d, plan, hidden, w_lm, ws, status, st);
}

}  // namespace jet
