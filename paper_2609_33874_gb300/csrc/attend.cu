// Shared-prefix cascade attention (Sec. 4.1, Fig. 1 "KV-cache text models"):
// the plan of both types, and the float32 kernels (prefix chunks, then their merge
// with the candidates' own keys); bf16 runs in attend_tc.cu. Partials are in base 2:
// m = max of score log2(e), l = sum of 2^(score log2(e) - m).
//
// Every row of request r attends to the request's P_r prefix keys; a row fed
// with y_{c,t} additionally attends to y_{c,1..t} of its own candidate. The
// prefix part is identical for all of the request's rows, so it is computed
// per (request, key/value head) with all n_r * g query vectors of the group
// sharing each prefix K/V tile (g = Hq / Hkv): the tile is read from memory
// once per group, not once per candidate. Long prefixes are split into
// chunks; each chunk leaves an unnormalised partial (max, sum of exp, sum of
// exp-weighted values) that the merge kernel combines with the short causal
// candidate part by the usual log-sum-exp rescaling.
#include <algorithm>

#include "jet_device.cuh"
#include "jet_internal.h"

namespace jet {
namespace {

constexpr int kQV = 16;       // query vectors per CTA
constexpr int kKT = 32;       // keys per tile
constexpr int kThreads = 256;
constexpr long long kTargetCtas = 4 * kPlanSMs;
constexpr int kMinChunkTc = 640;        // keys
constexpr int kFewGroups = 22, kFewItems = 44, kLeastChunk = 192;

// rows of Q, K and P are padded by 16 bytes: 16-byte reads of eight consecutive
// rows then fall in different banks
template <int DH>
constexpr size_t prefix_smem_bytes() {
  return sizeof(float) * (size_t(kQV) * (DH + 4) + size_t(kKT) * (DH + 4) + size_t(kKT) * DH +
                          size_t(kQV) * (kKT + 4));
}

// One CTA: one prefix chunk of one (request, key/value head) for kQV query
// vectors. Thread (vec = tid / 16, sub = tid % 16) scores keys sub and sub+16
// of each tile for its vector and accumulates output dims 4 sub + 64 i .. + 3.
// Small batches are bound by the chain of loads: the query block and a tile are
// fetched by 16-byte loads that are all in flight at once, and chunks go down to
// one tile (7 rows over 128 keys: 13.2 -> 4.9 us).
template <int DH>
__global__ void __launch_bounds__(kThreads)
attend_prefix_kernel(const int32_t* __restrict__ prefix_offset, const int32_t* __restrict__ row_offset,
                     int R, int N, int total_prefix, int Hq, int Hkv, int chunk,
                     const float* __restrict__ q, const float* __restrict__ k_pre,
                     const float* __restrict__ v_pre, float* __restrict__ o_part,
                     float2* __restrict__ ml_part, int* status) {
  pdl_begin();
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;                          // [kQV][DH+4], pre-scaled by log2(e)/sqrt(d)
  float* Ks = Qs + kQV * (DH + 4);           // [kKT][DH+4]
  float* Vs = Ks + kKT * (DH + 4);           // [kKT][DH]
  float* Ps = Vs + kKT * DH;                 // [kQV][kKT+4]

  const int split = blockIdx.x, qg = blockIdx.y;
  const int r = blockIdx.z / Hkv, kh = blockIdx.z % Hkv;
  const int g = Hq / Hkv;
  if (r >= R) return;
  const int n0 = row_offset[r], nr = row_offset[r + 1] - n0;
  const int p0 = prefix_offset[r], P = prefix_offset[r + 1] - p0;
  // (a request longer than the plan's chunks or vector groups is left out too)
  if (n0 < 0 || nr < 1 || n0 + nr > N || p0 < 0 || P < 0 || p0 + P > total_prefix ||
      P > chunk * int(gridDim.x) || nr * g > kQV * int(gridDim.y)) {
    if (threadIdx.x == 0) flag(status, JET_ERR_DEVICE);
    return;
  }
  const int nvec = nr * g;
  const int vbase = qg * kQV;
  if (vbase >= nvec) return;
  const int k_begin = split * chunk;
  const int k_end = min(P, k_begin + chunk);

  constexpr int C4 = DH / 4;                       // 16-byte pieces of a row
  constexpr int QI = kQV * C4 / kThreads;          // of the query block per thread
  constexpr int KI = kKT * C4 / kThreads;          // of a K (or V) tile per thread
  const int tid = threadIdx.x;
  const int vec = tid >> 4, sub = tid & 15;
  const float scale = 1.4426950408889634f * rsqrtf(float(DH));  // base-2 scores
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  // a tile's keys past k_end are zeros
  float4 kr[KI], vr[KI];
  auto fetch = [&](int kb) {
#pragma unroll
    for (int i = 0; i < KI; ++i) {
      const int e = tid + i * kThreads, j = e / C4, c = e % C4;
      const bool in = kb + j < k_end;
      const size_t idx = (size_t(p0 + kb + (in ? j : 0)) * Hkv + kh) * DH + 4 * c;
      kr[i] = in ? *reinterpret_cast<const float4*>(k_pre + idx) : zero;
      vr[i] = in ? *reinterpret_cast<const float4*>(v_pre + idx) : zero;
    }
  };
  if (k_begin < k_end) fetch(k_begin);
#pragma unroll
  for (int i = 0; i < QI; ++i) {
    const int e = tid + i * kThreads, vv = e / C4, c = e % C4, gv = vbase + vv;
    float4 x = zero;
    if (gv < nvec) {
      const int n = n0 + gv / g, h = kh * g + gv % g;
      x = *reinterpret_cast<const float4*>(q + (size_t(n) * Hq + h) * DH + 4 * c);
    }
    *reinterpret_cast<float4*>(Qs + vv * (DH + 4) + 4 * c) =
        make_float4(x.x * scale, x.y * scale, x.z * scale, x.w * scale);
  }

  constexpr int PER = DH / 64;
  float4 acc[PER];
#pragma unroll
  for (int i = 0; i < PER; ++i) acc[i] = zero;
  float m = -INFINITY, l = 0.f;

  for (int kb = k_begin; kb < k_end; kb += kKT) {
    const int nk = min(kKT, k_end - kb);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < KI; ++i) {
      const int e = tid + i * kThreads, j = e / C4, c = e % C4;
      *reinterpret_cast<float4*>(Ks + j * (DH + 4) + 4 * c) = kr[i];
      *reinterpret_cast<float4*>(Vs + j * DH + 4 * c) = vr[i];
    }
    __syncthreads();
    if (kb + kKT < k_end) fetch(kb + kKT);  // the next tile, while this one is used

    const float* qv = Qs + vec * (DH + 4);
    const float* k0 = Ks + sub * (DH + 4);
    const float* k1 = Ks + (sub + 16) * (DH + 4);
    float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
    for (int dd = 0; dd < DH; dd += 4) {
      const float4 x = *reinterpret_cast<const float4*>(qv + dd);
      const float4 a = *reinterpret_cast<const float4*>(k0 + dd);
      const float4 b = *reinterpret_cast<const float4*>(k1 + dd);
      s0 = fmaf(x.x, a.x, s0);
      s1 = fmaf(x.x, b.x, s1);
      s0 = fmaf(x.y, a.y, s0);
      s1 = fmaf(x.y, b.y, s1);
      s0 = fmaf(x.z, a.z, s0);
      s1 = fmaf(x.z, b.z, s1);
      s0 = fmaf(x.w, a.w, s0);
      s1 = fmaf(x.w, b.w, s1);
    }
    if (sub >= nk) s0 = -INFINITY;
    if (sub + 16 >= nk) s1 = -INFINITY;
    float tmax = fmaxf(s0, s1);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
    const float mn = fmaxf(m, tmax);            // finite: key 0 of the tile is valid
    const float corr = exp2f(m - mn);           // 0 on the first tile
    const float e0 = exp2f(s0 - mn), e1 = exp2f(s1 - mn);
    float psum = e0 + e1;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) psum += __shfl_xor_sync(0xffffffffu, psum, o);
    l = l * corr + psum;
    m = mn;
    Ps[vec * (kKT + 4) + sub] = e0;
    Ps[vec * (kKT + 4) + sub + 16] = e1;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < PER; ++i)
      acc[i] = make_float4(acc[i].x * corr, acc[i].y * corr, acc[i].z * corr, acc[i].w * corr);
    for (int j = 0; j < nk; ++j) {
      const float pj = Ps[vec * (kKT + 4) + j];
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const float4 x = *reinterpret_cast<const float4*>(Vs + j * DH + 4 * sub + 64 * i);
        acc[i].x = fmaf(pj, x.x, acc[i].x);
        acc[i].y = fmaf(pj, x.y, acc[i].y);
        acc[i].z = fmaf(pj, x.z, acc[i].z);
        acc[i].w = fmaf(pj, x.w, acc[i].w);
      }
    }
  }

  const int gv = vbase + vec;
  if (gv < nvec) {
    const int n = n0 + gv / g, h = kh * g + gv % g;
    const size_t base = (size_t(split) * N + n) * Hq + h;
#pragma unroll
    for (int i = 0; i < PER; ++i)
      *reinterpret_cast<float4*>(o_part + base * DH + 4 * sub + 64 * i) = acc[i];
    if (sub == 0) ml_part[base] = make_float2(m, l);
  }
}

// One warp per (row, query head), float32: the prefix chunks' partials, then the
// row's own causal candidate keys, normalised. The loads that do not depend on
// each other go out together: the chunks' (m, l) one a lane, their outputs and
// the candidate's keys and values four at a time.
template <int DH>
__global__ void __launch_bounds__(128)
attend_merge_kernel(const int32_t* __restrict__ row_req, const int32_t* __restrict__ row_cand,
                    const int32_t* __restrict__ cand_row_offset, int N, int R, int C, int Hq, int Hkv,
                    int splits, const float* __restrict__ q, const float* __restrict__ k_cand,
                    const float* __restrict__ v_cand, const float* __restrict__ o_part,
                    const float2* __restrict__ ml_part, float* __restrict__ o, int* status) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const long long idx = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (idx >= (long long)N * Hq) return;
  const int n = int(idx / Hq), h = int(idx % Hq);
  const int kh = h / (Hq / Hkv);
  const int c = row_cand[n], r = row_req[n];
  constexpr int PER = DH / 32;
  float qv[PER];
#pragma unroll
  for (int i = 0; i < PER; ++i) qv[i] = q[(size_t(n) * Hq + h) * DH + lane + 32 * i];
  float acc[PER];
  float m, l;
  combine_chunks<DH>(true, splits, N, Hq, n, h, lane, ml_part, o_part, m, l, acc);
  if (c >= 0) {
    const int first = (c < C) ? cand_row_offset[c] : -1;
    if (first < 0 || first > n || r < 0 || first - r - 1 < 0 || n - r - 1 >= N - R) {
      if (lane == 0) flag(status, JET_ERR_DEVICE);
    } else {
      const float scale = 1.4426950408889634f * rsqrtf(float(DH));  // base 2
      for (int n4 = first; n4 <= n; n4 += 4) {
        float kv[4][PER], vv[4][PER], sc[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const size_t kb = (size_t(min(n4 + t, n) - r - 1) * Hkv + kh) * DH + lane;
#pragma unroll
          for (int i = 0; i < PER; ++i) {
            kv[t][i] = k_cand[kb + 32 * i];
            vv[t][i] = v_cand[kb + 32 * i];
          }
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float sp = 0.f;
#pragma unroll
          for (int i = 0; i < PER; ++i) sp = fmaf(qv[i] * scale, kv[t][i], sp);
          sc[t] = sp;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
          for (int t = 0; t < 4; ++t) sc[t] += __shfl_xor_sync(0xffffffffu, sc[t], off);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (n4 + t > n) break;
          const float mn = fmaxf(m, sc[t]);
          const float a = exp2f(m - mn), b = exp2f(sc[t] - mn);
#pragma unroll
          for (int i = 0; i < PER; ++i) acc[i] = acc[i] * a + b * vv[t][i];
          l = l * a + b;
          m = mn;
        }
      }
    }
  }
  const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
  for (int i = 0; i < PER; ++i) o[(size_t(n) * Hq + h) * DH + lane + 32 * i] = acc[i] * inv;
}

template <int DH>
cudaError_t launch_dh(const jet_layout& lay, const jet_dims& d, const AttnPlan& plan,
                         const void* q, const void* k_pre, const void* v_pre, const void* k_cand,
                         const void* v_cand, void* o, void* ws, int* status, cudaStream_t st) {
  const jet_sizes& n = lay.n;
  float* o_part = static_cast<float*>(ws);
  float2* ml_part = reinterpret_cast<float2*>(o_part + size_t(plan.splits) * n.N * d.Hq * DH);
  cudaError_t e;
  if (d.dtype == JET_DTYPE_BF16) {
    // the tensor-core path covers the candidates' own keys and the combine
    return launch_attend_tc(lay, d, plan, q, k_pre, v_pre, k_cand, v_cand, o, o_part, ml_part,
                            status, st);
  } else {
    const size_t smem = prefix_smem_bytes<DH>();
    e = cudaFuncSetAttribute(attend_prefix_kernel<DH>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    dim3 grid(plan.splits, plan.qgroups, unsigned(n.R * d.Hkv));
    e = launch_pdl(attend_prefix_kernel<DH>, grid, dim3(kThreads), smem, st, lay.prefix_offset,
                   lay.row_offset, n.R, n.N, n.total_prefix, d.Hq, d.Hkv, plan.chunk,
                   static_cast<const float*>(q), static_cast<const float*>(k_pre),
                   static_cast<const float*>(v_pre), o_part, ml_part, status);
  }
  if (e != cudaSuccess) return e;
  const long long warps = (long long)n.N * d.Hq;
  return launch_pdl(attend_merge_kernel<DH>, dim3(unsigned((warps + 3) / 4)), dim3(128), 0, st,
                    lay.row_req, lay.row_cand, lay.cand_row_offset, n.N, n.R, n.C, d.Hq, d.Hkv,
                    plan.splits, static_cast<const float*>(q), static_cast<const float*>(k_cand),
                    static_cast<const float*>(v_cand), o_part, ml_part, static_cast<float*>(o),
                    status);
}

}  // namespace

AttnPlan attn_plan(const jet_sizes& n, const jet_dims& d) {
  AttnPlan p{};
  if (n.R <= 0 || n.N <= 0 || d.Hkv <= 0 || d.Hq <= 0) return p;
  const int g = d.Hq / d.Hkv;
  const bool tc = d.dtype == JET_DTYPE_BF16;
  const int gran = tc ? 64 : kKT;                 // keys per tile
  // query vectors per CTA: the tensor-core kernel takes whole rows (128 / g
  // rows of g heads), the float32 kernel kQV vectors
  const int qv = tc ? std::max(1, attn_tc_block() / g) * g : kQV;
  p.qgroups = (n.max_rows * g + qv - 1) / qv;
  // query blocks of an average request: blocks past a request's vectors exit
  // at once, so they do not count as work
  const long long avg_vecs = ((long long)n.N * g + n.R - 1) / n.R;
  const long long groups = (long long)n.R * d.Hkv * std::max<long long>(1, (avg_vecs + qv - 1) / qv);
  const int max_splits = std::max(1, (n.max_prefix + gran - 1) / gran);
  int chunk;
  if (tc) {
    // the persistent kernel (one CTA per SM; items dealt out by their requests'
    // lengths, or longest first from a list: `sorted` below) splits a request's
    // prefix into near-equal chunks: no shorter than kMinChunkTc keys (an item's
    // fixed cost - query block in, f32 partial out and read back by the combine - is
    // worth about five 64-key tiles), and no finer than half of one SM's share of all
    // key tiles, so that the schedule can balance
    const double avg_tiles = double(n.total_prefix) / n.R / 64.0 + 0.5;
    const double share = double(groups) * avg_tiles / kPlanSMs;  // tiles per SM
    int least = kMinChunkTc;
    // a few long prefixes leave most SMs idle at that length: then about
    // kFewItems chunks in all, of at least kLeastChunk keys (one 6,000-key request
    // with two kv heads: 320 keys 17.5 us, 640 keys 19.8 us, 128 keys 21.3 us). Past
    // kFewGroups the combine costs what shorter chunks gain, and from 19 groups on in
    // prefixes of up to 448 keys too (d 256; as here and at 640 keys: 8 groups of 1,000
    // keys 13.2 and 17.7 us, 16 groups 15.2 and 17.9, of 400 12.9 and 13.3; 20 groups
    // of 200 - 1,200 16.5 and 18.7, of 200 - 600 14.9 and 15.5, of 400 14.0 and 13.4;
    // 24 groups of 400 14.0 and 13.4, of 700 to 4,000 the same)
    if (groups <= kFewGroups && (groups <= 18 || n.max_prefix > 448)) {
      const long long even = (long long)(double(groups) * avg_tiles / kFewItems + 0.999) * 64;
      least = int(std::max<long long>(kLeastChunk, std::min<long long>(kMinChunkTc, even)));
    }
    chunk = std::max(least, int(share / 2.0 + 0.999) * 64);
    chunk = std::min(chunk, max_splits * 64);  // one chunk holds the longest prefix
  } else {
    // about four CTAs per SM
    long long want = (kTargetCtas + groups - 1) / groups;
    int splits = int(std::min<long long>(std::max<long long>(want, 1), max_splits));
    chunk = (n.max_prefix + splits - 1) / splits;
    chunk = (chunk + gran - 1) / gran * gran;
  }
  p.chunk = chunk;
  p.splits = (n.max_prefix + chunk - 1) / chunk;
  const size_t vecs = size_t(p.splits) * n.N * d.Hq;
  p.bytes = vecs * d.d * sizeof(float) + vecs * sizeof(float2);
  // Items dealt out back and forth in the order of the requests' lengths balance well
  // when that is the order of the items' own lengths: unsplit requests, or lengths
  // within a quarter of their mean's. Long chunks (16 key tiles or more) of uneven
  // requests do not come in that order, and with at most 2.5 groups an SM a CTA has
  // too few of them to even out; then a longest-first list and a shared counter pay
  // for their launch (requests of 2,048 - 8,192 keys, two kv heads: 128 with the list
  // 240 us, dealt 245; 90 181 and 188; 256 unsplit 438 and 426; 64 of 4,096 111 and
  // 106; 400 groups of 300 - 4,000 keys 175 and 171).
  p.sorted = tc && p.splits > 1 && chunk >= 16 * 64 && 2 * groups <= 5 * kPlanSMs &&
             4LL * n.max_prefix * n.R > 5LL * n.total_prefix;
  // the work list: (request, kv head, query block, chunk) items plus two counters,
  // 16-byte aligned, after the partials
  if (p.sorted) p.bytes += 32 + 16 * size_t(n.R) * d.Hkv * p.qgroups * p.splits;
  return p;
}

cudaError_t launch_prefix_attend(const jet_layout& lay, const jet_dims& d, const AttnPlan& plan,
                                 const void* q, const void* k_pre, const void* v_pre,
                                 const void* k_cand, const void* v_cand, void* o, void* ws,
                                 int* status, cudaStream_t st) {
#define JET_ATT(DH) \
  return launch_dh<DH>(lay, d, plan, q, k_pre, v_pre, k_cand, v_cand, o, ws, status, st)
  if (d.d == 64) JET_ATT(64);
  if (d.d == 128) JET_ATT(128);
  if (d.d == 256) JET_ATT(256);
#undef JET_ATT
  return cudaErrorInvalidValue;
}

}  // namespace jet
