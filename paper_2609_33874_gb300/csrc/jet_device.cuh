// Device helpers shared by the kernels of libjet (header-only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "jet.h"

namespace jet {

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename T>
__device__ __forceinline__ T from_f32(float x);
template <>
__device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}

// ---- programmatic dependent launch -------------------------------------------
// Every kernel of libjet is launched with programmatic stream serialization
// (launch_pdl), so it may start while the kernel before it in the stream still
// runs. pdl_begin() lets the kernel after it start early in turn, then waits
// until all earlier work in the stream has completed and its writes are
// visible. A kernel touches no global memory before pdl_begin(); setting up
// shared memory and barriers may come first.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// record the first error a kernel meets; later ones keep the first code
__device__ __forceinline__ void flag(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// (max, sum of exp relative to max) pair combination; an empty pair is
// (-inf, 0)
__device__ __forceinline__ void ms_combine(float& m, float& s, float m2, float s2) {
  const float mn = fmaxf(m, m2);
  if (mn == -INFINITY) return;
  s = s * __expf(m - mn) + s2 * __expf(m2 - mn);
  m = mn;
}

// the same in base 2: s = sum 2^(x - m)
__device__ __forceinline__ void ms_combine2(float& m, float& s, float m2, float s2) {
  const float mn = fmaxf(m, m2);
  if (mn == -INFINITY) return;
  s = s * exp2f(m - mn) + s2 * exp2f(m2 - mn);
  m = mn;
}

// A warp combines the base-2 partials (m, l, O) of row n, head h over its prefix
// chunks: l and acc (elements lane + 32 i of the head) relative to m, the largest
// of their maxima. The (m, l) of 32 chunks are read one a lane and the chunks'
// outputs four at a time, with `ahead` the first four beside the (m, l): up to four
// chunks then cost one memory latency (64 requests of 100 - 2,000 keys: the whole call 47.9 ->
// 46.0 us; eight at a time 48.1 us; one 6,000-key request in 19 chunks 18.9 ->
// 18.5 us).
template <int DH>
__device__ __forceinline__ void combine_chunks(bool ahead, int splits, int N, int Hq, int n, int h,
                                               int lane, const float2* __restrict__ ml_part,
                                               const float* __restrict__ o_part, float& m,
                                               float& l, float (&acc)[DH / 32]) {
  constexpr int PER = DH / 32, kGroup = 4;
  const size_t base = size_t(n) * Hq + h, step = size_t(N) * Hq;
  float v[kGroup][PER];
  auto load = [&](int s0) {
#pragma unroll
    for (int g = 0; g < kGroup; ++g) {
      if (s0 + g < splits) {
        const float* p = o_part + (base + size_t(s0 + g) * step) * DH + lane;
#pragma unroll
        for (int i = 0; i < PER; ++i) v[g][i] = p[32 * i];
      }
    }
  };
  m = -INFINITY;
  l = 0.f;
#pragma unroll
  for (int i = 0; i < PER; ++i) acc[i] = 0.f;
  auto load_ml = [&](int s32) {
    return s32 + lane < splits ? ml_part[base + size_t(s32 + lane) * step]
                               : make_float2(-INFINITY, 0.f);
  };
  float2 ml = load_ml(0);
  if (ahead) load(0);
  for (int s32 = 0; s32 < splits; s32 += 32) {
    if (s32 > 0) ml = load_ml(s32);
    // an empty chunk has l = 0; a NaN l (a NaN score) counts, whatever its maximum,
    // and so does a chunk whose weight underflows (0 x an infinite output is NaN)
    const bool held = ml.y != 0.f;
    if (!held) ml.x = -INFINITY;
    const float mn = fmaxf(m, warp_max(ml.x));
    const float keep = mn == -INFINITY ? 1.f : exp2f(m - mn);
    const float w = held ? exp2f(ml.x - mn) : 0.f;
    l = l * keep + warp_sum(ml.y * w);
    m = mn;
#pragma unroll
    for (int i = 0; i < PER; ++i) acc[i] *= keep;
    const unsigned some = __ballot_sync(0xffffffffu, held);
    for (int s0 = s32; s0 < min(s32 + 32, splits); s0 += kGroup) {
      if (!(some >> (s0 & 31) & ((1u << kGroup) - 1))) continue;  // all empty
      if (!ahead || s0 > 0) load(s0);
#pragma unroll
      for (int g = 0; g < kGroup; ++g) {
        const float ws = __shfl_sync(0xffffffffu, w, (s0 + g) & 31);
        // an empty chunk's outputs were not written
        if (some >> ((s0 + g) & 31) & 1u) {
#pragma unroll
          for (int i = 0; i < PER; ++i) acc[i] = fmaf(ws, v[g][i], acc[i]);
        }
      }
    }
  }
}

}  // namespace jet
