// Causal self-attention over every request's prefix (the prefill, Sec. 4.1) on
// pairs of SMs with the 5th-generation tensor cores; bf16, head dimensions 128
// and 256 (64, and batches of prefixes that fill less than a pair's block, run on
// single SMs with the scoring step's kernel, attend_tc.cu).
//
// What bounds it: every query vector needs its own softmax and the key/value
// tiles come from L2, and one SM that streams tiles for 128 query vectors
// alone needs 64 KB of K and V per 64 keys (d = 256) - at two tiles in flight
// that hand-off, not the tensor pipe, set the pace (1.27 us per 64 keys where
// the MMAs need 0.53). So two SMs share a tile (tcgen05 cta_group::2, M = 256):
// each holds its own 128 query vectors and half of every tile - 64 of 128 keys
// of K, half of the columns of V - which halves the bytes an SM takes in and
// doubles the keys its shared memory holds. Keys come 128 at a time (an N = 64
// product costs as much tensor time as N = 128), the output drain has warps of
// its own, and the next item's products start under it.
// Measured against one SM per query block, 64 keys at a time: 90,016 positions
// of 16 requests (16/2 heads, d 256) 4,602 -> 2,792 us (1.65 PFLOP/s), 12,519
// positions of 16 short requests (24/4 heads) 198 -> 145 us, where the start and
// end of each item (1 to 10 tiles long) is what is left.
//
// An item is (request, kv head, block of 2 rb positions), rb = 128 / g whole
// positions of g = Hq / Hkv heads per SM. Roles of each CTA of the pair:
//   warp 0       TMA producer: its query block, K and V halves (2-stage rings)
//   warp 1       TMEM allocation; in the even CTA the MMA issuer:
//                  S_j  = Q K_j^T  (256 vectors x 128 keys)
//                  O   += P_j V_j  (256 vectors x d)
//                two S tiles alternate; P_j (bf16) takes the place of the first
//                half of S_j. The issuing thread's MMAs run in order, so S_j
//                overwrites P_{j-2} after its P V.
//   warp 2       schedule: which items this pair runs, one ahead
//   warps 3..6   softmax: thread = query vector = TMEM lane
//   warps 7..10  output: O / l to memory
// All barriers an MMA waits for live in the even CTA; the commits reach both.
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

constexpr int kBV = 128;       // query vectors per CTA (TMEM lanes)
constexpr int kBN = 128;       // keys per tile of the pair
constexpr int kHalfN = kBN / 2;
constexpr int kStages = 2;
constexpr int kThreads = 352;
constexpr uint64_t kDrainNs = 200000000ull;
constexpr float kRescaleLog2 = 8.f;  // rescale O only when the max grows by > 2^8

template <int DH>
struct Geo {
  static constexpr int kSlices = DH / 64;                       // 64-wide d slices of Q and K
  static constexpr int kVSlices = DH / 128;                     // of this CTA's half of V
  static constexpr uint32_t kQBytes = kBV * DH * 2;
  static constexpr uint32_t kKBytes = kHalfN * DH * 2;          // this CTA's 64 keys
  static constexpr uint32_t kVBytes = kBN * DH;                 // 128 keys x d / 2 columns
  static constexpr uint32_t kOffK = kQBytes;
  static constexpr uint32_t kOffV = kOffK + kStages * kKBytes;
  static constexpr uint32_t kOffStage = kOffV + kStages * kVBytes;  // 4 KB per output warp
  static constexpr uint32_t kOffL = kOffStage + 4 * 4096;           // 1 / l, two items
  static constexpr uint32_t kOffBar = kOffL + 2 * kBV * 4;
  static constexpr uint32_t kBytes = kOffBar + 512;
  // TMEM: the two S tiles, then O
  static constexpr uint32_t kOCol = 2 * kBN;
  static constexpr uint32_t kTmemCols = 512;
};
static_assert(Geo<256>::kBytes + 1024 <= 232448, "shared memory of one CTA");

struct PreArgs {
  const int32_t* prefix_offset;
  const int32_t* req_order;
  __nv_bfloat16* o;
  int* status;
  int R, total, Hq, Hkv, g, rb;
  float scale_log2;  // log2(e) / sqrt(d)
  uint64_t wait_ns;  // budget of one bounded wait (jet_set_wait_budget_ns)
  int hold_first;    // test hook (jet_set_test_stall): withhold the first query block
};

// One item as the schedule warp publishes it (ntiles 0: no more items).
struct __align__(16) Item {
  int p0;      // the request's first position in the packed prefixes
  int kh;      // key/value head
  int row0;    // this CTA's first position within the request
  int nv;      // this CTA's query vectors (may be 0 in the odd CTA)
  int k_end;   // keys of the block: the request's first k_end positions
  int ntiles;
  int pad[2];
};

// SW128 K-major position of 16-byte chunk c of row i inside one 64-wide slice
__device__ __forceinline__ uint32_t sw128(int i, int c) {
  return uint32_t(i) * 128u + (uint32_t(c ^ (i & 7)) << 4);
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// 3-D tiled load into this CTA's shared memory, counted on the even CTA's
// barrier (a mapa address)
__device__ __forceinline__ void tma_load_3d_pair(void* dst, const CUtensorMap* map, uint32_t bar,
                                                 int32_t x, int32_t y, int32_t z,
                                                 uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2"
      ".L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar), "l"(policy)
      : "memory");
}

__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int32_t x, int32_t y,
                                                int32_t z) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(z)
               : "memory");
}

template <int DH>
__global__ void __launch_bounds__(kThreads, 1)
prefill_pair_kernel(const __grid_constant__ CUtensorMap tmQ,
                    const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const PreArgs a) {
  using G = Geo<DH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  float* linv = reinterpret_cast<float*>(smem + G::kOffL);       // [2][kBV]
  Item* ring = reinterpret_cast<Item*>(smem + G::kOffBar);       // [2]
  uint64_t* k_full = reinterpret_cast<uint64_t*>(ring + 2);      // even CTA
  uint64_t* k_empty = k_full + kStages;
  uint64_t* v_full = k_empty + kStages;                          // even CTA
  uint64_t* v_empty = v_full + kStages;
  uint64_t* s_full = v_empty + kStages;                          // [2]
  uint64_t* p_full = s_full + 2;                                 // [2], even CTA
  uint64_t* item_full = p_full + 2;                              // [2]
  uint64_t* item_empty = item_full + 2;                          // [2]
  uint64_t* q_full = item_empty + 2;                             // even CTA
  uint64_t* q_free = q_full + 1;   // the item's last QK^T is done
  uint64_t* o_full = q_free + 1;   // the item's last PV is done
  uint64_t* o_free = o_full + 1;   // O has been read out (even CTA)
  uint64_t* l_full = o_free + 1;   // [2]: the item's 1 / l are in linv
  uint64_t* l_free = l_full + 2;   // [2]: and have been read
  uint64_t* drain = l_free + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = int(blockIdx.x >> 1), npairs = int(gridDim.x >> 1);
  const int g = a.g, rb = a.rb;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(k_full + s, 1);
      mbar_init(k_empty + s, 1);
      mbar_init(v_full + s, 1);
      mbar_init(v_empty + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(s_full + b, 1);
      mbar_init(p_full + b, 8);  // both CTAs' softmax warps
      mbar_init(item_full + b, 1);
      mbar_init(l_full + b, 4);
      mbar_init(l_free + b, 4);
      // producer, softmax and output warps, and the even CTA's MMA thread
      mbar_init(item_empty + b, rank == 0 ? 10 : 9);
    }
    mbar_init(q_full, 1);
    mbar_init(q_free, 1);
    mbar_init(o_full, 1);
    mbar_init(o_free, 8);  // both CTAs' output warps
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  // the query blocks arrive by TMA (rows [0, rb g)); zero the rows past them
  // once so that no stale shared memory enters the MMA
  for (int e = int(threadIdx.x); e < (kBV - rb * g) * (DH / 8); e += kThreads) {
    const int i = rb * g + e / (DH / 8), c = e % (DH / 8);
    *reinterpret_cast<uint4*>(smem + (c >> 3) * (kBV * 128) + sw128(i, c & 7)) =
        make_uint4(0, 0, 0, 0);
  }
  fence_proxy_async_shared();
  // global memory and TMEM only after the previous kernel of the stream is done
  pdl_begin();
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, G::kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the even CTA's barriers and both query tails are ready
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 2) {
    // ---------------------------------------------------------------- schedule
    // Items in the order: requests by decreasing length, a request's blocks
    // from the last (longest) to the first, kv heads fastest, so that the pairs
    // at work share one request's K and V in L2. The pairs deal them out back
    // and forth (0 .. n-1, n-1 .. 0, ...): neighbours differ by at most a block,
    // so every pair gets nearly the same work, without a work list or a counter.
    // Both CTAs derive the same items.
    long long before = 0;  // items of the requests before this window of 32
    int base = 0, total = -1, cnt = 0, inc = 0, r = 0, P = 0;
    for (int u = 0, round = 0;; ++round) {
      const long long k =
          (long long)round * npairs + ((round & 1) ? npairs - 1 - pair : pair);
      Item it{};
      for (;;) {
        if (total < 0) {  // the window's block counts
          const int ri = base + lane;
          cnt = r = P = 0;
          if (ri < a.R) {
            r = a.req_order[ri];
            if (r >= 0 && r < a.R) {
              const int p0 = a.prefix_offset[r];
              P = a.prefix_offset[r + 1] - p0;
              if (p0 < 0 || P < 1 || p0 + P > a.total) {
                flag(a.status, JET_ERR_DEVICE);
                P = 0;
              }
            } else {
              flag(a.status, JET_ERR_DEVICE);
            }
            cnt = a.Hkv * ((P + 2 * rb - 1) / (2 * rb));
          }
          inc = cnt;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
          }
          total = __shfl_sync(0xffffffffu, inc, 31);
        }
        if (k < before + total) {
          const unsigned hit = __ballot_sync(0xffffffffu, k < before + inc);
          const int src = __ffs(hit) - 1;
          const int kk = int(k - before) - __shfl_sync(0xffffffffu, inc - cnt, src);
          const int rr = __shfl_sync(0xffffffffu, r, src);
          const int PP = __shfl_sync(0xffffffffu, P, src);
          const int nq = __shfl_sync(0xffffffffu, cnt, src) / a.Hkv;
          const int qb = nq - 1 - kk / a.Hkv;
          it.p0 = a.prefix_offset[rr];
          it.kh = kk % a.Hkv;
          it.row0 = (2 * qb + int(rank)) * rb;
          it.nv = min(rb, max(0, PP - it.row0)) * g;
          it.k_end = min(PP, (qb + 1) * 2 * rb);
          it.ntiles = (it.k_end + kBN - 1) / kBN;
          break;
        }
        before += total;
        base += 32;
        if (base >= a.R) break;  // no more items
        total = -1;
      }
      const int slot = u & 1;
      bool okw = true;
      if (lane == 0) okw = mbar_wait(item_empty + slot, ((u >> 1) & 1) ^ 1u, a.wait_ns, abort_flag);
      if (!__shfl_sync(0xffffffffu, okw ? 1 : 0, 0)) {
        if (lane == 0) {
          *abort_flag = 1;
          flag(a.status, JET_ERR_TIMEOUT);
        }
        break;
      }
      if (lane == 0) {
        ring[slot] = it;
        mbar_arrive(item_full + slot);
        if (it.nv > 0) {  // start the query block on its way into L2
#pragma unroll
          for (int sl = 0; sl < G::kSlices; ++sl)
            tma_prefetch_3d(&tmQ, sl * 64, it.kh * g, it.p0 + it.row0);
        }
      }
      ++u;
      if (it.ntiles == 0) break;
    }
  } else if (warp == 0) {
    // ---------------------------------------------------------------- producer
    if (elect_one()) {
      const uint64_t pol_kv = policy_evict_normal(), pol_q = policy_evict_first();
      const uint32_t bar_q = mapa_shared(q_full, 0), bar_k = mapa_shared(k_full, 0),
                     bar_v = mapa_shared(v_full, 0);
      uint32_t k_issued = 0, k_par = 0, v_issued = 0, v_par = 0, q_issued = 0, q_par = 0;
      int T = 0, v = 0;  // tiles and items so far
      bool ok = true;
      for (int u = 0; ok; ++u) {
        const int slot = u & 1;
        if (!mbar_wait(item_full + slot, (u >> 1) & 1, a.wait_ns, abort_flag)) {
          ok = false;
          break;
        }
        const Item e = ring[slot];
        mbar_arrive(item_empty + slot);
        if (e.ntiles == 0) break;
        int jq = 0, jk = 0, jv = 0;  // issued: the query block, K and V tiles
        IdleClock clk;
        while (jq == 0 || jv < e.ntiles) {
          bool progressed = false;
          // the query block, once the previous item's last QK^T has read its own
          if (jq == 0 && (v == 0 || mbar_test(q_free, (v - 1) & 1))) {
            if (v == 0 && a.hold_first) {
              // test hook: the first query block never lands
            } else {
              if (rank == 0) mbar_arrive_expect_tx(q_full, 2u * G::kSlices * 64 * 2 * g * rb);
#pragma unroll
              for (int sl = 0; sl < G::kSlices; ++sl)
                tma_load_3d_pair(smem + sl * (kBV * 128), &tmQ, bar_q, sl * 64, e.kh * g,
                                 e.p0 + e.row0, pol_q);
              q_issued = 1;
              q_par = v & 1;
            }
            jq = 1;
            progressed = true;
          }
          if (jk < e.ntiles) {
            const int s = (T + jk) % kStages;
            const uint32_t ph = ((T + jk) / kStages) & 1;
            if (mbar_test(k_empty + s, ph ^ 1u)) {
              uint8_t* ks = smem + G::kOffK + s * G::kKBytes;
              if (rank == 0) mbar_arrive_expect_tx(k_full + s, 2 * G::kKBytes);
#pragma unroll
              for (int sl = 0; sl < G::kSlices; ++sl)
                tma_load_3d_pair(ks + sl * (kHalfN * 128), &tmK, bar_k + 8 * s, sl * 64, e.kh,
                                 e.p0 + jk * kBN + int(rank) * kHalfN, pol_kv);
              k_issued |= 1u << s;
              k_par = (k_par & ~(1u << s)) | (ph << s);
              ++jk;
              progressed = true;
            }
          }
          if (jv < jk) {
            const int s = (T + jv) % kStages;
            const uint32_t ph = ((T + jv) / kStages) & 1;
            if (mbar_test(v_empty + s, ph ^ 1u)) {
              uint8_t* vs = smem + G::kOffV + s * G::kVBytes;
              if (rank == 0) mbar_arrive_expect_tx(v_full + s, 2 * G::kVBytes);
#pragma unroll
              for (int sl = 0; sl < G::kVSlices; ++sl)
                tma_load_3d_pair(vs + sl * (kBN * 128), &tmV, bar_v + 8 * s,
                                 int(rank) * (DH / 2) + sl * 64, e.kh, e.p0 + jv * kBN, pol_kv);
              v_issued |= 1u << s;
              v_par = (v_par & ~(1u << s)) | (ph << s);
              ++jv;
              progressed = true;
            }
          }
          if (clk.expired(progressed, abort_flag, a.wait_ns)) {
            ok = false;
            break;
          }
        }
        T += e.ntiles;
        ++v;
      }
      if (!ok) {
        *abort_flag = 1;
        flag(a.status, JET_ERR_TIMEOUT);
        // let the copies in flight land: the even CTA's barriers count both
        // CTAs' bytes; the odd CTA waits out a fixed bounded time
        if (rank == 0) {
          if (q_issued) mbar_wait(q_full, q_par, kDrainNs, nullptr);
          for (int t = 0; t < kStages; ++t) {
            if (k_issued & (1u << t)) mbar_wait(k_full + t, (k_par >> t) & 1u, kDrainNs, nullptr);
            if (v_issued & (1u << t)) mbar_wait(v_full + t, (v_par >> t) & 1u, kDrainNs, nullptr);
          }
        } else if (q_issued | k_issued | v_issued) {
          const uint64_t t0 = global_timer_ns();
          while (global_timer_ns() - t0 < kDrainNs / 16) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (rank == 0 && elect_one()) {
      const uint32_t id_s = idesc_bf16_f32(2 * kBV, kBN);
      const uint32_t id_o = idesc_bf16_f32(2 * kBV, DH) | (1u << 16);  // B (V) is MN-major
      const uint32_t qs = smem_u32(smem);
      const uint64_t dq = desc_k_sw128(qs);
      // QK^T runs at most two tiles ahead of PV (the two S tiles), across items:
      // tq / tp tiles issued of each, vq / vp items begun, jq / jp tiles of them
      int tq = 0, tp = 0, vq = 0, vp = 0, jq = 0, jp = 0, nq = 0;
      int nt[2] = {0, 0}, kend[2] = {0, 0};  // tiles and keys of the items in the ring
      bool more = true, ok = true;
      IdleClock clk;
      while (ok && (more || tp < tq)) {
        bool progressed = false;
        if (more && tq - tp < 2) {
          bool ready = true;
          if (jq == 0 && nq == 0) {
            // the next item (the ring holds two: its slot's previous item is done)
            const int slot = vq & 1;
            if (vq - vp < 2 && mbar_test(item_full + slot, (vq >> 1) & 1)) {
              nq = ring[slot].ntiles;
              nt[slot] = nq;
              kend[slot] = ring[slot].k_end;
              mbar_arrive(item_empty + slot);
              if (nq == 0) more = false;
              progressed = true;
            }
            ready = nq > 0;
          }
          if (ready && jq == 0) ready = mbar_test(q_full, vq & 1);
          const int s = tq % kStages, b = tq & 1;
          if (ready && mbar_test(k_full + s, (tq / kStages) & 1)) {
            tc_fence_after();
            const uint64_t dk = desc_k_sw128(smem_u32(smem + G::kOffK + s * G::kKBytes));
#pragma unroll
            for (int st = 0; st < DH / 16; ++st) {
              const int sl = st >> 2, k = st & 3;
              mma_f16_pair(tmem + b * kBN, dq + (sl * (kBV * 128) >> 4) + 2 * k,
                           dk + (sl * (kHalfN * 128) >> 4) + 2 * k, id_s, st != 0);
            }
            mma_commit_pair(s_full + b, 0x3);
            mma_commit_pair(k_empty + s, 0x3);
            ++tq;
            if (++jq == nq) {
              mma_commit_pair(q_free, 0x3);  // the query blocks may be replaced
              ++vq;
              jq = nq = 0;
            }
            progressed = true;
          }
        }
        if (tp < tq) {
          const int s = tp % kStages, b = tp & 1, slot = vp & 1;
          // the item's first PV overwrites O: the previous item's O must be out
          if (mbar_test(p_full + b, (tp >> 1) & 1) && mbar_test(v_full + s, (tp / kStages) & 1) &&
              (jp > 0 || vp == 0 || mbar_test(o_free, (vp - 1) & 1))) {
            tc_fence_after();
            const uint32_t pt = tmem + b * kBN;  // P_j over the first columns of S_j
            const uint64_t dv =
                desc_mn_sw128(smem_u32(smem + G::kOffV + s * G::kVBytes), kBN * 128);
            // the keys past the block's last are not read (16 per instruction)
            const int steps = min(kBN, kend[slot] - jp * kBN + 15) >> 4;
#pragma unroll
            for (int k = 0; k < kBN / 16; ++k)
              if (k < steps)
                mma_f16_ta_pair(tmem + G::kOCol, pt + uint32_t(8 * k), dv + (k * 16 * 128 >> 4),
                                id_o, (jp | k) != 0);
            mma_commit_pair(v_empty + s, 0x3);
            ++tp;
            if (++jp == nt[slot]) {
              mma_commit_pair(o_full, 0x3);
              jp = 0;
              ++vp;
            }
            progressed = true;
          }
        }
        if (clk.expired(progressed, abort_flag, a.wait_ns)) ok = false;
      }
      if (!ok) {
        *abort_flag = 1;
        flag(a.status, JET_ERR_TIMEOUT);
        mma_commit_pair(drain, 0x1);
        mbar_wait(drain, 0, kDrainNs, nullptr);
      }
    }
  } else if (warp >= 3 && warp < 7) {
    // ---------------------------------------------------------------- softmax
    const int q4 = warp & 3;
    const int i = q4 * 32 + lane;  // query vector within the block = TMEM lane
    const uint32_t lane_off = uint32_t(q4 * 32) << 16;
    const uint32_t p_full_even = mapa_shared(p_full, 0);
    bool ok = true;
    int T = 0;
    for (int u = 0; ok; ++u) {
      const int slot = u & 1;
      if (!warp_mbar_wait(item_full + slot, (u >> 1) & 1, a.wait_ns, abort_flag)) {
        ok = false;
        break;
      }
      const int row0 = ring[slot].row0, ntiles = ring[slot].ntiles;
      __syncwarp();
      if (lane == 0) mbar_arrive(item_empty + slot);
      if (ntiles == 0) break;
      const int vis_end = row0 + i / g + 1;                // keys this vector sees
      const int vis_min = row0 + (q4 * 32) / g + 1;        // the warp's first vector's
      float m_used = -INFINITY, l = 0.f;
      for (int j = 0; j < ntiles; ++j) {
        const int Tj = T + j, b = Tj & 1;
        if (!warp_mbar_wait(s_full + b, (Tj >> 1) & 1, a.wait_ns, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t scol = tmem + lane_off + b * kBN;
        float sv[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld_32cols(scol + 32 * c, sv[c]);
        tmem_wait_ld();
        const int vis = vis_end - j * kBN;  // visible keys of this tile
        if (vis_min - j * kBN < kBN) {      // some vector of the warp does not see all 128
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int x = 0; x < 32; ++x)
              if (32 * c + x >= vis) sv[c][x] = -INFINITY;
        }
        float mq[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) mq[x] = fmaxf(sv[0][x], sv[1][x]);
#pragma unroll
        for (int x = 0; x < 8; ++x) mq[x] = fmaxf(fmaxf(mq[x], sv[2][x]), sv[3][x]);
#pragma unroll
        for (int x = 8; x < 32; ++x)
#pragma unroll
          for (int c = 0; c < 4; c += 2)
            mq[x & 7] = fmaxf(fmaxf(mq[x & 7], sv[c][x]), sv[c + 1][x]);
        const float mt = a.scale_log2 * fmaxf(fmaxf(fmaxf(mq[0], mq[1]), fmaxf(mq[2], mq[3])),
                                              fmaxf(fmaxf(mq[4], mq[5]), fmaxf(mq[6], mq[7])));
        const bool grow = mt > m_used + kRescaleLog2;
        if (__any_sync(0xffffffffu, grow)) {
          const float m_new = grow ? mt : m_used;
          if (j >= 1) {
            // O holds this item's PV so far: wait for the last one (its V stage
            // drained), rescale in TMEM
            const int Tp = Tj - 1;
            if (!warp_mbar_wait(v_empty + Tp % kStages, (Tp / kStages) & 1, a.wait_ns,
                                abort_flag)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const float f = grow ? ex2(m_used - m_new) : 1.f;
#pragma unroll 1
            for (int c0 = 0; c0 < DH; c0 += 16) {
              float ov[16];
              tmem_ld_16cols(tmem + lane_off + G::kOCol + c0, ov);
              tmem_wait_ld();
#pragma unroll
              for (int c = 0; c < 16; ++c) ov[c] *= f;
              tmem_st_16cols(tmem + lane_off + G::kOCol + c0, ov);
            }
            l *= f;
          }
          m_used = m_new;
        }
        // P = 2^(s scale - m_used) as bf16 pairs over this lane's S columns; the
        // row sum uses the rounded values, which are what the tensor core
        // multiplies
        const float mneg = -m_used;
        float ps[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) ps[x] = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float pw[16];
#pragma unroll
          for (int x = 0; x < 16; ++x) {
            const float x0 = ex2(fmaf(sv[c][2 * x], a.scale_log2, mneg));
            const float x1 = ex2(fmaf(sv[c][2 * x + 1], a.scale_log2, mneg));
            const uint32_t w = pack_bf16(x0, x1);
            pw[x] = __uint_as_float(w);
            ps[x & 7] += __uint_as_float(w << 16) + __uint_as_float(w & 0xffff0000u);
          }
          tmem_st_16cols(scol + 16 * c, pw);
        }
        l += ((ps[0] + ps[1]) + (ps[2] + ps[3])) + ((ps[4] + ps[5]) + (ps[6] + ps[7]));
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(p_full_even + 8u * b);
      }
      if (!ok) break;
      // the output warps have read what the item before last left there (with
      // one-tile items the softmax runs up to two items ahead of them)
      if (!warp_mbar_wait(l_free + slot, ((u >> 1) & 1) ^ 1u, a.wait_ns, abort_flag)) {
        ok = false;
        break;
      }
      linv[slot * kBV + i] = l > 0.f ? 1.f / l : 0.f;
      __syncwarp();
      if (lane == 0) mbar_arrive(l_full + slot);
      T += ntiles;
    }
    if (!ok) {
      *abort_flag = 1;
      flag(a.status, JET_ERR_TIMEOUT);
    }
  } else {
    // ---------------------------------------------------------------- output
    const int q4 = warp & 3;
    const int i = q4 * 32 + lane;
    const uint32_t lane_off = uint32_t(q4 * 32) << 16;
    const uint32_t o_free_even = mapa_shared(o_free, 0);
    // the output is transposed through this warp's 4 KB of the stage so that
    // every global store covers whole 128-byte pieces of one vector
    uint4* stage = reinterpret_cast<uint4*>(smem + G::kOffStage + q4 * 4096);
    bool ok = true;
    for (int u = 0; ok; ++u) {
      const int slot = u & 1;
      if (!warp_mbar_wait(item_full + slot, (u >> 1) & 1, a.wait_ns, abort_flag)) {
        ok = false;
        break;
      }
      const Item e = ring[slot];
      __syncwarp();
      if (lane == 0) mbar_arrive(item_empty + slot);
      if (e.ntiles == 0) break;
      // destinations of the vectors this lane stores (4 s + lane / 8, 16 bytes
      // each), as element offsets; -1 past the block's vectors
      long long dst[8];
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const int gi = q4 * 32 + 4 * s + (lane >> 3);
        dst[s] = gi < e.nv
                     ? (long long)(size_t(e.p0 + e.row0 + gi / g) * a.Hq + e.kh * g + gi % g) * DH
                     : -1;
      }
      if (!warp_mbar_wait(l_full + slot, (u >> 1) & 1, a.wait_ns, abort_flag) ||
          !warp_mbar_wait(o_full, u & 1, a.wait_ns, abort_flag)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const float inv = linv[slot * kBV + i];
      __syncwarp();
      if (lane == 0) mbar_arrive(l_free + slot);
      // all of O into registers as bf16, so that the next item's PV waits only
      // for these reads and not for the stores
      uint32_t pk[DH / 2];
#pragma unroll
      for (int c0 = 0; c0 < DH; c0 += 32) {
        float ov[32];
        tmem_ld_32cols(tmem + lane_off + G::kOCol + c0, ov);
        tmem_wait_ld();
#pragma unroll
        for (int x = 0; x < 16; ++x)
          pk[c0 / 2 + x] = pack_bf16(ov[2 * x] * inv, ov[2 * x + 1] * inv);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(o_free_even);
#pragma unroll
      for (int c0 = 0; c0 < DH; c0 += 64) {
#pragma unroll
        for (int x = 0; x < 8; ++x)
          stage[lane * 8 + (x ^ (lane & 7))] =
              make_uint4(pk[c0 / 2 + 4 * x], pk[c0 / 2 + 4 * x + 1], pk[c0 / 2 + 4 * x + 2],
                         pk[c0 / 2 + 4 * x + 3]);
        __syncwarp();
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const int iv = 4 * s + (lane >> 3), c = lane & 7;
          const uint4 val = stage[iv * 8 + (c ^ (iv & 7))];
          if (dst[s] >= 0) *reinterpret_cast<uint4*>(a.o + dst[s] + c0 + c * 8) = val;
        }
        __syncwarp();
      }
    }
    if (!ok) {
      *abort_flag = 1;
      flag(a.status, JET_ERR_TIMEOUT);
    }
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA leaves (or frees its TMEM) while the partner's MMAs, copies or
  // arrivals may still use its shared memory or TMEM
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, G::kTmemCols);
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

// packed [rows, heads, DH] bf16: box of 64 d x box_heads heads x box_rows rows
bool encode_3d(CUtensorMap* map, const void* base, int rows, int heads, int DH, int box_heads,
               int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {cuuint64_t(DH), cuuint64_t(heads), cuuint64_t(rows)};
  const cuuint64_t strides[2] = {cuuint64_t(DH) * 2, cuuint64_t(heads) * DH * 2};
  const cuuint32_t box[3] = {64, cuuint32_t(box_heads), cuuint32_t(box_rows)};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

template <int DH>
cudaError_t launch_prefill_pair(const jet_layout& lay, const jet_dims& d, const void* q,
                                const void* k, const void* v, void* o, int* status,
                                cudaStream_t st) {
  const jet_sizes& n = lay.n;
  const int g = d.Hq / d.Hkv;
  if (g > kBV) return cudaErrorInvalidValue;
  CUtensorMap tmQ, tmK, tmV;
  if (!encode_3d(&tmQ, q, n.total_prefix, d.Hq, DH, g, kBV / g) ||
      !encode_3d(&tmK, k, n.total_prefix, d.Hkv, DH, 1, kHalfN) ||
      !encode_3d(&tmV, v, n.total_prefix, d.Hkv, DH, 1, kBN))
    return cudaErrorInvalidValue;
  PreArgs a{};
  a.wait_ns = wait_budget_ns();
  a.hold_first = test_stall();
  a.prefix_offset = lay.prefix_offset;
  a.req_order = lay.req_order;
  a.o = static_cast<__nv_bfloat16*>(o);
  a.status = status;
  a.R = n.R;
  a.total = n.total_prefix;
  a.Hq = d.Hq;
  a.Hkv = d.Hkv;
  a.g = g;
  a.rb = kBV / g;
  a.scale_log2 = 1.4426950408889634f / sqrtf(float(DH));
  const size_t smem = Geo<DH>::kBytes + 1024;
  auto kern = prefill_pair_kernel<DH>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  const long long items =
      (long long)n.R * d.Hkv * ((n.max_prefix + 2 * a.rb - 1) / (2 * a.rb));
  // the static schedule deals the items to the pairs that are resident at once
  const int held = resident_pairs(reinterpret_cast<const void*>(kern), kThreads, smem);
  const int pairs = int(std::max<long long>(1, std::min<long long>(held, items)));
  return launch_pdl_pairs(kern, dim3(unsigned(2 * pairs)), dim3(kThreads), smem, st, tmQ, tmK,
                          tmV, a);
}

template cudaError_t launch_prefill_pair<128>(const jet_layout&, const jet_dims&, const void*,
                                              const void*, const void*, void*, int*, cudaStream_t);
template cudaError_t launch_prefill_pair<256>(const jet_layout&, const jet_dims&, const void*,
                                              const void*, const void*, void*, int*, cudaStream_t);

}  // namespace jet
