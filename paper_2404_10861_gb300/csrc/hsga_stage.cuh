// hsga_stage.cuh -- staging of island groups in shared memory by bulk
// asynchronous copies: the barrier and copy primitives, also the flat kernel's
// (hsga_flat.cuh), and the parts of the staged generation kernel
// (hsga_staged.cu).
//
// A warp of it owns a ring of up to kStagedStages stages; a stage holds one group of
// eight (or four) 32-agent islands: 1,024 bytes of traits, then 2,048 bytes of
// surfaces, each contiguous in the island-major planes, copied by one lane with
// cp.async.bulk and completing on the stage's mbarrier.
#pragma once

#include <cuda_runtime.h>

#include "hsga_internal.h"
#include "hsga_island.cuh"
#include "hsga_moves.cuh"
#include "hsga_sync.cuh"

namespace hsga {

constexpr uint32_t kStagedWarps = kStagedThreads / 32;
// Islands per stage: eight; four on grids that so take one round of groups.
constexpr uint32_t kStageGroup = 8, kSmallStageGroup = 4;
template <uint32_t GR>
constexpr uint32_t kTraitBytes = GR * 32 * 4;
template <uint32_t GR>
constexpr uint32_t kSurfBytes = GR * 32 * 8;
constexpr uint32_t kMaxPolls = 1u << 24;

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}

// Makes the barrier initialisation visible to the asynchronous proxy.
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Orders this thread's earlier shared-memory accesses (and, after a warp
// barrier, its warp's) before later bulk copies into the same memory.
__device__ __forceinline__ void proxy_fence() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}

// Global -> shared bulk copy (16-byte aligned addresses, size a multiple of
// 16) that completes `bytes` of the barrier's transaction count.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for the phase of `parity` to complete.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
  if (mbar_test(bar, parity)) return true;
  const uint64_t t0 = now_ns();
  for (uint32_t i = 1; i < kMaxPolls; ++i) {
    if (mbar_test(bar, parity)) return true;
    if ((i & 63u) == 0 && now_ns() - t0 > kWaitNs) return false;
  }
  return false;
}

// A lane's immigrant to a staged group of GR islands, lane 4i + d the one of
// island i from direction d: the agent of the group that it overwrites (none:
// kNoArrival) and its genome.
constexpr uint32_t kNoArrival = 0xFFFFFFFFu;
struct Arrival {
  uint32_t at, it;
  uint64_t is;
};

// The lane's move (hsga_moves.cuh; 0: none) derived here.
template <uint32_t GR>
__device__ __forceinline__ uint32_t derive_move(const RunParams &p, uint32_t isl0, uint32_t G) {
  const uint32_t lane = threadIdx.x & 31u, d = lane & 3u, i = min(lane >> 2, GR - 1u);
  const Words4 v =
      philox_rk(p, kSlotImmigrant, isl0 + min(lane, GR - 1u), G, kPurposeMigration);
  const uint32_t plan =
      v.x >> 27 | (v.y >> 27) << 8 | (v.z >> 27) << 16 | (v.w >> 27) << 24;
  const Words4 m =
      philox_rk(p, kSlotEmigrant, neighbour(p, isl0 + i, d), G, kPurposeMigration);
  const bool arrive = lane < 4u * GR && (m.y >> 30) == (d ^ 2u);
  const uint32_t to = __shfl_sync(kFull, plan, i);
  const uint32_t bits = (__ballot_sync(kFull, arrive) >> (lane & 28u)) & 0xFu;
  const uint32_t slot = (to >> (8u * d)) & 0xFFu;
  bool lands = arrive;
#pragma unroll
  for (uint32_t e = 1; e < 4; ++e)  // the latest of N, E, S, W wins a shared slot
    lands = lands && !(e > d && (bits >> e & 1u) && ((to >> (8u * e)) & 0xFFu) == slot);
  return lands ? kMoveLands | (m.x >> 27) << 6 | slot : 0u;
}

// The immigrant of the lane's move.
template <bool TRACKED>
__device__ __forceinline__ Arrival arrival_of(const RunParams &p, uint32_t move, uint32_t isl0,
                                              const uint32_t *__restrict__ tin,
                                              const uint64_t *__restrict__ sin) {
  const uint32_t lane = threadIdx.x & 31u, i = lane >> 2;
  Arrival r{kNoArrival, 0u, 0ull};
  if (move & kMoveLands) {
    const uint32_t x = neighbour(p, isl0 + i, lane & 3u) * 32u + (move >> 6 & 31u);
    r.at = 32u * i + (move & 31u);
    r.it = __ldg(tin + x);
    if constexpr (TRACKED) r.is = __ldg(sin + x);
  }
  return r;
}

// a3-a6 of child `lane` of every island of a staged group (parents of island
// i at tr + 32 i, sr + 32 i), stored to to + 32 i, so + 32 i.  All of the
// group's reads come before its first store: the stores order memory for the
// compiler, which would otherwise finish one island before it reads the next.
template <bool TRACKED, bool T2, bool TWO, bool DEL, uint32_t GR, class More>
__device__ __forceinline__ void replicate_group(const RunParams &p, const Deposit &dep,
                                                const Words4 (&w)[GR], const uint32_t *tr,
                                                const uint64_t *sr, uint32_t *to, uint64_t *so,
                                                const More &more) {
  uint32_t best[GR], fbest[GR];
  uint64_t cs[GR];
#pragma unroll
  for (uint32_t i = 0; i < GR; ++i) {
    best[i] = w[i].x >> 27;
    fbest[i] = tr[32u * i + best[i]];
  }
  if (T2 || p.tournament >= 2) {
    uint32_t fc[GR];
#pragma unroll
    for (uint32_t i = 0; i < GR; ++i) fc[i] = tr[32u * i + (w[i].y >> 27)];
#pragma unroll
    for (uint32_t i = 0; i < GR; ++i) {
      best[i] = fc[i] > fbest[i] ? w[i].y >> 27 : best[i];
      fbest[i] = max(fc[i], fbest[i]);
    }
  }
  if constexpr (!T2) {
    for (uint32_t c0 = 2; c0 < p.tournament; c0 += 4) {
#pragma unroll
      for (uint32_t i = 0; i < GR; ++i) {
        const Words4 e = more(i, (c0 - 2) / 4);
        const uint32_t ew[4] = {e.x >> 27, e.y >> 27, e.z >> 27, e.w >> 27};
        uint32_t fc[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) fc[r] = tr[32u * i + ew[r]];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const bool take = c0 + r < p.tournament && fc[r] > fbest[i];
          best[i] = take ? ew[r] : best[i];
          fbest[i] = take ? fc[r] : fbest[i];
        }
      }
    }
  }
  if constexpr (TRACKED) {
#pragma unroll
    for (uint32_t i = 0; i < GR; ++i) cs[i] = sr[32u * i + best[i]];
  }
#pragma unroll
  for (uint32_t i = 0; i < GR; ++i) {
    __stcs(to + 32u * i, mutate<DEL>(p, fbest[i], w[i].z));
    if constexpr (TRACKED) __stcs(so + 32u * i, deposit_into<TWO>(dep, cs[i], w[i].w));
  }
}

// a2-a6 of one 32-agent island in registers (lane = agent).
template <bool TRACKED, bool T2, bool MIG>
__device__ __noinline__ void single_island(const RunParams &p, const Deposit &dep, uint32_t G,
                                           uint32_t isl, const uint32_t *__restrict__ tin,
                                           const uint64_t *__restrict__ sin,
                                           uint32_t *__restrict__ tout,
                                           uint64_t *__restrict__ sout) {
  const size_t a = (size_t)isl * 32u + (threadIdx.x & 31u);
  uint32_t pt[1] = {__ldcs(tin + a)}, ct[1];
  uint64_t ps[1] = {0}, cs[1];
  if constexpr (TRACKED) ps[0] = __ldcs(sin + a);
  Words4 w[1];
  replication_words<1>(p, isl, G, w);
  if constexpr (MIG) {
    const Arrival in = arrival_of<TRACKED>(p, derive_move<1>(p, isl, G), isl, tin, sin);
    const uint32_t landing = __ballot_sync(kFull, in.at != kNoArrival);
#pragma unroll
    for (uint32_t d = 0; d < 4; ++d)
      if (landing >> d & 1u)
        land<1, TRACKED>(__shfl_sync(kFull, in.at, d), d, in.it, in.is, pt, ps);
  }
  if (dep.two) replicate<1, TRACKED, T2, true>(p, dep, isl, G, w, pt, ps, ct, cs);
  else replicate<1, TRACKED, T2, false>(p, dep, isl, G, w, pt, ps, ct, cs);
  __stcs(tout + a, ct[0]);
  if constexpr (TRACKED) __stcs(sout + a, cs[0]);
}

template <uint32_t GR>
constexpr uint32_t kStageBytes = kTraitBytes<GR> + kSurfBytes<GR>;
template <uint32_t GR>
constexpr size_t kRingBytes = (size_t)kStagedWarps * kStagedStages * kStageBytes<GR>;
template <uint32_t GR>
constexpr int kStagedBlocks = GR == kStageGroup ? kStagedBlocksPerSM : kSmallStagedBlocksPerSM;

// Shared memory requested per block: the ring, padded so that one block
// more than kStagedBlocks does not fit on an SM.  Otherwise the next
// generation's launch, scheduled early by programmatic dependent launch,
// parks a block in the free slot that competes with the running blocks for
// issue slots until it may start (107 us per generation at 16.8M agents
// with a free slot, 75.3 us without).
template <uint32_t GR>
size_t staged_smem_bytes() {
  static size_t bytes = 0;
  if (bytes == 0) {
    int dev = 0, per_sm = 0, per_block = 0, reserved = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    size_t pad = (size_t)per_sm / (kStagedBlocks<GR> + 1) + 128;
    pad = pad > (size_t)reserved ? pad - (size_t)reserved : pad;
    size_t b = kRingBytes<GR> > pad ? kRingBytes<GR> : pad;
    if (per_block > 0 && b > (size_t)per_block - 1024) b = kRingBytes<GR>;  // no room to pad
    bytes = (b + 127) & ~(size_t)127;
  }
  return bytes;
}

}  // namespace hsga
