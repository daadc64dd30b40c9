// hsga_flat.cuh -- one synchronous generation of a group of up to eight
// consecutive islands by one warp, for any island size, fitness model and
// surface width: the streamed kernel of everything but 32-agent integer islands
// (hsga_flat.cu) and the batch engine's tick (hsga_batch.cu).
//
// The group's parents, one contiguous run of each island-major plane, are
// staged in shared memory by a bulk asynchronous copy, and its children are
// numbered flat over the lanes: 8 n children fill 8 n / 32 rounds whatever n
// is, where a lane per agent leaves 16 of 64 lanes idle at n = 48 and 15 of
// 32 at n = 17.  Migration takes two Philox evaluations of the warp: lane i <
// 8 the placement slots of island i, then lane 4i + d the emigrant of island
// i's neighbour in direction d, gathered from the parent planes when it is
// aimed here.  The gather and the copy are in flight while the first
// children's draws are evaluated; children are written once all of a round's
// reads are done, with coalesced streaming stores.
//
// us per generation, here and on the kernels before it (a lane per agent in
// registers; for binary32 fitness and wide surfaces a warp per island after
// two migration launches): 128x256 islands of 48 8.0 (18.5), of 17 4.5
// (10.3), of 64 with tournament 5 18.8 (43.0); 500x500 of 32, tournament 5,
// binary32 89.7 (110); 256x512 of 32 with four surface words 46.1 (66.2), of
// which 44.5 are its 72 bytes per agent at the measured copy bandwidth; 20x20
// of 32, binary32 2.5 (14.4).
//
// Children in flight against warps per SM, us: integer, tournament 2: three
// children and 20-28 warps (128x256x48 takes a fifth longer with four, a tenth
// with two and 32 warps).  Larger tournaments hold more blocks at once: 64 agents,
// tournament 5, three children and 16 warps 19.3, 20 warps 21.4, 24 22.7, two
// children and 28 warps 20.2.  binary32: four and 16 warps 89.7, three and 16
// 91.2, 20 94.6, two and 32 96.4, four and 12 97.3.  Two surface words: two
// children 25.5, three 27.4.  (Closing the mutating children up over the lanes
// before their amounts are drawn: 89.2, but 3.3 on 20x20; generator heads for
// the second tournament block as well: 64 agents 21.9 for 21.4.)
//
// Bound by issue, but for four words: 113 warp instructions per 32 children at
// n = 48, 51 of them on the ALU pipe (two cycles each); binary32 274, 129 on
// the ALU and 85 on the multiplier pipe, which binds three blocks a child.
#pragma once

#include "hsga_moves.cuh"
#include "hsga_stage.cuh"

namespace hsga {

constexpr uint32_t kFlatGroup = 8;    // most islands per warp visit
// Children per lane in flight.
template <int K, bool T2, bool FLT>
constexpr uint32_t kFlatUnroll = FLT ? 4 : T2 && K >= 2 ? 2 : 3;
constexpr int kFlatThreads = 128;
constexpr uint32_t kFlatWarps = kFlatThreads / 32;

// Bytes of one warp's stage: K-word surfaces, traits, the generator heads of
// the slots, the group's island products, placement slots.
__host__ __device__ __forceinline__ uint32_t flat_stage_bytes(uint32_t n, uint32_t words) {
  return kFlatGroup * n * (4u + 8u * words) + 16u * n + 8u * kFlatGroup + 4u * kFlatGroup;
}

// A single run's parameters stay in the kernel's parameter space; a batch
// run's round keys are copied from its descriptor into registers.
struct RoundKeys {
  uint32_t rk0[10], rk1[10];
};

// What a generation writes into K-word surfaces, per 32-bit half as in
// Deposit: half = (half & clear) | ((value << shift) & ~clear).
template <int K>
struct FlatDeposit {
  uint32_t clear[K > 0 ? 2 * K : 1], clear2[K > 0 ? 2 * K : 1];
  uint32_t shift, shift2, two;
};

template <int K>
__host__ __device__ __forceinline__ FlatDeposit<K> flat_deposit(const RunParams &p, uint32_t G) {
  FlatDeposit<K> f{};
  if constexpr (K == 1) {
    const Deposit d = deposit_for(p, G);
    f.clear[0] = d.clear_lo;
    f.clear[1] = d.clear_hi;
    f.clear2[0] = d.clear2_lo;
    f.clear2[1] = d.clear2_hi;
    f.shift = d.shift;
    f.shift2 = d.shift2;
    f.two = d.two;
  }
  if constexpr (K > 1) {
#ifndef __CUDA_ARCH__
    const WideDeposit d = wide_deposit_for(p, G);
    for (int h = 0; h < 2 * K; ++h) f.clear[h] = f.clear2[h] = 0xFFFFFFFFu;
    if (d.word1 >= 0) f.clear[2 * d.word1 + d.shift1 / 32] = ~((uint32_t)p.vmask << (d.shift1 % 32));
    if (d.word2 >= 0) f.clear2[2 * d.word2 + d.shift2 / 32] = ~((uint32_t)p.vmask << (d.shift2 % 32));
    f.shift = d.shift1 % 32;
    f.shift2 = d.shift2 % 32;
    f.two = d.word2 >= 0 ? 1u : 0u;
#endif
  }
  return f;
}

template <int K>
__device__ __forceinline__ void flat_put(const FlatDeposit<K> &d, uint64_t (&s)[K > 0 ? K : 1],
                                         uint32_t value) {
  const uint32_t v = value << d.shift;
#pragma unroll
  for (int w = 0; w < K; ++w) {
    uint32_t lo = (uint32_t)s[w], hi = (uint32_t)(s[w] >> 32);
    lo = (lo & d.clear[2 * w]) | (v & ~d.clear[2 * w]);
    hi = (hi & d.clear[2 * w + 1]) | (v & ~d.clear[2 * w + 1]);
    if (d.two) {
      const uint32_t v2 = (value >> 16) << d.shift2;
      lo = (lo & d.clear2[2 * w]) | (v2 & ~d.clear2[2 * w]);
      hi = (hi & d.clear2[2 * w + 1]) | (v2 & ~d.clear2[2 * w + 1]);
    }
    s[w] = ((uint64_t)hi << 32) | lo;
  }
}

template <uint32_t N>
struct Count {
  static constexpr uint32_t value = N;
};

// One warp's stage and the state of its barrier.  head[j] holds what the first
// three rounds of child slot j's block need that does not depend on the island
// (LaneHead b2, l1, l2, l3), isl[i] the product of rounds 1-2 that depends on
// the island alone: two shared-memory reads replace 5 of a block's 20 wide
// multiplies.
struct FlatStage {
  uint64_t *surf;
  uint32_t *trait, *plan;
  uint4 *head;
  uint2 *isl;
  uint64_t *bar;
  uint32_t phase;
  uint32_t x0;  // word 0 after round 1, before the island
};

__device__ __forceinline__ FlatStage flat_stage(unsigned char *base, uint64_t *bar, uint32_t n,
                                                uint32_t words) {
  FlatStage s;
  s.surf = (uint64_t *)base;
  s.trait = (uint32_t *)(base + 8u * words * kFlatGroup * n);
  s.head = (uint4 *)(s.trait + kFlatGroup * n);
  s.isl = (uint2 *)(s.head + n);
  s.plan = (uint32_t *)(s.isl + kFlatGroup);
  s.bar = bar;
  s.phase = 0;
  s.x0 = 0;
  return s;
}

// Generator heads of generation G for a warp's stage (a warp barrier must
// follow before they are used).
template <class Keys>
__device__ __forceinline__ void flat_heads(const Keys &keys, uint32_t n, uint32_t G,
                                           FlatStage &st) {
  for (uint32_t j = threadIdx.x & 31u; j < n; j += 32u) {
    const LaneHead h = lane_head(keys, j, G, kPurposeReplicate);
    st.head[j] = make_uint4(h.b2, h.l1, h.l2, h.l3);
  }
  st.x0 = (uint32_t)(((uint64_t)G * kPhiloxM1) >> 32) ^ keys.rk0[0];
}

// Children that the next generation finds in L2 (StreamPlan::back) are stored
// as any other data (four words 46.2 against 47.9 us), others as data not read
// again soon.
template <bool KEEP, class T>
__device__ __forceinline__ void flat_store(T *at, T value) {
  if constexpr (KEEP) *at = value;
  else __stcs(at, value);
}

// Advances `group` (<= kFlatGroup) islands from isl0 on (fewer at the end of the
// grid) from the parent planes to the child planes.  K: surface words (0: no surface).  NN:
// island size when known (32), else 0.  T2: the tournament size is exactly 2.
// FLT: binary32 fitness.  planned: `move` is the lane's
// migration move (0: none).  first: wait for the launch
// before this one once the draws are done.  bulk: the planes allow 16-byte bulk
// copies.
// Returns false (on every lane) when the copy did not arrive in time.
template <int K, bool T2, int NN, bool FLT, bool KEEP = false, class Keys>
__device__ __forceinline__ bool flat_group(const RunParams &p, const Keys &keys,
                                           const FlatDeposit<K> &dep, bool migrate, bool bulk,
                                           uint32_t isl0, uint32_t group, uint32_t G,
                                           bool planned, uint32_t move, bool first,
                                           const uint32_t *__restrict__ tin,
                                           const uint64_t *__restrict__ sin,
                                           uint32_t *__restrict__ tout,
                                           uint64_t *__restrict__ sout, FlatStage &st) {
  constexpr int KS = K > 0 ? K : 1;
  constexpr uint32_t U0 = kFlatUnroll<K, T2, FLT>;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t n = NN ? (uint32_t)NN : p.n;
  const uint32_t cnt = min(group, p.islands - isl0), total = cnt * n;
  const size_t base = (size_t)isl0 * n;
  const auto island_of = [&](uint32_t c) {  // child number -> island of the group
    if constexpr (NN == 32) return c >> 5;
    else return (c * p.n_recip) >> 16;  // exact for c < kFlatGroup n, n <= 64
  };
  // stages the parents (the previous group's reads are behind a warp barrier)
  const bool copy = bulk && ((total | (uint32_t)base) & 3u) == 0u;  // whole 16-byte pieces
  const auto stage = [&] {
    if (copy) {
      if (lane == 0) {
        proxy_fence();
        mbar_expect_tx(st.bar, total * (4u + 8u * K));
        bulk_load(st.trait, tin + base, 4u * total, st.bar);
        if constexpr (K > 0) bulk_load(st.surf, sin + base * K, 8u * K * total, st.bar);
      }
    } else {
      for (uint32_t c = lane; c < total; c += 32u) st.trait[c] = __ldcs(tin + base + c);
      if constexpr (K > 0)
        for (uint32_t c = lane; c < total * K; c += 32u) st.surf[c] = __ldcs(sin + base * K + c);
    }
  };
  if (!first) stage();
  // a1, a2: draws, and the gather of the emigrants aimed at this group
  uint32_t it = 0, src = 0, src_slot = 0;
  uint64_t is[KS];
#pragma unroll
  for (int w = 0; w < KS; ++w) is[w] = 0;
  bool arrive = false;
  const auto gather = [&] {
    const size_t a = (size_t)src * n + src_slot;
    it = __ldg(tin + a);
    if constexpr (K > 0) {
#pragma unroll
      for (int w = 0; w < KS; ++w) is[w] = __ldg(sin + a * K + w);
    }
  };
  if (planned) {
    if (move & kMoveLands) {
      src = neighbour(p, isl0 + (lane >> 2), lane & 3u);
      src_slot = move >> 6 & 63u;
      gather();
    }
  } else if (migrate) {
    if (lane < cnt) {
      const Words4 v = philox_keys(keys, kSlotImmigrant, isl0 + lane, G, kPurposeMigration);
      st.plan[lane] = uindex_nn<NN>(v.x, n) | (uindex_nn<NN>(v.y, n) << 8) |
                      (uindex_nn<NN>(v.z, n) << 16) | (uindex_nn<NN>(v.w, n) << 24);
    }
    const uint32_t d = lane & 3u;
    const bool valid = (lane >> 2) < cnt;
    src = neighbour(p, valid ? isl0 + (lane >> 2) : isl0, d);
    const Words4 m = philox_keys(keys, kSlotEmigrant, src, G, kPurposeMigration);
    arrive = valid && (m.y >> 30) == (d ^ 2u);
    src_slot = uindex_nn<NN>(m.x, n);
    if (arrive && !first) gather();
  }
  if (lane < kFlatGroup) {
    const uint64_t u = (uint64_t)(st.x0 ^ (isl0 + lane)) * kPhiloxM0;
    st.isl[lane] = make_uint2((uint32_t)u, (uint32_t)(u >> 32));
  }
  __syncwarp();
  // replication draws of children c0 + 32 u + lane, the last child's beyond the end
  const auto draw = [&](uint32_t c0, uint32_t u, uint32_t &isl, uint32_t &slot) {
    const uint32_t c = min(c0 + 32u * u + lane, total - 1u);
    isl = island_of(c);
    slot = c - isl * n;
    const uint4 h = st.head[slot];
    const uint2 x = st.isl[isl];
    const uint64_t v = (uint64_t)(x.y ^ h.x) * kPhiloxM1;
    uint32_t a0 = (uint32_t)(v >> 32) ^ h.y, a1 = (uint32_t)v, a2 = x.x ^ h.z, a3 = h.w;
#pragma unroll
    for (int r = 3; r < 10; ++r) {
      const uint64_t p0 = (uint64_t)a0 * kPhiloxM0;
      const uint64_t p1 = (uint64_t)a2 * kPhiloxM1;
      const uint32_t n0 = (uint32_t)(p1 >> 32) ^ a1 ^ keys.rk0[r];
      const uint32_t n2 = (uint32_t)(p0 >> 32) ^ a3 ^ keys.rk1[r];
      a0 = n0;
      a1 = (uint32_t)p1;
      a2 = n2;
      a3 = (uint32_t)p0;
    }
    return Words4{a0, a1, a2, a3};
  };
  // the first round's draws, while the copy and the gather are in flight
  uint32_t isl_first[U0], slot_first[U0];
  Words4 w_first[U0];
  const bool early = total > 32u * (U0 - 1u);
  if (early) {
#pragma unroll
    for (uint32_t u = 0; u < U0; ++u) w_first[u] = draw(0, u, isl_first[u], slot_first[u]);
  }
  if (first) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    stage();
    if (arrive) gather();
  }
  if (copy) {
    if (!__all_sync(kFull, mbar_wait(st.bar, st.phase))) return false;
    st.phase ^= 1u;
  }
  __syncwarp();
  if (planned || migrate) {
    const uint32_t d = lane & 3u;
    uint32_t at = (move & kMoveLands) ? (lane >> 2) * n + (move & 63u) : kNoArrival;
    const uint32_t bits = (__ballot_sync(kFull, arrive) >> (lane & 28u)) & 0xFu;
    if (arrive) {
      const uint32_t pl = st.plan[lane >> 2];
      const uint32_t sl = (pl >> (8u * d)) & 0xFFu;
      bool last = true;  // no later direction lands on the same slot
#pragma unroll
      for (uint32_t e = 1; e < 4; ++e)
        if (e > d && (bits >> e & 1u) && ((pl >> (8u * e)) & 0xFFu) == sl) last = false;
      if (last) at = (lane >> 2) * n + sl;
    }
    if (at != kNoArrival) {
      st.trait[at] = it;
      if constexpr (K > 0) {
#pragma unroll
        for (int w2 = 0; w2 < KS; ++w2) st.surf[at * K + w2] = is[w2];
      }
    }
    __syncwarp();
  }
  // a3-a6 of children c0 + 32 u + lane, u < U
  uint32_t *const tlane = tout + base + lane;
  uint64_t *const slane = K > 0 ? sout + (base + lane) * K : sout;
  const bool del = p.has_del != 0u;
  const auto children = [&](auto count, uint32_t c0, const uint32_t (&isl)[decltype(count)::value],
                            const uint32_t (&slot)[decltype(count)::value],
                            const Words4 (&w)[decltype(count)::value]) {
    constexpr uint32_t U = decltype(count)::value;
    uint32_t best[U], fbest[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      best[u] = isl[u] * n + uindex_nn<NN>(w[u].x, n);
      fbest[u] = st.trait[best[u]];
    }
    if (T2 || p.tournament >= 2u) {
      uint32_t c[U], fc[U];
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) {
        c[u] = isl[u] * n + uindex_nn<NN>(w[u].y, n);
        fc[u] = st.trait[c[u]];
      }
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) {
        const bool take = fitter<FLT>(fc[u], fbest[u]);
        best[u] = take ? c[u] : best[u];
        fbest[u] = take ? fc[u] : fbest[u];
      }
    }
    if constexpr (!T2) {
      for (uint32_t t0 = 2; t0 < p.tournament; t0 += 4) {
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
          const Words4 e = philox_keys(keys, slot[u], isl0 + isl[u], G,
                                       kPurposeReplicate + 1 + (t0 - 2) / 4);
          const uint32_t ew[4] = {e.x, e.y, e.z, e.w};
          uint32_t c[4], fc[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            c[q] = isl[u] * n + uindex_nn<NN>(ew[q], n);
            fc[q] = st.trait[c[q]];
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const bool take = t0 + q < p.tournament && fitter<FLT>(fc[q], fbest[u]);
            best[u] = take ? c[q] : best[u];
            fbest[u] = take ? fc[q] : fbest[u];
          }
        }
      }
    }
    [[maybe_unused]] uint64_t cs[U][KS];
    if constexpr (K > 0) {
#pragma unroll
      for (uint32_t u = 0; u < U; ++u)
#pragma unroll
        for (int q = 0; q < KS; ++q) cs[u][q] = st.surf[best[u] * K + q];
    }
    uint32_t ct[U];
    if constexpr (FLT) {
      // amounts for all of the round's children at once if any of them mutates
      // (independent chains; a branch per child would run them one by one)
      bool any = false;
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) any = any || mutates_float(p, w[u].z);
      float amount[U];
      if (__any_sync(kFull, any)) {
#pragma unroll
        for (uint32_t u = 0; u < U; ++u)
          amount[u] = gauss_amount(
              p, philox_keys(keys, slot[u], isl0 + isl[u], G, kPurposeGauss));
      } else {
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) amount[u] = 0.0f;
      }
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) ct[u] = apply_float(p, fbest[u], w[u].z, amount[u]);
    }
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      if constexpr (!FLT)
        ct[u] = del ? mutate(p, fbest[u], w[u].z) : mutate<false>(p, fbest[u], w[u].z);
      if constexpr (K > 0) flat_put<K>(dep, cs[u], w[u].w);
    }
    uint32_t *const to = tlane + c0;
    [[maybe_unused]] uint64_t *const so = slane + (size_t)c0 * K;
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      if (c0 + 32u * u + lane < total) {
        flat_store<KEEP>(to + 32u * u, ct[u]);
        if constexpr (K == 1) flat_store<KEEP>(so + 32u * u, cs[u][0]);
        if constexpr (K == 2 || K == 4) {
          uint64_t *const o = so + 32u * u * K;
          if (bulk) {  // 16-byte aligned planes
#pragma unroll
            for (int q = 0; q < KS; q += 2)
              flat_store<KEEP>((ulonglong2 *)(o + q), make_ulonglong2(cs[u][q], cs[u][q + 1]));
          } else {
#pragma unroll
            for (int q = 0; q < KS; ++q) flat_store<KEEP>(o + q, cs[u][q]);
          }
        }
      }
    }
  };
  const auto round = [&](auto count, uint32_t c0) {
    constexpr uint32_t U = decltype(count)::value;
    uint32_t isl[U], slot[U];
    Words4 w[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) w[u] = draw(c0, u, isl[u], slot[u]);
    children(count, c0, isl, slot, w);
  };
  uint32_t c0 = 0;
  if (early) {
    children(Count<U0>{}, 0u, isl_first, slot_first, w_first);
    c0 = 32u * U0;
  }
  // full rounds, then the remainder (at most three) in smaller ones: no lane works beyond the last
  // 32 children (a fixed unroll wastes 2 of 8 rounds at n = 24)
  for (; total > c0 + 32u * (U0 - 1u); c0 += 32u * U0)
    round(Count<U0>{}, c0);
  if (total > c0 + 32u) {
    round(Count<2>{}, c0);
    c0 += 64u;
  }
  if (total > c0) round(Count<1>{}, c0);
  __syncwarp();  // every lane is done with the stage before it is refilled
  return true;
}

}  // namespace hsga
