// hsga_moves.cuh -- migration moves worked out ahead of their generation.
//
// Which agent leaves an island, in which direction, and where immigrants land
// depend on the generation number alone, never on the population.  A launch
// that derives its own moves evaluates, for every island, the emigrant block
// of all four neighbours and the island's placement block, and searches for
// later arrivals on the same slot.  Instead generation G writes, beside its own
// work, the emigrants ("leave") of G + 2, one byte per island, and from the
// bytes that G - 1 wrote the moves of G + 1: per island and direction 16 bits,
// source slot, landing slot and whether the immigrant lands.  That is two
// blocks per island, 32 islands to a warp, where there were five lanes of a
// block per island, and generation G + 1 only gathers.  The first two
// generations of a call derive their own, and the last two plan no further.
// 16.8M agents in islands of 32 67.6 us per generation against 69.0 (groups of
// 8 with and without), tournament 5 on 500x500 62.7 against 64.6, untracked
// 55.2 against 59.8, 500x500 islands of 8 24.1 against 28.0.
#pragma once

#include "hsga_internal.h"
#include "hsga_island.cuh"

namespace hsga {

constexpr uint32_t kMoveLands = 0x8000u;  // | source slot << 6 | landing slot

// Moves and emigrants of the coming generations for islands 32 c .. 32 c + 31
// (a lane each).
template <int NN, class Keys>
__device__ __forceinline__ void plan_moves(const RunParams &p, const Keys &keys, const Moves &mv,
                                           uint32_t c, uint32_t G) {
  const uint32_t isl = 32u * c + (threadIdx.x & 31u);
  if (isl >= p.islands) return;
  uint32_t from[4] = {0u, 0u, 0u, 0u};
  if (mv.next) {
#pragma unroll
    for (uint32_t d = 0; d < 4; ++d) from[d] = mv.leave_next[neighbour(p, isl, d)];
  }
  if (mv.leave_after) {
    const Words4 m = philox_keys(keys, kSlotEmigrant, isl, G + 2u, kPurposeMigration);
    mv.leave_after[isl] = (uint8_t)((m.y >> 30) << 6 | uindex_nn<NN>(m.x, p.n));
  }
  if (mv.next) {
    const Words4 v = philox_keys(keys, kSlotImmigrant, isl, G + 1u, kPurposeMigration);
    const uint32_t to[4] = {uindex_nn<NN>(v.x, p.n), uindex_nn<NN>(v.y, p.n),
                            uindex_nn<NN>(v.z, p.n), uindex_nn<NN>(v.w, p.n)};
    uint32_t m[4];
#pragma unroll
    for (uint32_t d = 0; d < 4; ++d) {
      bool lands = (from[d] >> 6) == (d ^ 2u);
      m[d] = (from[d] & 63u) << 6 | to[d];
#pragma unroll
      for (uint32_t e = d + 1u; e < 4; ++e)  // the latest of N, E, S, W wins a shared slot
        lands = lands && !((from[e] >> 6) == (e ^ 2u) && to[e] == to[d]);
      m[d] |= lands ? kMoveLands : 0u;
    }
    reinterpret_cast<uint2 *>(mv.next)[isl] = make_uint2(m[0] | m[1] << 16, m[2] | m[3] << 16);
  }
}

// The lane's move in a group of islands from isl0 on: island lane / 4,
// direction lane % 4 (0: none), of the first cnt islands.
__device__ __forceinline__ uint32_t load_move(const Moves &mv, uint32_t isl0, uint32_t cnt) {
  const uint32_t lane = threadIdx.x & 31u;
  return lane < 4u * cnt ? (uint32_t)mv.now[(size_t)isl0 * 4u + lane] : 0u;
}

// Spreads a launch's planning over its warps' visits to groups of islands, so
// that it fills the time that they wait for memory: 32 islands are planned
// for every 32 that the warp has advanced.
struct Planner {
  uint32_t chunk, chunks, stride, credit;
  __device__ __forceinline__ Planner(const RunParams &p, const Moves &mv, uint32_t warp,
                                     uint32_t nwarps)
      : chunk(nwarps - 1u - warp),  // the last warps have the fewest groups
        chunks(mv.next || mv.leave_after ? (p.islands + 31u) / 32u : 0u),
        stride(nwarps),
        credit((warp & 7u) * 4u) {}
  template <int NN, class Keys>
  __device__ __forceinline__ void visit(const RunParams &p, const Keys &keys, const Moves &mv,
                                        uint32_t G, uint32_t islands) {
    credit += islands;
    if (credit < 32u) return;
    credit -= 32u;
    one<NN>(p, keys, mv, G);
  }
  template <int NN, class Keys>
  __device__ __forceinline__ void rest(const RunParams &p, const Keys &keys, const Moves &mv,
                                       uint32_t G) {
    while (chunk < chunks) one<NN>(p, keys, mv, G);
  }
  template <int NN, class Keys>
  __device__ __forceinline__ void one(const RunParams &p, const Keys &keys, const Moves &mv,
                                      uint32_t G) {
    if (chunk < chunks) {
      plan_moves<NN>(p, keys, mv, chunk, G);
      chunk += stride;
    }
  }
};

}  // namespace hsga
