// hsga_resident_warp.cu -- many synchronous generations per launch for small
// grids whose islands are not 32 agents: one island per warp with its genomes
// in registers (lane = agent, AP agents per lane).
//
// A few islands run in one block, with a block barrier per migration.  More are
// cut into tiles of four to a block: neighbours inside a tile exchange emigrants
// through shared memory after one block barrier per migration, and only tile
// edges publish records in global memory (four 64-bit words, each stamped with
// the migration's number), which neighbouring tiles poll.  Latency bounds such a
// grid, and this kernel has less of it than groups of islands per warp on a tile
// per SM (hsga_resident.cu): us per generation 15x15 islands of 22 1.30 against
// 1.82, 8x19 of 27 with a tournament of 5 1.43 against 2.15, 64x64 of 17 1.70
// against 1.92; 64x64 of 48 2.34 against 2.25.
//
// Waits are bounded (kWaitNs, kMaxSpins); a warp whose wait gave up reaches the
// block's next barrier, whose reduction makes the block leave together.
#include <cuda_runtime.h>

#include <algorithm>

#include "hsga_internal.h"
#include "hsga_island.cuh"
#include "hsga_sync.cuh"

namespace hsga {
namespace {

constexpr uint32_t kBatch = 16;  // generations whose per-island RNG blocks are batched

// Islands that one block takes alone, of up to 32 agents and of more.  us per
// generation in one block and in tiles, whose polls differ by 0.1 between
// devices: 2x4 islands of 17 0.73 and 1.06, 4x4 0.89 and 1.03, 3x7 1.07 and
// 1.05-1.17, 4x6 1.10 and 1.00-1.08; of 64 3x4 1.11 and 1.23, 2x7 1.25 and 1.19.
// Where fewer than every other generation migrates, tiles do not poll often
// enough to lose: 4x4 of 17 0.65 and 0.61 with an interval of 4.
constexpr uint32_t kOneBlockIslands = 22, kOneBlockLarge = 12;

// Blocks of a tile per SM: 64 registers a thread, to which the launch bound of
// 1,024 holds the compiler.  68x71 islands of 24 in nine to an SM 2.03 us per
// generation, in eight 1.84.
constexpr int kTilesPerSM = 8;

// Most islands of n agents for which tiles of four are the faster kernel.  A
// lane per agent takes as long for 17 agents as for 31, and for 33 as for 64; a
// large tile's children are numbered flat.  us here and in large tiles: 64x64
// islands of 9 1.72, 65x66 1.85 and 1.63, 64x76 1.88 and 1.68; of 17 to 31 64x76
// 1.89 and 2.00 (tournament 5 2.50 and 2.72); of 48 54x54 1.88 and 2.03, 60x60
// 2.12 and 2.04; of 64 54x54 1.89 and 2.27, 65x66 2.61 and 2.59, 66x66 2.62 and
// 2.88.  (Beyond 4,864 islands on 152 SMs the tiles do not fit.)
constexpr uint32_t most_islands(uint32_t n) {
  return n <= 16 ? 4096u : n <= 32 || n > 48 ? 0xFFFFFFFFu : 3072u;
}

// Whether generation G migrates, and its migration number G / interval, in
// 32-bit arithmetic with the every-generation case first: a 64-bit modulo
// and a division per generation made up about half of the kernel's
// instructions on the 64x64-island grid.
__device__ __forceinline__ bool migration_of(const RunParams &p, uint32_t G, uint32_t *m_idx) {
  if (p.interval == 1u) {
    *m_idx = G;
    return true;
  }
  if (p.interval == 0u) return false;
  const uint32_t q = G / p.interval;
  *m_idx = q;
  return q * p.interval == G;
}

// The whole warp waits for the records of its island's neighbours
// in other tiles at once.  Lane 4d + j (< 16) polls word j of the record of
// direction d (if `polled`: that neighbour lies in another tile), so every
// poll fetches whole records in one round trip; the wait ends when every
// polled word carries seq.  Lane 4d + j's word is returned in *word.
// Returns false (on every lane) when it gave up.
__device__ bool wait_records_warp(const uint64_t *r, bool polled, uint32_t seq, const int *err,
                                  uint32_t *word) {
  const uint64_t t0 = now_ns();
  for (uint32_t spin = 1; spin < kMaxSpins; ++spin) {
    bool ready = true;
    if (polled) {
      const uint64_t v = ld_relaxed64(r);
      ready = (uint32_t)(v >> 32) == seq;
      *word = (uint32_t)v;
    }
    if (__all_sync(kFull, ready)) return true;
    if ((spin & 255u) == 0) {
      const bool stop = *(volatile const int *)err != 0 || now_ns() - t0 > kWaitNs;
      if (__any_sync(kFull, stop)) return false;
    }
  }
  return false;
}

// ONE: the grid is one tile, and no record leaves the block.
template <int AP, bool TRACKED, bool ONE>
__global__ void __launch_bounds__(ONE ? 32 * kOneBlockIslands : 1024)
    step_resident_warp_kernel(RunParams p, uint32_t G0, uint32_t ngen, int premigrated,
                              uint32_t tile_r, uint32_t tile_c, uint32_t *__restrict__ tplane,
                              uint64_t *__restrict__ splane, uint64_t *__restrict__ rec,
                              int *__restrict__ err) {
  constexpr uint32_t kSlots = ONE ? kOneBlockIslands : 4;  // islands of a block
  __shared__ uint4 srec[2 * kSlots];
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t pt[AP];
  uint64_t ps[AP];
  // this warp's island, and per direction (lane d < 4) where its neighbour's
  // record is read: shared-memory slot, or global record
  uint32_t isl, nb_island = 0, nb_slot = 0;
  bool nb_inside = true, publish_global, polls;
  const uint64_t *poll_word;  // lane 4d + j: word j of direction d's record
  {
    const uint32_t tiles_c = (p.cols + tile_c - 1) / tile_c;
    const uint32_t r0 = blockIdx.x / tiles_c * tile_r, c0 = blockIdx.x % tiles_c * tile_c;
    const uint32_t w = threadIdx.x >> 5;
    const uint32_t r = r0 + w / tile_c, c = c0 + w % tile_c;
    const bool active = r < p.rows && c < p.cols;
    isl = active ? r * p.cols + c : p.islands;
    if (active && lane < 4) {
      nb_island = neighbour(p, isl, lane);
      const uint32_t nr = nb_island / p.cols - r0, nc = nb_island % p.cols - c0;  // wrap if outside
      nb_inside = nr < tile_r && nc < tile_c;
      nb_slot = nb_inside ? nr * tile_c + nc : 0u;
    }
    publish_global = !ONE && __any_sync(kFull, !nb_inside);
    // lane 4d + j polls word j of direction d's record (both buffers: +buf offset)
    const uint32_t d = (lane >> 2) & 3u;
    const uint32_t nb_d = __shfl_sync(kFull, nb_island, d);
    const bool inside_d = __shfl_sync(kFull, nb_inside, d);
    polls = lane < 16 && !inside_d;
    poll_word = rec + (size_t)nb_d * 4 + (lane & 3u);
  }
#pragma unroll
  for (int a = 0; a < AP; ++a) {
    const uint32_t j = lane + 32u * a;
    pt[a] = 0;
    ps[a] = 0;
    if (isl < p.islands && j < p.n) {
      pt[a] = tplane[(size_t)isl * p.n + j];
      if constexpr (TRACKED) ps[a] = splane[(size_t)isl * p.n + j];
    }
  }
  const bool any_mig = p.interval != 0;
  bool failed = false;  // leave now (block-uniform)
  bool wfail = false;   // this warp's wait gave up; the block learns at its barrier

  for (uint32_t g0 = 0; g0 < ngen && !failed; g0 += kBatch) {
    // Batched per-chunk draws: lane o (< 16) holds the emigrant block of
    // generation G0+g0+o, lane 16+o its placement block; every lane holds
    // the packed deposit of generation G0+g0+(lane & 15).
    const uint32_t Gl = G0 + g0 + (lane & (kBatch - 1));
    const uint32_t dpack = deposit_pack(p, Gl);
    Words4 mig{0, 0, 0, 0};
    if (any_mig && isl < p.islands)
      mig = philox_rk(p, lane < kBatch ? kSlotEmigrant : kSlotImmigrant, isl, Gl,
                      kPurposeMigration);
    const uint32_t steps = min(kBatch, ngen - g0);
    for (uint32_t o = 0; o < steps; ++o) {
      const uint32_t G = G0 + g0 + o;
      const uint32_t dp = __shfl_sync(kFull, dpack, o);
      const Deposit dep = deposit_unpack(dp, (uint32_t)p.vmask);
      uint32_t m_idx = 0;
      const bool do_mig = migration_of(p, G, &m_idx) && !(premigrated && g0 + o == 0);
      uint32_t buf = 0, seq = 0;
      if (do_mig) {
        buf = m_idx & 1u;
        seq = m_idx + 1u;
        // a1: publish the emigrant before reading any
        if (isl < p.islands && !wfail) {
          const uint32_t eslot = uindex(__shfl_sync(kFull, mig.x, o), p.n);
          const uint32_t dir = __shfl_sync(kFull, mig.y, o) >> 30;
          if (lane == (eslot & 31u)) {
            uint32_t tv = pt[0];
            uint64_t sv = ps[0];
            if constexpr (AP == 2) {
              if (eslot >> 5) {
                tv = pt[1];
                sv = ps[1];
              }
            }
            srec[buf * kSlots + (threadIdx.x >> 5)] =
                make_uint4(tv, (uint32_t)sv, (uint32_t)(sv >> 32), dir);
            if (publish_global) {
              uint64_t *r = rec + ((size_t)buf * p.islands + isl) * 4;
              const uint64_t stamp = (uint64_t)seq << 32;
              st_relaxed64(r, stamp | tv);
              st_relaxed64(r + 1, stamp | (uint32_t)sv);
              st_relaxed64(r + 2, stamp | (uint32_t)(sv >> 32));
              st_relaxed64(r + 3, stamp | dir);
            }
          }
        }
        {
          // every warp of the tile arrives here once per migration, also
          // after a failed wait, so the block leaves together
          if constexpr (ONE) {
            __syncthreads();
          } else if (__syncthreads_or(wfail ? 1 : 0)) {
            failed = true;
            break;
          }
        }
      }
      if (isl >= p.islands) continue;
      Words4 w[AP];
      replication_words<AP>(p, isl, G, w);
      if (do_mig) {
        // a2: records from other tiles: one warp-wide wait, then lane d < 4
        // gathers the four words of direction d
        uint4 r = make_uint4(0, 0, 0, 0);
        if constexpr (!ONE) {
          uint32_t word = 0;
          const bool ok =
              wait_records_warp(poll_word + (size_t)buf * p.islands * 4, polls, seq, err, &word);
          const uint32_t src = (lane & 3u) << 2;
          r.x = __shfl_sync(kFull, word, src);
          r.y = __shfl_sync(kFull, word, src + 1);
          r.z = __shfl_sync(kFull, word, src + 2);
          r.w = __shfl_sync(kFull, word, src + 3);
          // after a failed wait the warp stops work and goes on to the next
          // barrier, where the block leaves together
          if (!ok) {
            if (lane == 0) atomicCAS(err, 0, kDevErrWaitTimeout);
            wfail = true;
          }
          if (wfail) continue;
        }
        if (lane < 4 && nb_inside) r = srec[buf * kSlots + nb_slot];
        const bool arrive = lane < 4 && r.w == ((lane + 2u) & 3u);
        const uint32_t arrivals = __ballot_sync(kFull, arrive);
        const uint32_t place[4] = {mig.x, mig.y, mig.z, mig.w};
#pragma unroll
        for (uint32_t dd = 0; dd < 4; ++dd) {
          if (arrivals & (1u << dd)) {
            const uint32_t slot = uindex(__shfl_sync(kFull, place[dd], kBatch + o), p.n);
            land<AP, TRACKED>(slot, dd, r.x, ((uint64_t)r.z << 32) | r.y, pt, ps);
          }
        }
      }
      uint32_t ct[AP];
      uint64_t cs[AP];
      if (dep.two)
        replicate<AP, TRACKED, false, true>(p, dep, isl, G, w, pt, ps, ct, cs);
      else
        replicate<AP, TRACKED>(p, dep, isl, G, w, pt, ps, ct, cs);
#pragma unroll
      for (int a = 0; a < AP; ++a) {
        pt[a] = ct[a];
        ps[a] = cs[a];
      }
    }
  }
  if (failed || wfail) return;
#pragma unroll
  for (int a = 0; a < AP; ++a) {
    const uint32_t j = lane + 32u * a;
    if (isl < p.islands && j < p.n) {
      tplane[(size_t)isl * p.n + j] = pt[a];
      if constexpr (TRACKED) splane[(size_t)isl * p.n + j] = ps[a];
    }
  }
}

using WarpFn = void (*)(RunParams, uint32_t, uint32_t, int, uint32_t, uint32_t, uint32_t *,
                        uint64_t *, uint64_t *, int *);

template <bool ONE>
WarpFn pick(const RunParams &p) {
  if (p.policy != HSGA_NONE)
    return p.n <= 32 ? step_resident_warp_kernel<1, true, ONE>
                     : step_resident_warp_kernel<2, true, ONE>;
  return p.n <= 32 ? step_resident_warp_kernel<1, false, ONE>
                   : step_resident_warp_kernel<2, false, ONE>;
}

}  // namespace

// One block for a few islands; else tiles of four islands whose blocks are all
// resident at once: of 2x2, 1x4 and 4x1 the one with the fewest polled edges.
bool resident_warp_plan(const RunParams &p, ResidentPlan *out, bool grid_only) {
  if (p.n == 32 || p.islands > most_islands(p.n)) return false;
  if (!grid_only && p.islands <= (p.n <= 32 ? kOneBlockIslands : kOneBlockLarge) &&
      (p.islands < 8u || p.interval == 1u || p.interval == 2u)) {
    out->tile = ResidentTile{p.rows, p.cols, 1, 0, 0, 0};
    out->blocks = 1;
    out->threads = (int)p.islands * 32;
    out->smem = 0;
    out->one_block = true;
    out->warp = true;
    return true;
  }
  int dev = 0, sms = 0, coop = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (!coop || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pick<false>(p), 128, 0) !=
                   cudaSuccess)
    return false;
  double best = 1e30;
  for (uint32_t tr = 1; tr <= 4; tr *= 2) {
    const uint32_t tc = 4 / tr;
    const uint32_t tiles_c = (p.cols + tc - 1) / tc;
    const uint64_t tiles = (uint64_t)((p.rows + tr - 1) / tr) * tiles_c;
    if (tiles > (uint64_t)std::min(per_sm, kTilesPerSM) * sms) continue;
    const double edges = (p.rows > tr ? 2.0 * tc : 0.0) + (p.cols > tc ? 2.0 * tr : 0.0);
    if (edges < best) {
      best = edges;
      out->tile = ResidentTile{tr, tc, tiles_c, 0, 0, 0};
      out->blocks = (int)tiles;
    }
  }
  if (best >= 1e30) return false;
  out->threads = 128;
  out->smem = 0;
  out->one_block = false;
  out->warp = true;
  return true;
}

cudaError_t launch_step_resident_warp(const RunParams &p, const ResidentPlan &plan, uint32_t G0,
                                      uint32_t ngen, bool premigrated, uint32_t *t, uint64_t *s,
                                      uint64_t *rec, int *err, cudaStream_t stream) {
  RunParams pp = p;
  int prem = premigrated ? 1 : 0;
  uint32_t tile_r = plan.tile.rows, tile_c = plan.tile.cols;
  if (plan.one_block) {
    pick<true>(p)<<<1, plan.threads, 0, stream>>>(pp, G0, ngen, prem, tile_r, tile_c, t, s, rec, err);
    return cudaGetLastError();
  }
  void *args[] = {&pp, &G0, &ngen, &prem, &tile_r, &tile_c, &t, &s, &rec, &err};
  return cudaLaunchCooperativeKernel((const void *)pick<false>(p), dim3(plan.blocks), dim3(plan.threads),
                                     args, 0, stream);
}

}  // namespace hsga
