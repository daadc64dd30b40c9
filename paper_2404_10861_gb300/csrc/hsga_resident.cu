// hsga_resident.cu -- persistent resident generation kernels.
//
// One launch advances many synchronous generations with the whole population
// in shared memory.  The torus is cut into rectangular tiles of islands, one
// tile and one block per SM (a grid of few islands: one tile, one block); a
// cooperative launch keeps every block resident.  Children are written to the
// other of two buffers, so parents stay readable until the block's barrier at
// the end of a generation.  An island's emigrant of the next generation is
// copied to its record as soon as it is born, and each generation starts by
// landing the neighbours' records over the drawn members of the parents.
//
// A record is the whole genome and a stamp in 16 bytes: trait, surface low,
// surface high, (migration sequence number << 2 | direction).  Neighbours in
// the same tile read it from shared memory; an island on a tile's edge also
// stores it to global memory, in a slot double-buffered by migration parity,
// as one 16-byte relaxed store, which is single-copy atomic: a reader that
// sees the expected number holds the whole record, with no flag and no fence.
// Two buffers suffice: the record of migration m is overwritten at m+2 by a
// warp that has read its neighbours' m+1 records, and a neighbour stores its
// m+1 record only after its read of the m record has returned.
//
// Two kernels share this scheme.  step_small_kernel serves tiles of up to 64
// islands of 32 agents, which latency bounds; step_resident_kernel all others,
// which instruction issue bounds.  Per generation on a GB300 (tilted surface,
// tournament 2), against the kernel before them, which held an island per
// warp in registers and spent 294 warp instructions per island-generation:
//   4x4 islands    0.51 us (0.90)   87 warp instructions, 116 with migration
//   64x64          1.27 us (1.75)   120; a read of a remote record alone is
//                                   0.35 us, without migration 0.61 us
//   128x128        2.31 (6.4 on the streamed kernel: it did not fit before)
//                                   80; without migration 1.77 us, 64
// Polling harder makes the exchange slower (two reads of a record in flight:
// 2.88 us on the 64x64 grid; a delay of 300 cycles before the first read:
// 1.42 against 1.27): reads of a line in the other die's L2 hold up the store
// that they wait for.
//
// Every wait is bounded (1 s of %globaltimer); on expiry the warp records a
// timeout in the grid's error word and in its block's failure word, and the
// block leaves at its next barrier, which lets its neighbours time out in
// turn.  The cooperative launch guarantees that every tile is resident, so
// waits only expire on an inconsistent state.
#include <cuda_runtime.h>

#include "hsga_internal.h"
#include "hsga_island.cuh"
#include "hsga_sync.cuh"

namespace hsga {

namespace {

constexpr uint32_t kMaxGroup = 8;   // most islands that a warp takes together
// Warps of a block with groups of kg islands.  Groups of eight hold so many
// draws in registers that only half as many warps fit, and are still faster
// where a tile has the islands: 28 warps of four with 64 registers spend 131
// instructions per island-generation where 14 warps of eight spend 80 (2.84
// and 2.31 us per generation on the 128x128 grid).
constexpr uint32_t group_warps(uint32_t kg) { return kg == 8u ? 16u : 32u; }
constexpr uint32_t kSmallTile = 64; // largest tile of the small-tile kernel
static_assert(kSmallTile >= 64, "larger tiles of 32-agent islands take groups of eight");
constexpr uint32_t kChunk = 16;       // generations whose draws are tabulated together
constexpr uint32_t kRemote = 1u << 31;  // neighbour in another tile: record slot

// Slot of island g's record: a tile's islands one after another, tiles apart, so
// that no 128-byte line is written by two tiles (stride 0: no room for that,
// slots in island order).
__device__ __forceinline__ uint32_t record_slot(const RunParams &p, const ResidentTile &t,
                                                uint32_t g) {
  if (t.stride == 0u) return g;
  const uint32_t r = g / p.cols, c = g - r * p.cols;
  const uint32_t tr = r / t.rows, tc = c / t.cols;
  return (tr * t.tiles_c + tc) * t.stride + (r - tr * t.rows) * t.cols + c - tc * t.cols;
}
constexpr uint32_t kBuf1 = 1u << 31;    // migration word: record buffer 1

// A record as one single-copy atomic access: 16 bytes, or 8 (trait, stamp)
// when there is no surface.  (An untracked record is not simply a 16-byte one
// with unread middle words: the assembler then fetches the two words that are
// read separately, and they can belong to different records.)
template <bool TRACKED>
__device__ __forceinline__ uint4 ld_record(const uint4 *p) {
  uint64_t a, b;
  if constexpr (TRACKED) {
    asm volatile(
        "{\n .reg .b128 v;\n ld.relaxed.gpu.global.b128 v, [%2];\n mov.b128 {%0, %1}, v;\n}"
        : "=l"(a), "=l"(b)
        : "l"(p)
        : "memory");
  } else {
    const uint64_t v = ld_relaxed64((const uint64_t *)p);
    a = (uint32_t)v;
    b = v & 0xFFFFFFFF00000000ull;
  }
  return make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
}

template <bool TRACKED>
__device__ __forceinline__ void st_record(uint4 *p, const uint4 &r) {
  if constexpr (TRACKED) {
    const uint64_t a = ((uint64_t)r.y << 32) | r.x, b = ((uint64_t)r.w << 32) | r.z;
    asm volatile(
        "{\n .reg .b128 v;\n mov.b128 v, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], v;\n}" ::"l"(
            p),
        "l"(a), "l"(b)
        : "memory");
  } else {
    st_relaxed64((uint64_t *)p, ((uint64_t)r.w << 32) | r.x);
  }
}

// Bounded wait of a whole warp until ready() holds on every lane: gives up
// (on every lane, returning false) after limit_ns of the global timer or
// kMaxSpins polls, whichever comes first, or as soon as an error has been
// reported in *err.

template <class F>
__device__ __forceinline__ bool wait_warp(const F &ready, const int *err, uint64_t limit_ns) {
  if (__all_sync(kFull, ready())) return true;
  const uint64_t t0 = now_ns();
  for (uint32_t spin = 1; spin < kMaxSpins; ++spin) {
    if (__all_sync(kFull, ready())) return true;
    if ((spin & 255u) == 0) {
      const bool stop = *(volatile const int *)err != 0 || now_ns() - t0 > limit_ns;
      if (__any_sync(kFull, stop)) return false;
    }
  }
  return false;
}

// hsga_wait_probe: the kernel's bounded wait on a caller's record of four
// 64-bit words, each carrying seq in its high half, in two turns: lane 0
// watching all four words, then lanes 0..3 one word each.  out[0] = 1 if both
// saw seq, 0 if either gave up; out[1] = nanoseconds spent in all.
__global__ void wait_probe_kernel(const uint64_t *record, uint32_t seq, uint64_t limit_ns,
                                  int *err, uint64_t *out) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t t0 = now_ns();
  const auto carries = [&](uint32_t j) { return (uint32_t)(ld_relaxed64(record + j) >> 32) == seq; };
  const bool ok = wait_warp(
      [&] { return lane > 0 || (carries(0) && carries(1) && carries(2) && carries(3)); }, err,
      limit_ns);
  const bool ok_words = wait_warp([&] { return lane > 3 || carries(lane); }, err, limit_ns);
  if (lane == 0) {
    out[0] = (ok && ok_words) ? 1u : 0u;
    out[1] = now_ns() - t0;
  }
}

// Migration word of generation G: 0 when it does not migrate, else the
// record stamp's sequence number (1 .. 2^30 - 1, cyclic in the migration
// number G / interval, so that consecutive records differ and cleared memory
// never matches) and the record buffer in the top bit.
__device__ __forceinline__ uint32_t migration_word(const RunParams &p, uint32_t G) {
  if (p.interval == 0u) return 0u;
  const uint32_t m = G / p.interval;
  if (m * p.interval != G) return 0u;
  return (m % 0x3FFFFFFFu + 1u) | ((m & 1u) ? kBuf1 : 0u);
}

// First row and column of this block's tile.
__device__ __forceinline__ void tile_origin(const ResidentTile &t, uint32_t *r0, uint32_t *c0) {
  const uint32_t tiles_r = gridDim.x / t.tiles_c;
  const uint32_t r = t.by_cols ? blockIdx.x % tiles_r : blockIdx.x / t.tiles_c;
  const uint32_t c = t.by_cols ? blockIdx.x / tiles_r : blockIdx.x - r * t.tiles_c;
  *r0 = r * t.rows;
  *c0 = c * t.cols;
}

template <bool B>
struct Bool {
  static constexpr bool value = B;
};

// What a whole block needs to know about a generation.
struct GenInfo {
  uint32_t clear_lo, clear_hi, clear2_lo, clear2_hi;  // as in Deposit
  uint32_t shifts;    // shift | two << 8 | shift2 << 16
  uint32_t mig;       // migration word of this generation
  uint32_t mig_next;  // of the next one (whose emigrants are chosen among the children)
  uint32_t G;
};

// Shared-memory layout of a tile of I islands (byte offsets): two buffers of
// genomes, two buffers of records, the tables.  An island's genomes are three
// runs of n words (traits, surfaces low, surfaces high): a warp's random
// reads of 32 words never conflict, and with n known at compile time every
// address of a child is one register plus a constant.
struct TileLayout {
  uint32_t island, buffer;  // bytes of an island's genomes, of one buffer
  uint32_t rec, gen, nb, isl, edge, plan, emig, flag, bytes;
};

__host__ __device__ __forceinline__ TileLayout tile_layout(uint32_t I, uint32_t n, bool tracked) {
  TileLayout l;
  l.island = (tracked ? 12u : 4u) * n;
  l.buffer = (I * l.island + 15u) & ~15u;
  l.rec = 2u * l.buffer;
  l.gen = l.rec + 32u * I;
  l.nb = l.gen + (uint32_t)sizeof(GenInfo) * kChunk;
  l.isl = l.nb + 16u * I;
  l.edge = l.isl + 4u * I;
  l.plan = l.edge + 4u * I;
  l.emig = l.plan + 8u * kChunk * I;
  l.flag = (l.emig + kChunk * I + 3u) & ~3u;
  l.bytes = l.flag + 16u;
  return l;
}

// a3-a6 of one child of each of K islands: parents at from + k stride (the
// island's genomes), child written at to + k stride (its slot's trait).  w:
// the children's replication draws; ga, gb: the generation's GenInfo;
// more(k, q): island k's draws of candidates 2 + 4q ... 5 + 4q.  PLAIN: no
// deleterious mutations and one field written.  kept(k, genome): what the
// child became.  All the reads come before the first write: the compiler can
// not tell the parents' buffer from the children's, and would otherwise
// finish one child before it starts the next.
template <bool TRACKED, bool T2, int NN, bool PLAIN, uint32_t K, class More, class Kept>
__device__ __forceinline__ void make_children(const RunParams &p, const unsigned char *from,
                                              unsigned char *to, uint32_t stride,
                                              const Words4 (&w)[K], const uint4 &ga,
                                              const uint4 &gb, const More &more,
                                              const Kept &kept) {
  const uint32_t plane = NN ? 4u * NN : 4u * p.n;
  const auto offset = [&](uint32_t x) {  // a drawn candidate, in bytes
    if constexpr (NN == 32) return (x >> 25) & 0x7Cu;
    else return 4u * uindex(x, p.n);
  };
  const auto word = [&](uint32_t k, uint32_t b) {
    return *(const uint32_t *)(from + k * stride + b);
  };
  uint32_t best[K], fbest[K], lo[K], hi[K];
#pragma unroll
  for (uint32_t k = 0; k < K; ++k) {
    best[k] = offset(w[k].x);
    fbest[k] = word(k, best[k]);
  }
  if (T2 || p.tournament >= 2u) {
    uint32_t c[K], fc[K];
#pragma unroll
    for (uint32_t k = 0; k < K; ++k) {
      c[k] = offset(w[k].y);
      fc[k] = word(k, c[k]);
    }
#pragma unroll
    for (uint32_t k = 0; k < K; ++k) {
      best[k] = fc[k] > fbest[k] ? c[k] : best[k];
      fbest[k] = max(fc[k], fbest[k]);
    }
  }
  if constexpr (!T2) {
    for (uint32_t t0 = 2; t0 < p.tournament; t0 += 4) {
#pragma unroll
      for (uint32_t k = 0; k < K; ++k) {
        const Words4 x = more(k, (t0 - 2) / 4);
        const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
        uint32_t c[4], fc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          c[q] = offset(xw[q]);
          fc[q] = word(k, c[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const bool take = t0 + q < p.tournament && fc[q] > fbest[k];
          best[k] = take ? c[q] : best[k];
          fbest[k] = take ? fc[q] : fbest[k];
        }
      }
    }
  }
  if constexpr (TRACKED) {
#pragma unroll
    for (uint32_t k = 0; k < K; ++k) {
      lo[k] = word(k, best[k] + plane);
      hi[k] = word(k, best[k] + 2u * plane);
    }
  }
#pragma unroll
  for (uint32_t k = 0; k < K; ++k) {
    const uint32_t ct =
        PLAIN || !p.has_del ? mutate<false>(p, fbest[k], w[k].z) : mutate(p, fbest[k], w[k].z);
    unsigned char *const out = to + k * stride;
    *(uint32_t *)out = ct;
    if constexpr (TRACKED) {
      const uint32_t v = w[k].w << (gb.x & 31u);
      lo[k] = (lo[k] & ga.x) | (v & ~ga.x);
      hi[k] = (hi[k] & ga.y) | (v & ~ga.y);
      if (!PLAIN && (gb.x & 0x100u)) {
        const uint32_t v2 = (w[k].w >> 16) << (gb.x >> 16);
        lo[k] = (lo[k] & ga.z) | (v2 & ~ga.z);
        hi[k] = (hi[k] & ga.w) | (v2 & ~ga.w);
      }
      *(uint32_t *)(out + plane) = lo[k];
      *(uint32_t *)(out + 2u * plane) = hi[k];
    }
    kept(k, make_uint4(ct, TRACKED ? lo[k] : 0u, TRACKED ? hi[k] : 0u, 0u));
  }
}

// Tiles of any size: a warp takes groups of KG islands, lands their immigrants
// (four lanes per island), replicates them and copies their emigrants; one
// block barrier per generation.  The migration draws of 16 generations are
// evaluated at once into tables, one Philox block per thread.  Bound by issue
// and the generator's multiplies: 136 cycles per island-generation and
// scheduler without migration on the 128x128 grid, of which the multiplies
// hold the FMA-heavy pipe for 76.
// NN: agents per island when known at compile time (32), else 0.  T2: the
// tournament size is exactly 2.
template <bool TRACKED, bool T2, int NN, uint32_t KG>
__global__ void __launch_bounds__(group_warps(KG) * 32, 1)
    step_resident_kernel(RunParams p, ResidentTile tile, uint32_t G0, uint32_t ngen,
                         int premigrated, uint32_t *__restrict__ tplane,
                         uint64_t *__restrict__ splane, uint4 *__restrict__ grec,
                         int *__restrict__ err) {
  static_assert(KG == 2 || KG == 4 || KG == 8, "a group's indices are read as vectors");
  extern __shared__ __align__(16) unsigned char smem[];
  const uint32_t n = NN ? (uint32_t)NN : p.n;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, nthr = blockDim.x;
  const uint32_t warp = __shfl_sync(kFull, tid >> 5, 0), nwarp = nthr >> 5;
  // this block's tile: rows [r0, r0 + h), columns [c0, c0 + w)
  uint32_t r0, c0;
  tile_origin(tile, &r0, &c0);
  const uint32_t h = min(tile.rows, p.rows - r0), w = min(tile.cols, p.cols - c0);
  const uint32_t I = h * w, agents = I * n;
  const uint32_t groups = (I + KG - 1u) / KG, IP = groups * KG;  // padded with idle islands
  const TileLayout L = tile_layout(
      (tile.rows * tile.cols + kMaxGroup - 1u) / kMaxGroup * kMaxGroup, n, TRACKED);
  const uint32_t isz = NN ? (TRACKED ? 12u : 4u) * NN : L.island;  // an island's genomes
  uint4 *const srec = (uint4 *)(smem + L.rec);         // [buffer][island]
  GenInfo *const gens = (GenInfo *)(smem + L.gen);
  uint32_t *const nbloc = (uint32_t *)(smem + L.nb);   // 4 per island: local index or kRemote | global
  uint32_t *const gisl = (uint32_t *)(smem + L.isl);   // global index
  uint32_t *const edge = (uint32_t *)(smem + L.edge);  // a neighbour lies in another tile
  // [generation][island][direction]: landing slot | later directions with the same slot << 8
  uint16_t *const plan = (uint16_t *)(smem + L.plan);
  uint8_t *const emig = (uint8_t *)(smem + L.emig);    // [generation][island]: slot | dir << 6
  volatile uint32_t *const failed = (volatile uint32_t *)(smem + L.flag);
  if (tid == 0) *failed = ~0u;  // the launch's generation in which a wait gave up
  for (uint32_t i = tid; i < IP; i += nthr) {
    const uint32_t lr = i / w, lc = i - lr * w;
    const uint32_t g = (r0 + lr) * p.cols + c0 + lc;
    uint32_t e = 0;
#pragma unroll
    for (uint32_t d = 0; d < 4; ++d) {
      uint32_t loc = i;  // an idle island is its own neighbour
      if (i < I) {
        const uint32_t nb = neighbour(p, g, d);
        const uint32_t nr = nb / p.cols - r0, nc = nb % p.cols - c0;  // wraps if outside
        loc = nr < h && nc < w ? nr * w + nc : (record_slot(p, tile, nb) | kRemote);
      }
      nbloc[4 * i + d] = loc;
      e |= loc & kRemote;
    }
    gisl[i] = i < I ? g : 0u;
    edge[i] = e ? record_slot(p, tile, g) | kRemote : 0u;
  }
  __syncthreads();
  for (uint32_t f = tid; f < IP * n; f += nthr) {
    const uint32_t i = f / n, j = f - i * n;
    const size_t a = (size_t)gisl[i] * n + j;
    uint32_t *const t = (uint32_t *)(smem + i * isz) + j;
    t[0] = i < I ? tplane[a] : 0u;
    if constexpr (TRACKED) {
      const uint64_t sv = i < I ? splane[a] : 0ull;
      t[n] = (uint32_t)sv;
      t[2 * n] = (uint32_t)(sv >> 32);
    }
  }
  // a warp with a single group keeps what its lanes land in registers
  const bool single = groups <= nwarp;
  const uint32_t lane_loc = single && warp < groups && lane < 4u * KG ? nbloc[4u * KG * warp + lane] : 0u;
  const bool has_del = p.has_del != 0u;
  uint32_t cur = 0;  // byte offset of the parents' buffer: 0 or L.buffer
  for (uint32_t g0 = 0; g0 < ngen; g0 += kChunk) {
    // The chunk's tables: generation infos, landing slots of generations
    // G0 + g0 + o and emigrants of generations G0 + g0 + o + 1.
    const uint32_t steps = min(kChunk, ngen - g0);
    if (tid < kChunk) {
      const uint32_t G = G0 + g0 + tid;
      const Deposit d = deposit_for(p, G);
      GenInfo gi;
      gi.clear_lo = d.clear_lo;
      gi.clear_hi = d.clear_hi;
      gi.clear2_lo = d.clear2_lo;
      gi.clear2_hi = d.clear2_hi;
      gi.shifts = d.shift | (d.two << 8) | (d.shift2 << 16);
      gi.mig = (premigrated && g0 + tid == 0) ? 0u : migration_word(p, G);
      // no emigrants for a generation beyond this launch
      gi.mig_next = g0 + tid + 1u < ngen ? migration_word(p, G + 1u) : 0u;
      gi.G = G;
      gens[tid] = gi;
    }
    if (p.interval != 0u) {
      for (uint32_t o = warp; o < 2u * steps; o += nwarp) {
        const bool place = o >= steps;
        const uint32_t oo = place ? o - steps : o;
        for (uint32_t i = lane; i < IP; i += 32u) {
          const Words4 m = philox_rk(p, place ? kSlotImmigrant : kSlotEmigrant, gisl[i],
                                     G0 + g0 + oo + (place ? 0u : 1u), kPurposeMigration);
          if (place) {
            const uint32_t a = uindex_nn<NN>(m.x, n), b = uindex_nn<NN>(m.y, n);
            const uint32_t c = uindex_nn<NN>(m.z, n), d = uindex_nn<NN>(m.w, n);
            const uint32_t ea = (a == b ? 0x200u : 0u) | (a == c ? 0x400u : 0u) |
                                (a == d ? 0x800u : 0u);
            const uint32_t eb = (b == c ? 0x400u : 0u) | (b == d ? 0x800u : 0u);
            const uint32_t ec = c == d ? 0x800u : 0u;
            *(uint2 *)(plan + 4u * (oo * IP + i)) =
                make_uint2(a | ea | ((b | eb) << 16), c | ec | (d << 16));
          } else
            emig[oo * IP + i] = (uint8_t)(uindex_nn<NN>(m.x, n) | ((m.y >> 30) << 6));
        }
      }
    }
    __syncthreads();
    if (g0 == 0 && gens[0].mig != 0u) {
      // the first generation's emigrants come from the loaded population
      const uint32_t mw = gens[0].mig;
      for (uint32_t i = tid; i < I; i += nthr) {
        const Words4 m = philox_rk(p, kSlotEmigrant, gisl[i], G0, kPurposeMigration);
        const uint32_t *const t = (const uint32_t *)(smem + i * isz) + uindex_nn<NN>(m.x, n);
        const uint4 r = make_uint4(t[0], TRACKED ? t[n] : 0u, TRACKED ? t[2 * n] : 0u,
                                   (mw << 2) | (m.y >> 30));
        srec[(mw & kBuf1 ? IP : 0u) + i] = r;
        if (edge[i])
          st_record<TRACKED>(grec + (mw & kBuf1 ? tile.slots : 0u) + (edge[i] & ~kRemote), r);
      }
      __syncthreads();
    }
    for (uint32_t o = 0; o < steps; ++o) {
      const uint4 ga = ((const uint4 *)(gens + o))[0], gb = ((const uint4 *)(gens + o))[1];
      const uint32_t G = gb.w, mig = gb.y, mig_next = gb.z;
      unsigned char *const from = smem + cur;
      unsigned char *const to = smem + (L.buffer - cur);
      [[maybe_unused]] LaneHead head, head2;
      if constexpr (NN == 32) {
        head = lane_head(p, lane, G, kPurposeReplicate);
        if constexpr (!T2) head2 = lane_head(p, lane, G, kPurposeReplicate + 1u);
      }
      const bool plain = !has_del && !(gb.x & 0x100u);
      for (uint32_t grp = warp; grp < groups; grp += nwarp) {
        const uint32_t i0 = grp * KG;
        uint32_t gi[KG];
        if constexpr (KG >= 4) {
#pragma unroll
          for (uint32_t k = 0; k < KG; k += 4) {
            const uint4 v = *(const uint4 *)(gisl + i0 + k);
            gi[k] = v.x, gi[k + 1] = v.y, gi[k + 2] = v.z, gi[k + 3] = v.w;
          }
        } else {
          const uint2 v = *(const uint2 *)(gisl + i0);
          gi[0] = v.x, gi[1] = v.y;
        }
        unsigned char *const pa = from + i0 * isz, *const ch = to + i0 * isz;
        [[maybe_unused]] Words4 wd[KG];
        if constexpr (NN == 32) {
#pragma unroll
          for (uint32_t k = 0; k < KG; ++k) wd[k] = lane_tail(p, head, gi[k]);
        }
        if (mig != 0u) {
          // land: lane 4k + d handles direction d of island i0 + k
          const bool mine = lane < 4u * KG;
          const uint32_t loc = single ? lane_loc : mine ? nbloc[4u * i0 + lane] : 0u;
          const uint32_t pl = mine ? plan[4u * (o * IP + i0) + lane] : 0u;
          const uint4 *const in = grec + (mig & kBuf1 ? tile.slots : 0u) + (loc & ~kRemote);
          bool have = (loc & kRemote) == 0u;
          uint4 r = make_uint4(0, 0, 0, 0);
          if (have) r = srec[(mig & kBuf1 ? IP : 0u) + loc];
          const bool ok = wait_warp(
              [&] {
                if (!have) {
                  r = ld_record<TRACKED>(in);
                  have = (r.w >> 2) == (mig & 0x3FFFFFFFu);
                }
                return have;
              },
              err, kWaitNs);
          if (!ok) {
            if (lane == 0) {
              atomicCAS(err, 0, kDevErrWaitTimeout);
              *failed = g0 + o;
            }
            break;
          }
          const bool arrive = mine && ((r.w ^ lane) & 3u) == 2u;  // aimed back: d ^ 2
          const uint32_t later = __ballot_sync(kFull, arrive) >> (lane & 28u);
          if (arrive && (later & (pl >> 8)) == 0u) {
            uint32_t *const x = (uint32_t *)(pa + (lane >> 2) * isz) + (pl & 0xFFu);
            x[0] = r.x;
            if constexpr (TRACKED) {
              x[n] = r.y;
              x[2 * n] = r.z;
            }
          }
          __syncwarp();
        }
        if constexpr (NN == 32) {
          const auto all = [&](auto pln) {
            make_children<TRACKED, T2, NN, decltype(pln)::value, KG>(
                p, pa, ch + 4u * lane, isz, wd, ga, gb,
                [&](uint32_t k, uint32_t q) {
                  return q == 0 ? lane_tail(p, head2, gi[k])
                                : philox_rk(p, lane, gi[k], G, kPurposeReplicate + 1 + q);
                },
                [](uint32_t, const uint4 &) {});
          };
          if (plain) all(Bool<true>{});
          else all(Bool<false>{});
        } else {
          // the group's children numbered flat over the lanes
          for (uint32_t c = lane; c < KG * n; c += 32u) {
            const uint32_t k = c / n, j = c - k * n, g = gisl[i0 + k];
            const Words4 x[1] = {philox_rk(p, j, g, G, kPurposeReplicate)};
            make_children<TRACKED, T2, NN, false, 1>(
                p, pa + k * isz, ch + k * isz + 4u * j, 0u, x, ga, gb,
                [&](uint32_t, uint32_t q) {
                  return philox_rk(p, j, g, G, kPurposeReplicate + 1 + q);
                },
                [](uint32_t, const uint4 &) {});
          }
        }
        if (mig_next != 0u) {
          // next generation's emigrants: lane k copies island k's
          __syncwarp();
          if (lane < KG) {
            const uint32_t i = i0 + lane, e = emig[o * IP + i];
            const uint32_t *const x = (const uint32_t *)(ch + lane * isz) + (e & 63u);
            const uint4 r = make_uint4(x[0], TRACKED ? x[n] : 0u, TRACKED ? x[2 * n] : 0u,
                                       (mig_next << 2) | (e >> 6));
            if (edge[i])
              st_record<TRACKED>(
                  grec + (mig_next & kBuf1 ? tile.slots : 0u) + (edge[i] & ~kRemote), r);
            srec[(mig_next & kBuf1 ? IP : 0u) + i] = r;
          }
        }
      }
      cur = L.buffer - cur;
      __syncthreads();
      // (a warp ahead may already have failed in the next generation)
      if (*failed <= g0 + o) return;
    }
  }
  for (uint32_t f = tid; f < agents; f += nthr) {
    const uint32_t i = f / n, j = f - i * n;
    const size_t a = (size_t)gisl[i] * n + j;
    const uint32_t *const t = (const uint32_t *)(smem + cur + i * isz) + j;
    tplane[a] = t[0];
    if constexpr (TRACKED) splane[a] = ((uint64_t)t[2 * n] << 32) | t[n];
  }
}

// ------------------------------------------------------- small tiles ---
// Tiles of few 32-agent islands are bound by latency, not by instructions, so
// the phases of a generation run on warps of their own and overlap:
//   child warps   KC islands each: between the two barriers of a generation
//                 they select, mutate and deposit (the emigrating lane also
//                 writes its island's record); while the immigrants land they
//                 evaluate the generation's replication draws;
//   land warps    four lanes per island: read the neighbours' records (or
//                 wait for them) and land the arrivals;
//   draw warps    the migration draws of two generations ahead, one row of
//                 placement slots and emigrants per generation.
// Rows live in rings of kRows generations, generation infos (a warp's worth
// evaluated at a time) in a ring of 2 kGenBatch.
constexpr uint32_t kRows = 4;
constexpr uint32_t kGenBatch = 32;

// The block's barrier, from any of its warps' code.
__device__ __forceinline__ void block_barrier() {
  asm volatile("barrier.sync 0;" ::: "memory");
}

struct SmallLayout {  // byte offsets
  uint32_t buffer, rec, gen, plan, emig, flag, bytes;
};

__host__ __device__ __forceinline__ SmallLayout small_layout(uint32_t I, bool tracked) {
  SmallLayout l;
  l.buffer = I * (tracked ? 384u : 128u);
  l.rec = 2u * l.buffer;
  l.gen = l.rec + 16u * I;
  l.plan = l.gen + (uint32_t)sizeof(GenInfo) * 2u * kGenBatch;
  l.emig = l.plan + 8u * kRows * I;
  l.flag = (l.emig + kRows * I + 3u) & ~3u;
  l.bytes = l.flag + 16u;
  return l;
}

// Row r of the migration draws (generation G) of island i into the rings.
__device__ __forceinline__ void draw_row(const RunParams &p, uint32_t r, uint32_t G, uint32_t g,
                                         bool place, uint32_t i, uint32_t IP, uint16_t *plan,
                                         uint8_t *emig) {
  const Words4 m =
      philox_rk(p, place ? kSlotImmigrant : kSlotEmigrant, g, G, kPurposeMigration);
  const uint32_t a = m.x >> 27, b = m.y >> 27, c = m.z >> 27, d = m.w >> 27;
  const uint32_t at = (r % kRows) * IP + i;
  if (place) {
    const uint32_t ea =
        (a == b ? 0x200u : 0u) | (a == c ? 0x400u : 0u) | (a == d ? 0x800u : 0u);
    const uint32_t eb = (b == c ? 0x400u : 0u) | (b == d ? 0x800u : 0u);
    const uint32_t ec = c == d ? 0x800u : 0u;
    *(uint2 *)(plan + 4u * at) = make_uint2(a | ea | ((b | eb) << 16), c | ec | (d << 16));
  } else {
    emig[at] = (uint8_t)(a | ((m.y >> 30) << 6));
  }
}

// Generation info of generation number g of the launch (g < ngen).
__device__ __forceinline__ GenInfo gen_info(const RunParams &p, uint32_t G0, uint32_t g,
                                            uint32_t ngen, int premigrated) {
  const uint32_t G = G0 + g;
  const Deposit d = deposit_for(p, G);
  GenInfo gi;
  gi.clear_lo = d.clear_lo;
  gi.clear_hi = d.clear_hi;
  gi.clear2_lo = d.clear2_lo;
  gi.clear2_hi = d.clear2_hi;
  gi.shifts = d.shift | (d.two << 8) | (d.shift2 << 16);
  gi.mig = (premigrated && g == 0) ? 0u : migration_word(p, G);
  // no emigrants for a generation beyond this launch
  gi.mig_next = g + 1u < ngen ? migration_word(p, G + 1u) : 0u;
  gi.G = G;
  return gi;
}

// ONE: the grid is one tile, and no record leaves the block (4x4 islands 0.487 us
// per generation, 0.543 with the code for records and waits in place).
template <bool TRACKED, bool T2, uint32_t KC, bool ONE>
__global__ void __launch_bounds__(1024, 1)
    step_small_kernel(RunParams p, ResidentTile tile, uint32_t G0, uint32_t ngen, int premigrated,
                      uint32_t *__restrict__ tplane, uint64_t *__restrict__ splane,
                      uint4 *__restrict__ grec, int *__restrict__ err) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr uint32_t isz = TRACKED ? 384u : 128u;
  const uint32_t tid = threadIdx.x, lane = tid & 31u;
  const uint32_t warp = __shfl_sync(kFull, tid >> 5, 0);
  uint32_t r0, c0;
  tile_origin(tile, &r0, &c0);
  const uint32_t h = min(tile.rows, p.rows - r0), w = min(tile.cols, p.cols - c0);
  const uint32_t I = h * w;
  // roles are laid out for a full tile; a cut-off tile has idle warps
  const uint32_t IF = (tile.rows * tile.cols + KC - 1u) / KC * KC;
  const uint32_t nchild = IF / KC, nland = (IF + 7u) / 8u;  // the rest draw
  const SmallLayout L = small_layout(IF, TRACKED);
  uint4 *const srec = (uint4 *)(smem + L.rec);
  GenInfo *const gens = (GenInfo *)(smem + L.gen);
  uint16_t *const plan = (uint16_t *)(smem + L.plan);
  uint8_t *const emig = (uint8_t *)(smem + L.emig);
  volatile uint32_t *const failed = (volatile uint32_t *)(smem + L.flag);
  const auto global_index = [&](uint32_t i) {
    const uint32_t lr = i / w;
    return (r0 + lr) * p.cols + c0 + (i - lr * w);
  };
  // island li's neighbour in direction d: local index, or kRemote | global
  const auto locate = [&](uint32_t li, uint32_t d) {
    const uint32_t nb = neighbour(p, global_index(li), d);
    const uint32_t nr = nb / p.cols - r0, nc = nb % p.cols - c0;  // wraps if outside
    return nr < h && nc < w ? nr * w + nc : (record_slot(p, tile, nb) | kRemote);
  };
  if (tid == 0) *failed = ~0u;
  for (uint32_t f = tid; f < IF * 32u; f += blockDim.x) {
    const uint32_t i = f >> 5;
    uint32_t *const t = (uint32_t *)(smem + i * isz) + lane;
    const size_t a = i < I ? (size_t)global_index(i) * 32u + lane : 0u;
    t[0] = i < I ? tplane[a] : 0u;
    if constexpr (TRACKED) {
      const uint64_t sv = i < I ? splane[a] : 0ull;
      t[32] = (uint32_t)sv;
      t[64] = (uint32_t)(sv >> 32);
    }
  }
  for (uint32_t g = tid; g < min(2u * kGenBatch, ngen); g += blockDim.x)
    gens[g] = gen_info(p, G0, g, ngen, premigrated);
  if (p.interval != 0u)  // rows 0 and 1
    for (uint32_t q = tid; q < 4u * I; q += blockDim.x) {
      const uint32_t i = q >> 2, r = q & 1u;
      draw_row(p, r, G0 + r, global_index(i), (q & 2u) != 0u, i, IF, plan, emig);
    }
  block_barrier();
  if (gens[0].mig != 0u) {
    // the first generation's emigrants come from the loaded population
    const uint32_t mw = gens[0].mig;
    for (uint32_t i = tid; i < I; i += blockDim.x) {
      const uint32_t e = emig[i];
      const uint32_t *const t = (const uint32_t *)(smem + i * isz) + (e & 31u);
      const uint4 r = make_uint4(t[0], TRACKED ? t[32] : 0u, TRACKED ? t[64] : 0u,
                                 (mw << 2) | (e >> 6));
      srec[i] = r;
      uint32_t remote = 0;
#pragma unroll
      for (uint32_t d = 0; d < 4; ++d) remote |= locate(i, d);
      if (remote & kRemote)
        st_record<TRACKED>(
            grec + (mw & kBuf1 ? tile.slots : 0u) + record_slot(p, tile, global_index(i)), r);
    }
    block_barrier();
  }
  uint32_t cur = 0;  // byte offset of the parents' buffer
  if (warp < nchild) {
    // ---- child warps
    const uint32_t i0 = warp * KC;
    uint32_t g[KC];
    bool on_edge[KC];
    uint32_t slot[KC];  // of the record
#pragma unroll
    for (uint32_t k = 0; k < KC; ++k) {
      const bool live = i0 + k < I;
      g[k] = live ? global_index(i0 + k) : 0u;
      uint32_t remote = 0;
      if (live) {
#pragma unroll
        for (uint32_t d = 0; d < 4; ++d) remote |= locate(i0 + k, d);
      }
      on_edge[k] = !ONE && (remote & kRemote) != 0u;
      slot[k] = on_edge[k] ? record_slot(p, tile, g[k]) : 0u;
    }
    for (uint32_t gen = 0; gen < ngen; ++gen) {
      const uint4 *const info = (const uint4 *)(gens + (gen & (2u * kGenBatch - 1u)));
      const uint4 ga = info[0], gb = info[1];
      const uint32_t mig_next = gb.z;
      const LaneHead head = lane_head(p, lane, gb.w, kPurposeReplicate);
      [[maybe_unused]] LaneHead head2;
      if constexpr (!T2) head2 = lane_head(p, lane, gb.w, kPurposeReplicate + 1u);
      Words4 wd[KC];
#pragma unroll
      for (uint32_t k = 0; k < KC; ++k) wd[k] = lane_tail(p, head, g[k]);
      if (gb.y != 0u) {
        block_barrier();  // immigrants have landed
        if (*failed <= gen) return;
      }
      const unsigned char *const pa = smem + cur + i0 * isz;
      unsigned char *const ch = smem + (L.buffer - cur) + i0 * isz + 4u * lane;
      const uint8_t *const em = emig + ((gen + 1u) % kRows) * IF + i0;
      const bool plain = p.has_del == 0u && (gb.x & 0x100u) == 0u;
      const auto all = [&](auto pln) {
        make_children<TRACKED, T2, 32, decltype(pln)::value, KC>(
            p, pa, ch, isz, wd, ga, gb,
            [&](uint32_t k, uint32_t q) {
              return q == 0 ? lane_tail(p, head2, g[k])
                            : philox_rk(p, lane, g[k], gb.w, kPurposeReplicate + 1 + q);
            },
            [&](uint32_t k, uint4 r) {
              // next generation's emigrant, straight from its lane
              if (mig_next == 0u) return;
              const uint32_t e = em[k];
              if (((e ^ lane) & 31u) == 0u) {
                r.w = (mig_next << 2) | (e >> 6);
                if (on_edge[k])
                  st_record<TRACKED>(grec + (mig_next & kBuf1 ? tile.slots : 0u) + slot[k], r);
                srec[i0 + k] = r;
              }
            });
      };
      if (plain) all(Bool<true>{});
      else all(Bool<false>{});
      cur = L.buffer - cur;
      block_barrier();  // children and records are written
    }
  } else if (warp < nchild + nland) {
    // ---- land warps: lane 4k + d handles direction d of island i0 + k
    const uint32_t i0 = 8u * (warp - nchild), li = i0 + (lane >> 2);
    const bool mine = li < I;
    const uint32_t loc = mine ? locate(li, lane & 3u) : 0u;
    const bool local = ONE || (loc & kRemote) == 0u;
    const uint4 *const near = srec + (local ? loc : 0u);
    const uint4 *const far = grec + (loc & ~kRemote);
    for (uint32_t gen = 0; gen < ngen; ++gen) {
      const uint32_t mig = gens[gen & (2u * kGenBatch - 1u)].mig;
      if (mig != 0u) {
        const uint32_t pl = mine ? plan[4u * ((gen % kRows) * IF + i0) + lane] : 0u;
        const uint4 *const in = far + (mig & kBuf1 ? tile.slots : 0u);
        uint4 r = make_uint4(0, 0, 0, 0);
        if (local) r = *near;
        bool have = local;
        const bool ok = ONE || wait_warp(
                                   [&] {
                                     if (!have) {
                                       r = ld_record<TRACKED>(in);
                                       have = (r.w >> 2) == (mig & 0x3FFFFFFFu);
                                     }
                                     return have;
                                   },
                                   err, kWaitNs);
        if (ok) {
          const bool arrive = mine && ((r.w ^ lane) & 3u) == 2u;  // aimed back: d ^ 2
          const uint32_t later = __ballot_sync(kFull, arrive) >> (lane & 28u);
          if (arrive && (later & (pl >> 8)) == 0u) {
            uint32_t *const x = (uint32_t *)(smem + cur + li * isz) + (pl & 31u);
            x[0] = r.x;
            if constexpr (TRACKED) {
              x[32] = r.y;
              x[64] = r.z;
            }
          }
        } else if (lane == 0) {
          atomicCAS(err, 0, kDevErrWaitTimeout);
          *failed = gen;
        }
        block_barrier();
        if (*failed <= gen) return;
      }
      cur = L.buffer - cur;
      block_barrier();
    }
  } else {
    // ---- draw warps: row gen + 2 while generation gen runs
    const uint32_t dw = warp - nchild - nland, q = dw * 32u + lane, i = q >> 1;
    const bool draws = p.interval != 0u && i < I;
    const uint32_t g = draws ? global_index(i) : 0u;
    for (uint32_t gen = 0; gen < ngen; ++gen) {
      if (gens[gen & (2u * kGenBatch - 1u)].mig != 0u) {
        block_barrier();
        if (*failed <= gen) return;
      }
      if (draws && gen + 2u < ngen)
        draw_row(p, gen + 2u, G0 + gen + 2u, g, (q & 1u) != 0u, i, IF, plan, emig);
      // the half of the ring that the last batch of generations has used up
      if (dw == 0 && gen % kGenBatch == 0u && gen > 0u) {
        const uint32_t next = gen + kGenBatch + lane;
        if (next < ngen)
          gens[next & (2u * kGenBatch - 1u)] = gen_info(p, G0, next, ngen, premigrated);
      }
      cur = L.buffer - cur;
      block_barrier();
    }
  }
  for (uint32_t f = tid; f < I * 32u; f += blockDim.x) {
    const uint32_t i = f >> 5;
    const size_t a = (size_t)global_index(i) * 32u + lane;
    const uint32_t *const t = (const uint32_t *)(smem + cur + i * isz) + lane;
    tplane[a] = t[0];
    if constexpr (TRACKED) splane[a] = ((uint64_t)t[64] << 32) | t[32];
  }
}

// ------------------------------------------------------------- launch ---
using ResidentFn = void (*)(RunParams, ResidentTile, uint32_t, uint32_t, int, uint32_t *,
                            uint64_t *, uint4 *, int *);

template <int NN, uint32_t KG>
ResidentFn pick_group(const RunParams &p) {
  const bool t2 = p.tournament == 2;
  if (p.policy != HSGA_NONE)
    return t2 ? step_resident_kernel<true, true, NN, KG> : step_resident_kernel<true, false, NN, KG>;
  return t2 ? step_resident_kernel<false, true, NN, KG> : step_resident_kernel<false, false, NN, KG>;
}

template <uint32_t KC, bool ONE = false>
ResidentFn pick_small(const RunParams &p) {
  const bool t2 = p.tournament == 2;
  if (p.policy != HSGA_NONE)
    return t2 ? step_small_kernel<true, true, KC, ONE> : step_small_kernel<true, false, KC, ONE>;
  return t2 ? step_small_kernel<false, true, KC, ONE> : step_small_kernel<false, false, KC, ONE>;
}

// Warps of a small-tile block of I islands with kc islands per child warp.
uint32_t small_warps(uint32_t I, uint32_t kc) {
  const uint32_t IF = (I + kc - 1u) / kc * kc;
  return IF / kc + (IF + 7u) / 8u + (IF + 15u) / 16u;
}

// Islands per child warp of a small-tile block: the fewest whose warps fit in
// a block; 0 if the tile is not small or its islands do not fill a warp each.
uint32_t small_kc(uint32_t I, uint32_t n) {
  if (n != 32 || I > kSmallTile) return 0u;
  return small_warps(I, 1) <= 32u ? 1u : small_warps(I, 2) <= 32u ? 2u : 4u;
}

// Islands per group for any other tile of I islands: small groups where
// larger ones would leave most warps without one.  Islands of n > 24 agents fill
// a warp's lanes two at a time: 66x66 islands (33 to a tile) of 28 2.12 us per
// generation in groups of two, 2.29 of four; of 48 2.48 and 2.82; of 17 2.10 and
// 2.02; 76x80 (40) of 48 2.52 and 2.88; 80x80 (45) of 33 2.82 and 2.63.
uint32_t group_for(uint32_t I, uint32_t n) {
  return I <= (n > 24u ? 40u : 32u) ? 2u : I <= 64u ? 4u : kMaxGroup;
}

ResidentFn pick(const RunParams &p, const ResidentTile &t, bool one) {
  const uint32_t I = t.rows * t.cols, kg = group_for(I, p.n);
  if (one && small_kc(I, p.n) == 1u) return pick_small<1, true>(p);
  switch (small_kc(I, p.n)) {
    case 1: return pick_small<1>(p);
    case 2: return pick_small<2>(p);
    case 4: return pick_small<4>(p);
    default: break;
  }
  if (p.n == 32) return pick_group<32, kMaxGroup>(p);  // more than kSmallTile islands
  return kg == 2u ? pick_group<0, 2>(p) : kg == 4u ? pick_group<0, 4>(p) : pick_group<0, 8>(p);
}

// Threads of a block that holds I islands; with groups, one warp per group or
// as few rounds of at most 32 warps as the groups need.
uint32_t threads_for(uint32_t I, uint32_t n) {
  if (const uint32_t kc = small_kc(I, n)) return 32u * small_warps(I, kc);
  const uint32_t kg = group_for(I, n), groups = (I + kg - 1u) / kg;
  const uint32_t most = group_warps(kg), rounds = (groups + most - 1u) / most;
  return 32u * ((groups + rounds - 1u) / rounds);
}

}  // namespace

// Agents that one block takes alone instead of spreading over tiles, whose
// exchange costs about 0.2 us per generation (16 islands of 32: 0.51 us in one
// block, 0.69 in 16; 30 islands: 0.84 and 0.68).
constexpr uint32_t kOneBlockAgents = 768;

// Tiles of one island poll again just before their neighbours' records arrive
// once they spread over most of the device: 10x12 islands in 120 tiles 1.31 us
// per generation, in 60 tiles of two 0.76; 12x12 0.94 and 0.73; 8x12 in 96
// tiles 0.69.  A torus of one row is cut into pairs along it: 1x150 0.76, 2.6
// streamed.
constexpr uint32_t kMostSingles = 96;

// Islands of a tile up to which tiles keep their records apart.
constexpr uint32_t kMostApart = 96;

bool resident_plan(const RunParams &p, ResidentPlan *out, bool grid_only) {
  if (resident_warp_plan(p, out, grid_only)) return true;
  int dev = 0, sms = 0, coop = 0, smem = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const bool tracked = p.policy != HSGA_NONE;
  const auto bytes = [&](uint64_t I) {
    if (I <= kSmallTile)
      if (const uint32_t kc = small_kc((uint32_t)I, p.n))
        return small_layout(((uint32_t)I + kc - 1u) / kc * kc, tracked).bytes;
    const uint64_t padded = (I + kMaxGroup - 1) / kMaxGroup * kMaxGroup;
    return padded > 65536 ? ~0u : tile_layout((uint32_t)padded, p.n, tracked).bytes;
  };
  if (!grid_only && (uint64_t)p.islands * p.n <= kOneBlockAgents) {
    out->tile = ResidentTile{p.rows, p.cols, 1, 0, 0, 0};
    out->blocks = 1;
    out->one_block = true;
  } else {
    if (!coop) return false;
    // the smallest tile whose tiles are all resident at one per SM; among
    // tiles of a size, the shortest edge
    double best = 1e30;
    for (uint32_t tr = 1; tr <= p.rows && bytes(tr) <= (uint32_t)smem; ++tr) {
      const uint32_t tiles_r = (p.rows + tr - 1) / tr;
      if (tiles_r > (uint32_t)sms) continue;
      const uint32_t most_c = (uint32_t)sms / tiles_r;
      uint32_t tc = (p.cols + most_c - 1) / most_c;
      if (tr * tc == 1u && p.islands > kMostSingles) {
        if (p.rows > 1u) continue;  // tiles of two rows follow
        tc = 2u;
      }
      if (bytes((uint64_t)tr * tc) > (uint32_t)smem) continue;
      const double edge = (p.rows > tr ? 2.0 * tc : 0.0) + (p.cols > tc ? 2.0 * tr : 0.0);
      double cost = (double)tr * tc * p.n / 32.0 + 0.1 * edge;
      // small tiles (a warp or two per island) that all have the same size:
      // 64x64 islands 1.35 us in tiles of 4x8, 1.42 in 5x6 with ones cut off
      if (p.n == 32 && tr * tc <= kSmallTile && (p.rows % tr || p.cols % tc)) cost *= 1.1;
      if (cost < best) {
        best = cost;
        const uint32_t tiles_c = (p.cols + tc - 1) / tc;
        out->tile = ResidentTile{tr, tc, tiles_c, 0, 0, 0};
        out->blocks = (int)(tiles_r * tiles_c);
      }
    }
    if (best >= 1e30) return false;
    out->one_block = false;
  }
  const uint32_t I = out->tile.rows * out->tile.cols;
  // record slots: two buffers of at most two slots per island
  const uint64_t most = 2ull * p.islands, tiles = (uint64_t)out->blocks;
  const uint32_t apart = (I + 7u) & ~7u;
  // Slots apart: 64x64 islands 1.41 us against 1.57 in island order, 10x12 0.76
  // and 1.09, 100x100 1.95 and 2.00; but large tiles 128x128 2.40 and 2.32.
  out->tile.stride = I > kMostApart          ? 0u
                     : tiles * apart <= most ? apart
                     : tiles * I <= most     ? I
                                             : 0u;
  // Tiles down the columns: 64x64 islands 1.25 us against 1.35, 24x24 0.89 and
  // 0.94, 32x128 1.18 and 1.26; tiles of one or two 16x16 0.81 and 0.73, large
  // ones 100x100 1.98 and 1.95.
  out->tile.by_cols = p.n == 32 && I > 2u && I <= kSmallTile ? 1u : 0u;
  out->tile.slots = out->tile.stride ? (uint32_t)tiles * out->tile.stride : p.islands;
  out->threads = (int)threads_for(I, p.n);
  out->smem = bytes(I);
  return true;
}

cudaError_t launch_step_resident(const RunParams &p, const ResidentPlan &plan, uint32_t G0,
                                 uint32_t ngen, bool premigrated, uint32_t *t, uint64_t *s,
                                 uint64_t *rec, int *err, cudaStream_t stream) {
  if (plan.warp)
    return launch_step_resident_warp(p, plan, G0, ngen, premigrated, t, s, rec, err, stream);
  ResidentFn fn = pick(p, plan.tile, plan.one_block);
  // the device's limit, whatever the plan: other threads launch other tiles
  int dev = 0, limit = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
  if (e != cudaSuccess) return e;
  RunParams pp = p;
  ResidentTile tile = plan.tile;
  int prem = premigrated ? 1 : 0;
  uint4 *records = reinterpret_cast<uint4 *>(rec);
  if (plan.one_block) {
    fn<<<1, plan.threads, plan.smem, stream>>>(pp, tile, G0, ngen, prem, t, s, records, err);
    return cudaGetLastError();
  }
  void *args[] = {&pp, &tile, &G0, &ngen, &prem, &t, &s, &records, &err};
  return cudaLaunchCooperativeKernel((const void *)fn, dim3(plan.blocks), dim3(plan.threads), args,
                                     plan.smem, stream);
}

cudaError_t launch_wait_probe(const uint64_t *record, uint32_t seq, uint64_t limit_ns, int *err,
                              uint64_t *out, cudaStream_t stream) {
  wait_probe_kernel<<<1, 32, 0, stream>>>(record, seq, limit_ns, err, out);
  return cudaGetLastError();
}

}  // namespace hsga
