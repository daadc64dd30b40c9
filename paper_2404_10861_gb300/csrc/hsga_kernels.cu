// hsga_kernels.cu -- dispatch of the streamed generation kernels, explicit
// migration, end-state sampling, and the kernels that show the generator and the
// site functions by themselves.
//
// Streamed: one launch advances one synchronous generation of the whole
// grid (hsga_staged.cu, hsga_flat.cu); the population ping-pongs between two
// structure-of-arrays planes in HBM (uint32 traits, uint64 surfaces: 12 bytes per
// agent).  The kernel boundary is the generation barrier.  Migration needs no
// exchange buffer: the receiver works each neighbour's emigrant out from the
// counter-based generator and gathers that genome straight from the neighbour's
// parent plane.
#include <cuda_runtime.h>

#include "hsga_internal.h"
#include "hsga_island.cuh"

namespace hsga {

// ------------------------------------------------------ streamed step ---
// 32-agent integer islands with one surface word (the paper's shape) have a
// kernel of their own, whose bulk copies need planes on 16-byte boundaries; it
// and the flat kernel plan their launches themselves.

bool exceeds_l2(uint64_t bytes) {
  int dev = 0, l2 = 0;
  return cudaGetDevice(&dev) == cudaSuccess &&
         cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev) == cudaSuccess &&
         bytes > (uint64_t)l2;
}

bool planes_exceed_l2(const RunParams &p) {
  const uint64_t genome = 4u + 8u * (p.policy == HSGA_NONE ? 0u : p.words);
  return exceeds_l2(2u * genome * p.n * p.islands);
}

bool stream_plan(const RunParams &p, bool aligned, StreamPlan *out) {
  out->staged = p.n == 32 && p.words == 1 && !p.flt && aligned;
  return out->staged ? staged_stream_plan(p, out) : flat_stream_plan(p, out);
}

cudaError_t launch_step_streamed(const RunParams &p, const StreamPlan &plan, uint32_t G,
                                 bool do_mig, const Moves &mv, const uint32_t *tin,
                                 const uint64_t *sin, uint32_t *tout, uint64_t *sout, int *err,
                                 cudaStream_t stream) {
  if (plan.staged)
    return launch_step_staged(p, plan, G, do_mig, mv, tin, sin, tout, sout, err, stream);
  return launch_step_flat(p, plan, G, do_mig, mv, tin, sin, tout, sout, err, stream);
}

// --------------------------------------------------- explicit a1 + a2 ---
// Emigrants are written to per-island 16-byte records (one 128-bit store:
// trait, surface low, surface high, direction) before any immigrant lands;
// a second launch lands them in place.
__global__ void emigrate_kernel(RunParams p, uint32_t G, const uint32_t *__restrict__ t,
                                const uint64_t *__restrict__ s, uint4 *__restrict__ rec) {
  const uint32_t isl = blockIdx.x * blockDim.x + threadIdx.x;
  if (isl >= p.islands) return;
  const Words4 m = philox_rk(p, kSlotEmigrant, isl, G, kPurposeMigration);
  const size_t a = (size_t)isl * p.n + uindex(m.x, p.n);
  const uint64_t sv = s ? s[a] : 0ull;
  rec[isl] = make_uint4(t[a], (uint32_t)sv, (uint32_t)(sv >> 32), m.y >> 30);
}

__global__ void immigrate_kernel(RunParams p, uint32_t G, uint32_t *__restrict__ t,
                                 uint64_t *__restrict__ s, const uint4 *__restrict__ rec) {
  const uint32_t isl = blockIdx.x * blockDim.x + threadIdx.x;
  if (isl >= p.islands) return;
  const Words4 v = philox_rk(p, kSlotImmigrant, isl, G, kPurposeMigration);
  const uint32_t place[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (uint32_t d = 0; d < 4; ++d) {
    const uint4 r = rec[neighbour(p, isl, d)];
    if (r.w != ((d + 2u) & 3u)) continue;
    const size_t a = (size_t)isl * p.n + uindex(place[d], p.n);
    t[a] = r.x;
    if (s) s[a] = ((uint64_t)r.z << 32) | r.y;
  }
}

cudaError_t launch_migrate(const RunParams &p, uint32_t G, uint32_t *t, uint64_t *s,
                           uint4 *rec, cudaStream_t stream) {
  const uint32_t blocks = (p.islands + 255) / 256;
  emigrate_kernel<<<blocks, 256, 0, stream>>>(p, G, t, s, rec);
  immigrate_kernel<<<blocks, 256, 0, stream>>>(p, G, t, s, rec);
  return cudaGetLastError();
}

// ------------------------------------------------------------ a7 sample ---
// Partial Fisher-Yates over the islands, k draws r_j = j + floor(w_j (I-j) /
// 2^32), evaluated in parallel.  After all swaps, position j holds the value
// that position r_j held just before step j (no later step touches position
// j).  That value is r_j unless an earlier step i < j also drew r_i = r_j, in
// which case it is f(i) for the last such i, where f(i) is the value position
// i held at the start of step i: f(i) = i unless an earlier step i' < i drew
// r_i' = i, then f(i) = f(last such i').  "Last earlier step with draw p" is
// looked up in a hash table of the draws, chained per bucket (about one draw
// a bucket, in no particular order: the step numbers decide).
//
// Up to kSampleOneBlock draws the table lives in one block's shared memory;
// above, in scratch memory, filled by one kernel and read by a second, which
// spread over the whole device.  It replaces a bitonic sort of the draws in
// one block (k <= 12,288: 219 us for 10,000 genomes, now 13.7)
// and, above, the shuffle itself on one thread (1.8 ms for 16,384, now 13.8).
__device__ __forceinline__ uint32_t sample_draw(const RunParams &p, uint32_t G, uint32_t j) {
  const Words4 w = philox_rk(p, j, 0xFFFFFFFFu, G, kPurposeSampleDraw);
  return j + uindex(w.x, p.islands - j);
}

// head[b]: 1 + some draw of bucket b (0: none); node[i] = (draw, next).
struct DrawTable {
  uint32_t *head;
  uint2 *node;
  uint32_t mask;
};

__device__ __forceinline__ void insert_draw(const DrawTable &t, uint32_t j, uint32_t r) {
  const uint32_t next = atomicExch(&t.head[r & t.mask], j + 1u);
  t.node[j] = make_uint2(r, next);
}

// 1 + the last step before j that drew value p, or 0.
__device__ __forceinline__ uint32_t last_before(const DrawTable &t, uint32_t p, uint32_t j) {
  uint32_t best = 0;
  for (uint32_t e = t.head[p & t.mask]; e != 0u;) {
    const uint2 nd = t.node[e - 1u];
    if (nd.x == p && e <= j) best = max(best, e);
    e = nd.y;
  }
  return best;
}

__device__ __forceinline__ void emit_sample(const RunParams &p, uint32_t G, uint32_t j,
                                            const DrawTable &dt, uint32_t r,
                                            const uint32_t *__restrict__ t,
                                            const uint64_t *__restrict__ s,
                                            uint32_t *__restrict__ out_words,
                                            uint32_t *__restrict__ out_is,
                                            const uint32_t *__restrict__ T) {
  uint32_t island = r, e = last_before(dt, r, j);
  while (e != 0u) {  // f(e - 1): steps strictly decrease
    island = e - 1u;
    e = last_before(dt, island, island);
  }
  const Words4 w = philox_rk(p, kSlotSample, island, G, kPurposeMigration);
  const uint32_t slot = uindex(w.x, p.n);
  const size_t a = (size_t)island * p.n + slot;
  const uint64_t sv = s ? s[a] : 0ull;
  reinterpret_cast<uint4 *>(out_words)[j] =
      make_uint4(t[a], (uint32_t)sv, (uint32_t)(sv >> 32), T ? T[a] : G);
  if (out_is) reinterpret_cast<uint2 *>(out_is)[j] = make_uint2(island, slot);
}

constexpr uint32_t kSampleOneBlock = 1024;  // draws resolved by one block

__global__ void __launch_bounds__(kSampleOneBlock)
    sample_block_kernel(RunParams p, uint32_t G, uint32_t k, const uint32_t *__restrict__ t,
                        const uint64_t *__restrict__ s, uint32_t *__restrict__ out_words,
                        uint32_t *__restrict__ out_is, const uint32_t *__restrict__ T) {
  __shared__ uint2 node[kSampleOneBlock];
  __shared__ uint32_t head[kSampleOneBlock];
  const DrawTable dt{head, node, kSampleOneBlock - 1u};
  const uint32_t j = threadIdx.x;
  for (uint32_t b = j; b < kSampleOneBlock; b += blockDim.x) head[b] = 0u;
  __syncthreads();
  const uint32_t r = j < k ? sample_draw(p, G, j) : 0u;
  if (j < k) insert_draw(dt, j, r);
  __syncthreads();
  if (j < k) emit_sample(p, G, j, dt, r, t, s, out_words, out_is, T);
}

__global__ void sample_draw_kernel(RunParams p, uint32_t G, uint32_t k, DrawTable dt) {
  const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < k) insert_draw(dt, j, sample_draw(p, G, j));
}

__global__ void sample_emit_kernel(RunParams p, uint32_t G, uint32_t k, DrawTable dt,
                                   const uint32_t *__restrict__ t,
                                   const uint64_t *__restrict__ s,
                                   uint32_t *__restrict__ out_words,
                                   uint32_t *__restrict__ out_is,
                                   const uint32_t *__restrict__ T) {
  const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < k) emit_sample(p, G, j, dt, dt.node[j].x, t, s, out_words, out_is, T);
}

static uint32_t sample_buckets(uint32_t k) {  // the power of two at or above k
  uint32_t b = kSampleOneBlock;
  while (b < k && b < (1u << 31)) b <<= 1;
  return b;
}

size_t sample_scratch_bytes(uint32_t k) {
  return k <= kSampleOneBlock ? 0 : (size_t)k * sizeof(uint2) + (size_t)sample_buckets(k) * 4;
}

uint32_t sample_launches(uint32_t k) { return k <= kSampleOneBlock ? 1u : 2u; }

cudaError_t launch_sample(const RunParams &p, uint32_t G, uint32_t k, const uint32_t *t,
                          const uint64_t *s, uint32_t *out_words, uint32_t *out_is,
                          uint32_t *scratch, cudaStream_t stream, const uint32_t *T) {
  if (k == 0) return cudaSuccess;
  if (k <= kSampleOneBlock) {
    sample_block_kernel<<<1, (k + 31u) & ~31u, 0, stream>>>(p, G, k, t, s, out_words, out_is, T);
    return cudaGetLastError();
  }
  const uint32_t buckets = sample_buckets(k);
  const DrawTable dt{scratch + 2 * (size_t)k, reinterpret_cast<uint2 *>(scratch), buckets - 1u};
  cudaError_t e = cudaMemsetAsync(dt.head, 0, (size_t)buckets * 4, stream);
  if (e != cudaSuccess) return e;
  const uint32_t blocks = (k + 127u) / 128u;
  sample_draw_kernel<<<blocks, 128, 0, stream>>>(p, G, k, dt);
  sample_emit_kernel<<<blocks, 128, 0, stream>>>(p, G, k, dt, t, s, out_words, out_is, T);
  return cudaGetLastError();
}

// ------------------------------------------------------------ philox ---
__global__ void philox_sweep_kernel(uint32_t k0, uint32_t k1, uint32_t c0, uint32_t count,
                                    uint32_t c1, uint32_t c2, uint32_t c3,
                                    uint4 *__restrict__ out) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += gridDim.x * blockDim.x) {
    const Words4 w = philox(k0, k1, c0 + i, c1, c2, c3);
    out[i] = make_uint4(w.x, w.y, w.z, w.w);
  }
}

cudaError_t launch_philox_sweep(uint64_t seed, uint32_t c0, uint32_t count, uint32_t c1,
                                uint32_t c2, uint32_t c3, uint32_t *out, cudaStream_t stream) {
  if (count == 0) return cudaSuccess;
  uint32_t blocks = (count + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  philox_sweep_kernel<<<blocks, 256, 0, stream>>>((uint32_t)seed, (uint32_t)(seed >> 32), c0,
                                                  count, c1, c2, c3, (uint4 *)out);
  return cudaGetLastError();
}

// ---------------------------------------------------- Philox throughput ---
// Thread t draws the blocks for counters (i, t, c2, c3), i < m, in the form
// the generation kernels use (round keys in the parameter block), four
// independent chains at a time, and stores the xor of every word it drew
// (so that no draw can be optimised away).
__global__ void __launch_bounds__(256)
    philox_throughput_kernel(RunParams p, uint32_t threads, uint32_t m, uint32_t c2,
                             uint32_t c3, uint32_t *__restrict__ out) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= threads) return;
  uint32_t acc = 0;
  uint32_t i = 0;
  for (; i + 4 <= m; i += 4) {
    const Words4 a = philox_rk(p, i, t, c2, c3);
    const Words4 b = philox_rk(p, i + 1, t, c2, c3);
    const Words4 c = philox_rk(p, i + 2, t, c2, c3);
    const Words4 d = philox_rk(p, i + 3, t, c2, c3);
    acc ^= (a.x ^ a.y ^ a.z ^ a.w) ^ (b.x ^ b.y ^ b.z ^ b.w) ^ (c.x ^ c.y ^ c.z ^ c.w) ^
           (d.x ^ d.y ^ d.z ^ d.w);
  }
  for (; i < m; ++i) {
    const Words4 a = philox_rk(p, i, t, c2, c3);
    acc ^= a.x ^ a.y ^ a.z ^ a.w;
  }
  out[t] = acc;
}

cudaError_t launch_philox_throughput(uint64_t seed, uint32_t threads, uint32_t m, uint32_t c2,
                                     uint32_t c3, uint32_t *out, cudaStream_t stream) {
  if (threads == 0) return cudaSuccess;
  RunParams p{};
  p.k0 = (uint32_t)seed;
  p.k1 = (uint32_t)(seed >> 32);
  set_round_keys(p);
  const uint32_t blocks = (threads + 255) / 256;
  philox_throughput_kernel<<<blocks, 256, 0, stream>>>(p, threads, m, c2, c3, out);
  return cudaGetLastError();
}

// ------------------------------------------------------- site function ---
__global__ void sites_kernel(uint32_t policy, uint32_t S, uint32_t W, uint64_t T0,
                             uint64_t count, uint32_t *out) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = site_of(policy, S, W, T0 + i);
}

cudaError_t launch_sites(uint32_t policy, uint32_t S, uint32_t W, uint64_t T0, uint64_t count,
                         uint32_t *out, cudaStream_t stream) {
  if (count == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  uint64_t blocks = (count + 255) / 256;
  const uint64_t cap = (uint64_t)sms * 8;
  if (blocks > cap) blocks = cap;
  sites_kernel<<<(unsigned)blocks, 256, 0, stream>>>(policy, S, W, T0, count, out);
  return cudaGetLastError();
}

}  // namespace hsga
