// hsga_wide.cu -- explicit migration and sampling with surfaces of 2 or 4
// 64-bit words (128- or 256-bit fields; the paper draws a 256-bit field,
// section "Surface-based Hereditary Stratigraphy Algorithms", and names more
// and wider differentiae as the remedy for reconstruction precision, "Results ›
// Clade Reconstruction Trial").  Generations run in hsga_flat.cu.
//
// Surfaces are agent-major: word w of agent a at surf[a K + w]; site s
// occupies bits [s b mod 64, s b mod 64 + b) of word floor(s b / 64).  The
// explicit a1 + a2 pair uses (K + 1)-word records: trait | direction << 32,
// then the surface words.
#include <cuda_runtime.h>

#include "hsga_internal.h"
#include "hsga_island.cuh"

namespace hsga {
namespace {

template <int K>
__global__ void emigrate_wide_kernel(RunParams p, uint32_t G, const uint32_t *__restrict__ t,
                                     const uint64_t *__restrict__ s,
                                     uint64_t *__restrict__ rec) {
  const uint32_t isl = blockIdx.x * blockDim.x + threadIdx.x;
  if (isl >= p.islands) return;
  const Words4 m = philox_rk(p, kSlotEmigrant, isl, G, kPurposeMigration);
  const size_t a = (size_t)isl * p.n + uindex(m.x, p.n);
  uint64_t *r = rec + (size_t)isl * (K + 1);
  r[0] = (uint64_t)t[a] | ((uint64_t)(m.y >> 30) << 32);
#pragma unroll
  for (int w = 0; w < K; ++w) r[1 + w] = s[a * K + w];
}

template <int K>
__global__ void immigrate_wide_kernel(RunParams p, uint32_t G, uint32_t *__restrict__ t,
                                      uint64_t *__restrict__ s,
                                      const uint64_t *__restrict__ rec) {
  const uint32_t isl = blockIdx.x * blockDim.x + threadIdx.x;
  if (isl >= p.islands) return;
  const Words4 v = philox_rk(p, kSlotImmigrant, isl, G, kPurposeMigration);
  const uint32_t place[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (uint32_t d = 0; d < 4; ++d) {
    const uint64_t *r = rec + (size_t)neighbour(p, isl, d) * (K + 1);
    if ((uint32_t)(r[0] >> 32) != ((d + 2u) & 3u)) continue;
    const size_t a = (size_t)isl * p.n + uindex(place[d], p.n);
    t[a] = (uint32_t)r[0];
#pragma unroll
    for (int w = 0; w < K; ++w) s[a * K + w] = r[1 + w];
  }
}

// Sample records of 2 + 2K words (trait, surface words as (low, high)
// pairs, T = G) from (island, slot) pairs.
__global__ void gather_wide_kernel(uint32_t k, uint32_t n, uint32_t K, uint32_t G,
                                   const uint32_t *__restrict__ t,
                                   const uint64_t *__restrict__ s,
                                   const uint32_t *__restrict__ where,
                                   uint32_t *__restrict__ out) {
  const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= k) return;
  const size_t a = (size_t)where[2 * j] * n + where[2 * j + 1];
  uint32_t *o = out + (size_t)j * (2 + 2 * K);
  o[0] = t[a];
  for (uint32_t w = 0; w < K; ++w) {
    o[1 + 2 * w] = (uint32_t)s[a * K + w];
    o[2 + 2 * w] = (uint32_t)(s[a * K + w] >> 32);
  }
  o[1 + 2 * K] = G;
}

template <int K>
void launch_migrate_wide_t(const RunParams &p, uint32_t G, uint32_t *t, uint64_t *s,
                           uint64_t *rec, cudaStream_t stream) {
  const uint32_t blocks = (p.islands + 255) / 256;
  emigrate_wide_kernel<K><<<blocks, 256, 0, stream>>>(p, G, t, s, rec);
  immigrate_wide_kernel<K><<<blocks, 256, 0, stream>>>(p, G, t, s, rec);
}

}  // namespace

WideDeposit wide_deposit_for(const RunParams &p, uint64_t G) {
  WideDeposit d{-1, 0, -1, 0};
  const uint32_t k = p.coarsen;
  if (k > 1 && (G % k) != 0) return d;
  const uint64_t T = k > 1 ? G / k : G;
  const uint32_t a = site_of(p.policy, p.S, p.W, T);
  if (a < p.S) {
    d.word1 = (int)(a * p.bits / 64);
    d.shift1 = a * p.bits % 64;
  }
  if (p.policy == HSGA_HYBRID) {
    const uint32_t half = p.S / 2;
    const uint32_t b = site_of(HSGA_TILTED, half, p.W, T);
    if (b < half) {
      d.word2 = (int)((half + b) * p.bits / 64);
      d.shift2 = (half + b) * p.bits % 64;
    }
  }
  return d;
}

cudaError_t launch_migrate_wide(const RunParams &p, uint32_t G, uint32_t *t, uint64_t *s,
                                uint64_t *rec, cudaStream_t stream) {
  if (p.words == 2)
    launch_migrate_wide_t<2>(p, G, t, s, rec, stream);
  else
    launch_migrate_wide_t<4>(p, G, t, s, rec, stream);
  return cudaGetLastError();
}

cudaError_t launch_gather_wide(const RunParams &p, uint32_t G, uint32_t k, const uint32_t *t,
                               const uint64_t *s, const uint32_t *where, uint32_t *out,
                               cudaStream_t stream) {
  gather_wide_kernel<<<(k + 255) / 256, 256, 0, stream>>>(k, p.n, p.words, G, t, s, where, out);
  return cudaGetLastError();
}

}  // namespace hsga
