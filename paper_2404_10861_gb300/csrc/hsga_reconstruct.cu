// hsga_reconstruct.cu -- phylogeny reconstruction from sampled surfaces on
// the GPU.
//
// Section "Distributed Phylogenetic Tracking" (and "Results › On-hardware
// Trial", which reconstructs from 10,000-genome samples): each genome's
// retained differentiae, read in ascending deposition time, are a path in a
// trie; genomes share a path exactly as long as they share ancestry (up to
// differentia collisions), and the trie with its unifurcations collapsed is
// the reconstructed tree.  Node times: the root -1, a node reached after d
// differentiae the time of the d-th retained deposition, a leaf the
// generation count T.
//
// GPU formulation (all samples elapsed the same T, so they retain the same
// deposition times):
//   1. keys:  each surface's differentiae permuted into time order, oldest in
//             the most significant bits (of a key as wide as the surface), so
//             that numeric order is path order;
//   2. sort:  least-significant-digit radix sort of (key, sample) over the
//             key's significant bits (8-bit digits, stable).  Up to
//             kSmallSort one-word keys are sorted by one block in shared
//             memory; above, each pass counts digits per tile, scans the
//             counts of each digit over the tiles, and scatters;
//   3. lcp:   L[j] = number of leading differentiae shared by sorted keys j
//             and j + 1;
//   4. tree:  the collapsed trie's internal nodes are exactly the maximal
//             runs ("lcp intervals") of L >= l that contain an L == l, for
//             each l >= 1 -- the same correspondence that turns a suffix array
//             with its lcp array into a suffix tree.  An interval's parent is
//             the interval holding the larger of the two lcps just outside
//             it; a leaf hangs from the interval holding the larger of its
//             two neighbouring lcps; value 0 (or nothing) is the root.  An
//             interval is named by its leftmost position, the first lcp at
//             most l after the nearest smaller one.  The searches this needs
//             run inside blocks of 1,024 positions, against 32 values at a
//             time on bit planes; what lies outside a block is known per
//             value (an lcp is at most 256) from a scan over the blocks.
//             Nodes are numbered in the order of the naming positions, from
//             per-warp masks and counts.
//
// Latency bounds a sample of 10,000 genomes: 7 launches of 2.5-31 us, one
// allocation and one wait for the node count (33, 17 and 2 before); from host
// arrays to host arrays 127 us, 306 before.  1M genomes, all on the device:
// 202 us (1,662 before), of which the three-pass sort 90, lcps 12, intervals
// 34, nodes 17; 16.8M genomes 2.05 ms (41 before).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <vector>

#include "hsga.h"
#include "hsga_internal.h"

namespace hsga {
namespace {

constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr int kMaxWords = 4;
constexpr int kMaxFields = 64 * kMaxWords;

struct KeyPlan {
  uint32_t fields;           // retained differentiae m
  uint32_t bits;             // differentia width b
  uint32_t src[kMaxFields];  // bit offset of field j (time order) in the surface
};

// A key of K words: field j (time order) at key bits [j b, (j + 1) b)
// counted from the most significant bit of word 0.
struct KeyWords {
  uint64_t *w[kMaxWords];
};

template <int K>
__device__ __forceinline__ void make_key(const KeyPlan &kp, const uint64_t *__restrict__ surf,
                                         uint64_t (&out)[K]) {
  const uint64_t mask = (1ull << kp.bits) - 1;  // bits <= 16
  const uint32_t per_word = 64u / kp.bits;
  uint64_t s0 = K == 1 ? surf[0] : 0ull;
  uint32_t j = 0;
#pragma unroll
  for (int w = 0; w < K; ++w) {
    const uint32_t end = min(kp.fields, j + per_word);
    uint64_t acc = 0;
    const uint32_t first = j;
    for (; j < end; ++j) {
      const uint32_t src = kp.src[j];
      if constexpr (K > 1) s0 = surf[src >> 6];
      acc = (acc << kp.bits) | ((s0 >> (src & 63u)) & mask);
    }
    const uint32_t used = (j - first) * kp.bits;
    out[w] = used == 0u ? 0ull : acc << (64u - used);
  }
}

template <int K>
__global__ void make_keys_kernel(const __grid_constant__ KeyPlan kp,
                                 const uint64_t *__restrict__ surf, uint32_t k, KeyWords key,
                                 uint32_t *__restrict__ val) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= k) return;
  uint64_t out[K];
  make_key<K>(kp, surf + (size_t)i * K, out);
#pragma unroll
  for (int w = 0; w < K; ++w) key.w[w][i] = out[w];
  val[i] = i;
}

// ------------------------------------------------------------ radix sort ---
// Lanes of the warp with the same digit, from eight votes: a match
// instruction takes one step per distinct value (47 against 42 us for keys and
// sort of 10,000 samples by one block).
__device__ __forceinline__ uint32_t same_digit(uint32_t digit) {
  uint32_t peers = kAll;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const bool bit = digit >> b & 1u;
    const uint32_t set = __ballot_sync(kAll, bit);
    peers &= bit ? set : ~set;
  }
  return peers;
}

// A warp ranks its elements of one digit pass stably: 32 at a time, an
// element's rank among equal digits is (its warp's count so far) + (earlier
// lanes with the same digit).  cnt: the warp's 256 counts.
__device__ __forceinline__ uint32_t warp_rank(uint32_t *cnt, uint32_t digit, bool live,
                                              uint32_t lane) {
  const uint32_t peers = same_digit(digit) & __ballot_sync(kAll, live);
  const uint32_t old = cnt[digit];
  __syncwarp();
  const uint32_t before = __popc(peers & ((1u << lane) - 1u));
  if (live && before == 0u) cnt[digit] = old + __popc(peers);
  __syncwarp();
  return old + before;
}

// Exclusive sum of v over the block's threads in thread order (blockDim.x a
// multiple of 32, at most 1,024); sums: 32 words of shared memory.
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t *sums) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (uint32_t o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kAll, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31u) sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t t = lane < warps ? sums[lane] : 0u;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kAll, t, o);
      if (lane >= o) t += y;
    }
    if (lane < warps) sums[lane] = t;
  }
  __syncthreads();
  const uint32_t r = x - v + (warp ? sums[warp - 1u] : 0u);
  __syncthreads();
  return r;
}

constexpr uint32_t kSmallSort = 12288;  // one-word keys that one block sorts
constexpr uint32_t kSmallItems = kSmallSort / 1024;

constexpr size_t small_sort_smem(uint32_t k) {
  const size_t n = (k + 1023u) / 1024u * 1024u;
  return n * 8 + 2 * n * 2 + 32 * 256 * 4 + 32 * 4;
}

// Keys stay in place in shared memory and their 16-bit positions are sorted;
// the sorted keys and samples go out at the end.
__global__ void __launch_bounds__(1024)
    small_sort_kernel(const uint64_t *__restrict__ key_in, uint32_t k, uint32_t passes,
                      uint64_t *__restrict__ key_out, uint32_t *__restrict__ val_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint32_t rounds = (k + 1023u) / 1024u, n = rounds * 1024u;
  uint64_t *const key = (uint64_t *)smem;
  uint16_t *idx = (uint16_t *)(key + n), *idx2 = idx + n;
  uint32_t *const cnt = (uint32_t *)(idx2 + n);  // [warp][digit]
  uint32_t *const sums = cnt + 32 * 256;
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  for (uint32_t i = t; i < k; i += 1024u) {
    key[i] = key_in[i];
    idx[i] = (uint16_t)i;
  }
  __syncthreads();
  const uint32_t first = warp * rounds * 32u + lane;  // this warp's run of positions
  for (uint32_t ps = 0; ps < passes; ++ps) {
    const uint32_t byte = 7u - (passes - 1u - ps);  // little endian: byte 7 is the top digit
    for (uint32_t c = t; c < 32u * 256u; c += 1024u) cnt[c] = 0;
    __syncthreads();
    uint32_t held[kSmallItems], rank[kSmallItems];  // position of the key, digit << 16
#pragma unroll
    for (uint32_t r = 0; r < kSmallItems; ++r) {
      if (r < rounds) {
        const uint32_t e = first + 32u * r;
        const bool live = e < k;
        const uint32_t i = live ? idx[e] : 0u;
        const uint32_t d = live ? ((const unsigned char *)(key + i))[byte] : 0u;
        held[r] = i | (d << 16);
        rank[r] = warp_rank(cnt + 256u * warp, d, live, lane);
      }
    }
    __syncthreads();
    // thread 4d + q: digit d, warps 8q .. 8q + 7 -- thread order is (digit, warp) order
    const uint32_t d = t >> 2, w0 = 8u * (t & 3u);
    uint32_t s = 0;
#pragma unroll
    for (uint32_t w = 0; w < 8; ++w) s += cnt[256u * (w0 + w) + d];
    uint32_t run = block_exclusive(s, sums);
#pragma unroll
    for (uint32_t w = 0; w < 8; ++w) {
      const uint32_t c = cnt[256u * (w0 + w) + d];
      cnt[256u * (w0 + w) + d] = run;
      run += c;
    }
    __syncthreads();
#pragma unroll
    for (uint32_t r = 0; r < kSmallItems; ++r)
      if (r < rounds && first + 32u * r < k)
        idx2[cnt[256u * warp + (held[r] >> 16)] + rank[r]] = (uint16_t)held[r];
    __syncthreads();
    uint16_t *const x = idx;
    idx = idx2;
    idx2 = x;
  }
  for (uint32_t e = t; e < k; e += 1024u) {
    key_out[e] = key[idx[e]];
    val_out[e] = idx[e];
  }
}

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;

// Digit counts of every tile, digit-major; key: the key word that holds this
// pass's digit.
__global__ void __launch_bounds__(kSortThreads)
    digit_histogram_kernel(const uint64_t *__restrict__ key, uint32_t k, uint32_t shift,
                           uint32_t ntiles, uint32_t *__restrict__ hist) {
  __shared__ uint32_t cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  // equal digits of a warp (the rule, not the exception, in an evolved
  // population) are counted by one of its lanes
  const uint32_t base = blockIdx.x * kSortTile, lane = threadIdx.x & 31u;
  uint32_t d[kSortItems];
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const uint32_t e = base + r * kSortThreads + threadIdx.x;
    d[r] = e < k ? (uint32_t)(key[e] >> shift) & 0xFFu : 0u;
  }
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const bool live = base + r * kSortThreads + threadIdx.x < k;
    const uint32_t peers = same_digit(d[r]) & __ballot_sync(kAll, live);
    if (live && (peers & ((1u << lane) - 1u)) == 0u)
      atomicAdd(&cnt[d[r]], (uint32_t)__popc(peers));
  }
  __syncthreads();
  hist[threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
}

// Block d: exclusive scan of digit d's counts over the tiles, in place, and
// their total.
__global__ void __launch_bounds__(256)
    digit_scan_kernel(uint32_t *__restrict__ hist, uint32_t ntiles, uint32_t *__restrict__ total) {
  __shared__ uint32_t sums[32];
  __shared__ uint32_t carry;
  uint32_t *const row = hist + (size_t)blockIdx.x * ntiles;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (uint32_t i0 = 0; i0 < ntiles; i0 += 256u) {
    const uint32_t i = i0 + threadIdx.x;
    const uint32_t v = i < ntiles ? row[i] : 0u;
    const uint32_t x = block_exclusive(v, sums) + carry;
    if (i < ntiles) row[i] = x;
    __syncthreads();
    if (threadIdx.x == 255u) carry = x + v;
    __syncthreads();
  }
  if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

// Stable scatter of one digit pass.
template <int K>
__global__ void __launch_bounds__(kSortThreads)
    digit_scatter_kernel(KeyWords key_in, const uint32_t *__restrict__ val_in, uint32_t k,
                         uint32_t dword, uint32_t shift, uint32_t ntiles,
                         const uint32_t *__restrict__ offsets, const uint32_t *__restrict__ total,
                         KeyWords key_out, uint32_t *__restrict__ val_out) {
  constexpr int kWarps = kSortThreads / 32;
  __shared__ uint32_t cnt[kWarps][256];
  __shared__ uint32_t sums[32];
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) cnt[w][t] = 0;
  __syncthreads();
  const uint64_t *const dkey = key_in.w[dword];
  const uint32_t first = blockIdx.x * kSortTile + warp * (32u * kSortItems) + lane;
  uint32_t rank[kSortItems];  // rank in the warp | digit << 16
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const uint32_t e = first + 32u * r;
    rank[r] = e < k ? (uint32_t)(dkey[e] >> shift) & 0xFFu : 0u;
  }
#pragma unroll
  for (int r = 0; r < kSortItems; ++r)
    rank[r] = warp_rank(cnt[warp], rank[r], first + 32u * r < k, lane) | (rank[r] << 16);
  const uint32_t base = block_exclusive(total[t], sums);  // ends with a block barrier
  {  // thread t owns digit t: the tile's elements of it, warp by warp
    uint32_t run = base + offsets[(size_t)t * ntiles + blockIdx.x];
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t c = cnt[w][t];
      cnt[w][t] = run;
      run += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const uint32_t e = first + 32u * r;
    if (e < k) {
      const uint32_t pos = cnt[warp][rank[r] >> 16] + (rank[r] & 0xFFFFu);
#pragma unroll
      for (int w = 0; w < K; ++w) key_out.w[w][pos] = key_in.w[w][e];
      val_out[pos] = val_in[e];
    }
  }
}

// ----------------------------------------------------------------- lcp ---
constexpr uint32_t kBlockPos = 1024;  // lcp positions of a block
constexpr uint32_t kPlanes = 9;       // bits of an lcp (at most kMaxFields)
constexpr uint32_t kNoLcp = (1u << kPlanes) - 1;  // beyond the last: never smaller

// Lanes whose value, given as bit planes, is below x.
template <class Planes>
__device__ __forceinline__ uint32_t below(const Planes &plane, uint32_t x) {
  uint32_t lt = 0, eq = kAll;
#pragma unroll
  for (int b = kPlanes - 1; b >= 0; --b) {
    const uint32_t bit = plane(b), want = (x >> b & 1u) ? kAll : 0u;
    lt |= eq & want & ~bit;
    eq &= ~(want ^ bit);
  }
  return lt;
}

__device__ __forceinline__ uint32_t top_bit(uint32_t m) { return 31u - (uint32_t)__clz((int)m); }
__device__ __forceinline__ uint32_t low_bit(uint32_t m) { return (uint32_t)__ffs((int)m) - 1u; }

// A block's 1,024 lcps for searches: in shared memory, the bit planes of every
// warp's 32 values and (row 32) of the 32 warps' minima.  Positions are
// relative to the block.  (Planes of the own warp and the minima in registers
// left room for one block per SM instead of two: 38 against 34 us at 1M.)
using LcpPlanes = uint32_t[33][kPlanes];

struct BlockLcps {
  const uint32_t (*planes)[kPlanes];

  // planes_, wmin: shared memory; ends with a block barrier.
  __device__ __forceinline__ BlockLcps(uint32_t v, LcpPlanes &planes_, uint32_t *wmin)
      : planes(planes_) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    put(v, planes_[warp], lane);
    const uint32_t m = __reduce_min_sync(kAll, v);
    if (lane == 0) wmin[warp] = m;
    __syncthreads();
    if (warp == 0) put(wmin[lane], planes_[32], lane);
    __syncthreads();
  }
  static __device__ __forceinline__ void put(uint32_t v, uint32_t *row, uint32_t lane) {
    uint32_t mine = 0;
#pragma unroll
    for (uint32_t b = 0; b < kPlanes; ++b) {
      const uint32_t set = __ballot_sync(kAll, v >> b & 1u);
      mine = lane == b ? set : mine;
    }
    if (lane < kPlanes) row[lane] = mine;
  }
  __device__ __forceinline__ uint32_t in_warp(uint32_t w, uint32_t x) const {
    return below([&](int b) { return planes[w][b]; }, x);
  }
  __device__ __forceinline__ uint32_t warps(uint32_t x) const {  // with a value below x
    return in_warp(32u, x);
  }
  // First position >= q (q < 1,024) with a value below x, or -1.
  __device__ __forceinline__ int32_t first_from(uint32_t q, uint32_t x) const {
    const uint32_t w = q >> 5, here = in_warp(w, x) & (kAll << (q & 31u));
    if (here) return (int32_t)(32u * w + low_bit(here));
    const uint32_t later = warps(x) & ~((2u << w) - 1u);
    if (!later) return -1;
    const uint32_t w2 = low_bit(later);
    return (int32_t)(32u * w2 + low_bit(in_warp(w2, x)));
  }
};

// What the blocks around it tell a block about each value v (row v, column
// block): last / first, the nearest position before / after the block with a
// smaller lcp (-1: none); open, the position that names the interval of value
// v that runs into the block (-1: none does, or it has no v yet).
struct Carries {
  int32_t *last, *first, *open;
  uint32_t blocks;
};

// lcps, and per block and value: last / first position with a smaller lcp (-1:
// none), and the first with this one after the last smaller one (-1: none).
template <int K>
__global__ void __launch_bounds__(kBlockPos, 2)
    lcp_kernel(KeyWords key, uint32_t n, uint32_t fields, uint32_t bits,
               uint16_t *__restrict__ L, Carries c) {
  __shared__ LcpPlanes planes;
  __shared__ uint32_t wmin[32];
  const uint32_t base = blockIdx.x * kBlockPos, j = base + threadIdx.x;
  uint32_t v = kNoLcp;
  if (j < n) {
    v = fields;
    bool differ = false;
#pragma unroll
    for (int w = 0; w < K; ++w) {
      const uint64_t x = key.w[w][j] ^ key.w[w][j + 1];
      if (!differ && x) {
        v = min(fields, (w * 64u + (uint32_t)__clzll((long long)x)) / bits);
        differ = true;
      }
    }
    L[j] = (uint16_t)v;
  }
  const BlockLcps bl(v, planes, wmin);
  if (threadIdx.x <= fields) {
    const uint32_t x = threadIdx.x;
    const uint32_t ws = bl.warps(x);
    int32_t last = -1, first = -1;
    if (ws) {
      const uint32_t w1 = top_bit(ws), w0 = low_bit(ws);
      last = (int32_t)(32u * w1 + top_bit(bl.in_warp(w1, x)));
      first = (int32_t)(32u * w0 + low_bit(bl.in_warp(w0, x)));
    }
    const int32_t open =
        last + 1 < (int32_t)kBlockPos ? bl.first_from((uint32_t)(last + 1), x + 1u) : -1;
    const size_t at = (size_t)x * c.blocks + blockIdx.x;
    c.last[at] = last < 0 ? -1 : (int32_t)base + last;
    c.first[at] = first < 0 ? -1 : (int32_t)base + first;
    c.open[at] = open < 0 ? -1 : (int32_t)base + open;
  }
}

// Row v: from each block's own answers to what the blocks before it (last,
// open) and after it (first) tell it, in place.  One warp per row and
// direction; the loads of kAhead chunks of 32 blocks are in flight together.
constexpr uint32_t kAhead = 8;

__device__ __forceinline__ void carry_forward(int32_t *last, int32_t *open, uint32_t blocks,
                                              uint32_t lane) {
  int32_t run_last = -1, run_open = -1;
  for (uint32_t c0 = 0; c0 < blocks; c0 += 32u * kAhead) {
    int32_t ls[kAhead], os[kAhead];
#pragma unroll
    for (uint32_t i = 0; i < kAhead; ++i) {
      const uint32_t b = c0 + 32u * i + lane;
      ls[i] = b < blocks ? last[b] : -1;
      os[i] = b < blocks ? open[b] : -1;
    }
#pragma unroll
    for (uint32_t i = 0; i < kAhead; ++i) {
      const uint32_t b = c0 + 32u * i + lane;
      const int32_t l = ls[i], o = os[i];
      // blocks with a smaller lcp start afresh; the others keep what is open
      const uint32_t resets = __ballot_sync(kAll, l >= 0), opens = __ballot_sync(kAll, o >= 0);
      const uint32_t lower = (1u << lane) - 1u;
      const uint32_t r = resets & lower;
      const uint32_t from = r ? top_bit(r) : 0u;  // the last reset before this block
      const uint32_t since = opens & lower & (r ? kAll << from : kAll);
      const int32_t l_from = __shfl_sync(kAll, l, from);
      const int32_t o_first = __shfl_sync(kAll, o, since ? low_bit(since) : 0u);
      const int32_t in_last = r ? l_from : run_last;
      const int32_t in_open = !r && run_open >= 0 ? run_open : since ? o_first : -1;
      if (b < blocks) {
        last[b] = in_last;
        open[b] = in_open;
      }
      // the state after this chunk's last block
      const int32_t out_last = l >= 0 ? l : in_last;
      const int32_t out_open = l >= 0 ? o : in_open >= 0 ? in_open : o;
      run_last = __shfl_sync(kAll, out_last, 31);
      run_open = __shfl_sync(kAll, out_open, 31);
    }
  }
}

__device__ __forceinline__ void carry_backward(int32_t *first, uint32_t blocks, uint32_t lane) {
  int32_t run = -1;
  const uint32_t step = 32u * kAhead;
  for (uint32_t c0 = (blocks - 1u) / step * step;; c0 -= step) {
    int32_t fs[kAhead];
#pragma unroll
    for (uint32_t i = 0; i < kAhead; ++i) {
      const uint32_t b = c0 + 32u * i + lane;
      fs[i] = b < blocks ? first[b] : -1;
    }
#pragma unroll
    for (int i = kAhead - 1; i >= 0; --i) {
      const uint32_t b = c0 + 32u * i + lane;
      const int32_t f = fs[i];
      const uint32_t have = __ballot_sync(kAll, f >= 0) & ~((2u << lane) - 1u);
      const int32_t near = __shfl_sync(kAll, f, have ? low_bit(have) : 0u);
      if (b < blocks) first[b] = have ? near : run;
      const int32_t out = f >= 0 ? f : have ? near : run;
      run = __shfl_sync(kAll, out, 0);
    }
    if (c0 == 0u) break;
  }
}

__global__ void __launch_bounds__(64) carry_kernel(Carries c) {
  const size_t row = (size_t)blockIdx.x * c.blocks;
  const uint32_t lane = threadIdx.x & 31u;
  if (threadIdx.x < 32u) carry_forward(c.last + row, c.open + row, c.blocks, lane);
  else carry_backward(c.first + row, c.blocks, lane);
}

// Node numbering: position q names an interval iff bit q & 31 of mask[q >> 5]
// is set; its rank is base[q >> 10] + before[q >> 5] + the set bits below it.
struct NodeRanks {
  uint32_t *mask, *before, *base;
};

__device__ __forceinline__ uint32_t node_rank(const NodeRanks &nr, uint32_t q) {
  return nr.base[q >> 10] + nr.before[q >> 5] + __popc(nr.mask[q >> 5] & ((1u << (q & 31u)) - 1u));
}

// For each lcp position: rep, the position that names its interval; where
// that is the position itself and the value at least 1, also PS and NS, the
// previous and next strictly smaller positions.
__global__ void __launch_bounds__(kBlockPos, 2)
    intervals_kernel(const uint16_t *__restrict__ L, uint32_t n, Carries c,
                     int32_t *__restrict__ ps_out, int32_t *__restrict__ ns_out,
                     uint32_t *__restrict__ rep_out, NodeRanks nr) {
  __shared__ LcpPlanes planes;
  __shared__ uint32_t wmin[32];
  __shared__ uint32_t sums[32];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t base = blockIdx.x * kBlockPos, j = base + threadIdx.x;
  const uint32_t v = j < n ? L[j] : kNoLcp;
  const BlockLcps bl(v, planes, wmin);
  bool names = false;
  if (j < n) {
    const uint32_t lt = bl.in_warp(warp, v), ltw = bl.warps(v);
    const uint32_t left = lt & ((1u << lane) - 1u), leftw = ltw & ((1u << warp) - 1u);
    const size_t at = (size_t)v * c.blocks + blockIdx.x;
    int32_t ps, rep;
    if (left || leftw) {
      const uint32_t w = left ? warp : top_bit(leftw);
      const uint32_t q = 32u * w + top_bit(left ? left : bl.in_warp(w, v));
      ps = (int32_t)(base + q);
      // the first position after PS with a value of at most v (j at the latest)
      rep = (int32_t)base + bl.first_from(q + 1u, v + 1u);
    } else {
      ps = c.last[at];
      rep = c.open[at];
      if (rep < 0) rep = (int32_t)base + bl.first_from(0u, v + 1u);
    }
    rep_out[j] = (uint32_t)rep;
    names = rep == (int32_t)j && v >= 1u;
    if (names) {
      const uint32_t right = lt & ~((2u << lane) - 1u), rightw = ltw & ~((2u << warp) - 1u);
      int32_t ns;
      if (right) ns = (int32_t)(base + 32u * warp + low_bit(right));
      else if (rightw) {
        const uint32_t w = low_bit(rightw);
        ns = (int32_t)(base + 32u * w + low_bit(bl.in_warp(w, v)));
      } else {
        ns = c.first[at];
      }
      ps_out[j] = ps;
      ns_out[j] = ns;
    }
  }
  const uint32_t mask = __ballot_sync(kAll, names);
  const uint32_t x = block_exclusive(lane == 0 ? (uint32_t)__popc(mask) : 0u, sums);
  if (lane == 0 && j < n) {
    nr.mask[j >> 5] = mask;
    nr.before[j >> 5] = x;
  }
  if (threadIdx.x == kBlockPos - 1u) nr.base[blockIdx.x] = x;
}

// Exclusive prefix sum of n counts in place and their total, one block (each
// thread scans a contiguous chunk).
__global__ void __launch_bounds__(1024)
    scan_counts_kernel(uint32_t *__restrict__ a, uint32_t n, uint32_t *__restrict__ total) {
  __shared__ uint32_t sums[32];
  const uint32_t chunk = (n + 1023u) / 1024u;
  const uint32_t lo = min(n, threadIdx.x * chunk), hi = min(n, lo + chunk);
  uint32_t s = 0;
  for (uint32_t i = lo; i < hi; ++i) s += a[i];
  uint32_t run = block_exclusive(s, sums);
  if (threadIdx.x == 1023u) *total = run + s;
  for (uint32_t i = lo; i < hi; ++i) {
    const uint32_t v = a[i];
    a[i] = run;
    run += v;
  }
}

struct FieldTimes {
  int64_t t[kMaxFields];
};

// Node ids: 0 the root, 1 + rank of the naming position an interval, then the
// leaves in sorted order.
__global__ void nodes_kernel(const uint16_t *__restrict__ L, uint32_t k,
                             const int32_t *__restrict__ ps, const int32_t *__restrict__ ns,
                             const uint32_t *__restrict__ rep, NodeRanks nr,
                             const uint32_t *__restrict__ val,
                             const uint32_t *__restrict__ internal,
                             const __grid_constant__ FieldTimes times, int64_t T,
                             int64_t *__restrict__ parent, int64_t *__restrict__ time,
                             uint32_t *__restrict__ leaf_of_sample) {
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= k) return;
  const uint32_t n = k - 1u;
  const uint32_t total = *internal;
  if (p == 0) {
    parent[0] = -1;
    time[0] = -1;
  }
  const int32_t Lp = p < n ? (int32_t)L[p] : -1;
  if (p < n && (nr.mask[p >> 5] >> (p & 31u) & 1u)) {
    const uint32_t node = 1u + node_rank(nr, p);
    const int32_t a = ps[p], b = ns[p];
    const int32_t La = a >= 0 ? (int32_t)L[a] : -1, Lb = b >= 0 ? (int32_t)L[b] : -1;
    int64_t par = 0;
    if (La > 0 || Lb > 0) par = 1 + (int64_t)node_rank(nr, rep[La >= Lb ? a : b]);
    parent[node] = par;
    time[node] = times.t[Lp - 1];
  }
  const int32_t La = p >= 1u ? (int32_t)L[p - 1u] : -1;
  int64_t par = 0;
  if (La > 0 || Lp > 0) par = 1 + (int64_t)node_rank(nr, rep[La >= Lp ? p - 1u : p]);
  const uint32_t node = 1u + total + p;
  parent[node] = par;
  time[node] = T;
  leaf_of_sample[val[p]] = node;
}

inline uint32_t blocks_for(uint64_t n, uint32_t threads) {
  return (uint32_t)((n + threads - 1) / threads);
}

// Device memory of the current device that a kernel can read in place.
bool readable_here(const void *ptr) {
  int dev = 0;
  cudaPointerAttributes attr;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&attr, ptr) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return attr.type == cudaMemoryTypeDevice && attr.device == dev && ((uintptr_t)ptr & 7u) == 0;
}

// Keys of k surfaces, sorted: key[*cur], val[*cur].
template <int K>
cudaError_t sort_keys(const KeyPlan &kp, const uint64_t *surf, uint32_t k, KeyWords (&key)[2],
                      uint32_t *(&val)[2], uint32_t *hist, uint32_t *digits, int *cur,
                      cudaStream_t st) {
  // over the significant bits only (the top fields * bits, rounded up to whole
  // 8-bit digits, which then never straddle two key words)
  const uint32_t passes = (kp.fields * kp.bits + 7) / 8;
  *cur = 0;
  make_keys_kernel<K><<<blocks_for(k, 128), 128, 0, st>>>(kp, surf, k, key[0], val[0]);
  if (K == 1 && k <= kSmallSort) {
    // the limit for every k: other threads launch too
    const cudaError_t e =
        cudaFuncSetAttribute(small_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)small_sort_smem(kSmallSort));
    if (e != cudaSuccess) return e;
    small_sort_kernel<<<1, 1024, small_sort_smem(k), st>>>(key[0].w[0], k, passes, key[1].w[0], val[1]);
    *cur = 1;
    return cudaGetLastError();
  }
  const uint32_t ntiles = blocks_for(k, kSortTile);
  for (uint32_t i = 0; i < passes; ++i) {
    const uint32_t top = 8 * (passes - 1 - i);  // digit's first bit from the top
    const uint32_t dword = top / 64, shift = 64 - top % 64 - 8;
    digit_histogram_kernel<<<ntiles, kSortThreads, 0, st>>>(key[*cur].w[dword], k, shift, ntiles,
                                                            hist);
    digit_scan_kernel<<<256, 256, 0, st>>>(hist, ntiles, digits);
    digit_scatter_kernel<K><<<ntiles, kSortThreads, 0, st>>>(
        key[*cur], val[*cur], k, dword, shift, ntiles, hist, digits, key[1 - *cur],
        val[1 - *cur]);
    *cur = 1 - *cur;
  }
  return cudaGetLastError();
}

}  // namespace
}  // namespace hsga

using namespace hsga;

int hsga_reconstruct(const uint64_t *surf, uint32_t k, uint32_t surface_words, uint32_t policy,
                     uint32_t differentia_bits, uint32_t W, uint64_t generations,
                     uint32_t deposit_interval,
                     int64_t *parent_out, int64_t *time_out, uint32_t *leaf_of_sample,
                     uint32_t capacity, uint32_t *n_nodes, void *cuda_stream) {
  const uint32_t b = differentia_bits;
  if (!surf || !parent_out || !time_out || !leaf_of_sample || !n_nodes) return HSGA_ERR_INVALID_ARG;
  const uint32_t K = surface_words > 1 ? surface_words : 1;
  if (k == 0 || k > (1u << 28) || !(b == 1 || b == 2 || b == 4 || b == 8 || b == 16))
    return HSGA_ERR_INVALID_ARG;
  if (!(K == 1 || K == 2 || K == 4)) return HSGA_ERR_INVALID_ARG;
  if (policy > HSGA_HYBRID || policy == HSGA_NONE) return HSGA_ERR_INVALID_ARG;
  const uint64_t need_nodes = 2ull * k + 1;
  if (capacity < need_nodes) return HSGA_ERR_INVALID_ARG;
  if (stream_capturing((cudaStream_t)cuda_stream)) return HSGA_ERR_NOT_CAPTURABLE;
  // retained deposition times in ascending order (the same for every sample)
  const uint32_t S = 64 * K / b;
  const uint64_t kk = deposit_interval > 1 ? deposit_interval : 1;
  const uint64_t T = (generations + kk - 1) / kk;
  std::vector<int64_t> dep(S);
  if (hsga_lookup(policy, S, W, T, dep.data()) != HSGA_OK) return HSGA_ERR_INVALID_ARG;
  std::vector<uint32_t> order;
  for (uint32_t s = 0; s < S; ++s)
    if (dep[s] >= 0) order.push_back(s);
  std::stable_sort(order.begin(), order.end(),
                   [&](uint32_t x, uint32_t y) { return dep[x] < dep[y]; });
  KeyPlan kp{};
  kp.fields = (uint32_t)order.size();
  kp.bits = b;
  FieldTimes times{};
  for (uint32_t j = 0; j < kp.fields; ++j) {
    kp.src[j] = order[j] * b;
    times.t[j] = dep[order[j]] * (int64_t)kk;
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  AllocHooks al = current_allocator();
  const uint32_t ntiles = blocks_for(k, kSortTile);
  const uint32_t n = k - 1;  // lcp positions
  const uint32_t nblocks = blocks_for(n, kBlockPos);
  const bool dev_out = device_pointer(parent_out);
  const bool in_place = readable_here(surf);
  // scratch: one allocation, carved up
  size_t bytes = 0;
  const auto take = [&](size_t want) {
    const size_t at = bytes;
    bytes += (want + 255u) & ~(size_t)255u;
    return at;
  };
  size_t at_key[2][kMaxWords] = {}, at_val[2];
  for (int h = 0; h < 2; ++h) {
    for (uint32_t w = 0; w < K; ++w) at_key[h][w] = take(8ull * k);
    at_val[h] = take(4ull * k);
  }
  const size_t at_hist = take(4ull * 256 * ntiles), at_digits = take(4 * 256);
  const size_t at_surf = in_place ? 0 : take(8ull * k * K);
  const size_t at_L = take(2ull * n);
  const uint32_t rows = kp.fields + 1;
  const size_t at_carry = take(12ull * rows * nblocks);
  const size_t at_ps = take(4ull * n), at_ns = take(4ull * n), at_rep = take(4ull * n);
  const size_t at_mask = take(4ull * 32 * nblocks), at_before = take(4ull * 32 * nblocks);
  const size_t at_base = take(4ull * nblocks), at_total = take(4);
  const size_t at_parent = dev_out ? 0 : take(8 * need_nodes);
  const size_t at_time = dev_out ? 0 : take(8 * need_nodes);
  const size_t at_leaf = dev_out ? 0 : take(4ull * k);
  unsigned char *const mem = (unsigned char *)device_alloc(al, bytes, st);
  if (!mem) return HSGA_ERR_OOM;
  KeyWords key[2] = {};
  uint32_t *val[2];
  for (int h = 0; h < 2; ++h) {
    for (uint32_t w = 0; w < K; ++w) key[h].w[w] = (uint64_t *)(mem + at_key[h][w]);
    val[h] = (uint32_t *)(mem + at_val[h]);
  }
  uint16_t *const L = (uint16_t *)(mem + at_L);
  int32_t *const carry = (int32_t *)(mem + at_carry);
  const size_t per = (size_t)rows * nblocks;
  const Carries carries{carry, carry + per, carry + 2 * per, nblocks};
  uint32_t *const hist = (uint32_t *)(mem + at_hist), *const digits = (uint32_t *)(mem + at_digits);
  int32_t *const ps = (int32_t *)(mem + at_ps), *const ns = (int32_t *)(mem + at_ns);
  uint32_t *const rep = (uint32_t *)(mem + at_rep), *const total = (uint32_t *)(mem + at_total);
  const NodeRanks nr{(uint32_t *)(mem + at_mask), (uint32_t *)(mem + at_before),
                     (uint32_t *)(mem + at_base)};
  int64_t *const dparent = dev_out ? parent_out : (int64_t *)(mem + at_parent);
  int64_t *const dtime = dev_out ? time_out : (int64_t *)(mem + at_time);
  uint32_t *const dleaf = dev_out ? leaf_of_sample : (uint32_t *)(mem + at_leaf);
  cudaError_t e = cudaSuccess;
  const uint64_t *dsurf = surf;
  if (!in_place) {
    e = cudaMemcpyAsync(mem + at_surf, surf, 8ull * k * K, cudaMemcpyDefault, st);
    dsurf = (const uint64_t *)(mem + at_surf);
  }
  int cur = 0;
  if (e == cudaSuccess)
    e = K == 1   ? sort_keys<1>(kp, dsurf, k, key, val, hist, digits, &cur, st)
        : K == 2 ? sort_keys<2>(kp, dsurf, k, key, val, hist, digits, &cur, st)
                 : sort_keys<4>(kp, dsurf, k, key, val, hist, digits, &cur, st);
  if (e == cudaSuccess) {
    if (n > 0) {
      if (K == 1)
        lcp_kernel<1><<<nblocks, kBlockPos, 0, st>>>(key[cur], n, kp.fields, b, L, carries);
      else if (K == 2)
        lcp_kernel<2><<<nblocks, kBlockPos, 0, st>>>(key[cur], n, kp.fields, b, L, carries);
      else
        lcp_kernel<4><<<nblocks, kBlockPos, 0, st>>>(key[cur], n, kp.fields, b, L, carries);
      carry_kernel<<<rows, 64, 0, st>>>(carries);
      intervals_kernel<<<nblocks, kBlockPos, 0, st>>>(L, n, carries, ps, ns, rep, nr);
    }
    scan_counts_kernel<<<1, 1024, 0, st>>>(nr.base, n > 0 ? nblocks : 0u, total);
    nodes_kernel<<<blocks_for(k, 256), 256, 0, st>>>(L, k, ps, ns, rep, nr, val[cur],
                                                     total, times, (int64_t)generations, dparent,
                                                     dtime, dleaf);
    e = cudaGetLastError();
  }
  uint32_t internal = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&internal, total, 4, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  const uint32_t nodes = 1 + internal + k;
  if (e == cudaSuccess && !dev_out) {
    e = cudaMemcpyAsync(parent_out, dparent, 8ull * nodes, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(time_out, dtime, 8ull * nodes, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(leaf_of_sample, dleaf, 4ull * k, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e != cudaSuccess) cudaStreamSynchronize(st);  // the scratch may still be in use
  device_free(al, mem, st);
  *n_nodes = nodes;
  return e == cudaSuccess ? HSGA_OK : HSGA_ERR_CUDA;
}
