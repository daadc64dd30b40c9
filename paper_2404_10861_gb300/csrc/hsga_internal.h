// hsga_internal.h -- kernel launch interface between the C-ABI runtime
// (hsga_capi.cu) and the kernel translation units.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "hsga_device.cuh"

namespace hsga {

constexpr int kStagedThreads = 256;     // staged streamed kernel (n = 32) block: 8 warps
// 16 resident warps per SM (<= 128 registers), a group of 8 islands each, all
// of its children in flight: us per generation at 16.8M agents / tournament 5
// on 500x500 islands / on 256x256 islands, 16 warps 67.3 / 60.8 / 11.2; 24 warps
// with the children of 4 islands in flight 68.6 / 62.9 / 11.0, of 8 (80
// registers spill) 68.2 / 69.2 / 10.7; 32 with 4 72.7 / 72.5 / 11.1; 16 with
// groups of 16 in two halves 70.5 / 61.3 / 10.8.  Groups of 6 on 24 warps, before:
// 71.7 / 65.7 / 11.9.
constexpr int kStagedBlocksPerSM = 2;
constexpr int kSmallStagedBlocksPerSM = 3;  // groups of four islands: 24 warps
constexpr uint32_t kStagedStages = 2;   // most groups in flight per warp
constexpr int kFreeThreads = 128;       // free-running kernels: 4 warps
constexpr uint64_t kWaitNs = 1000000000ull; // bounded device wait: 1 s

// The resident kernel cuts the torus into tiles of rows x cols islands (the
// last tile of a row or column may be smaller), tiles_c to a row of tiles.
struct ResidentTile {
  uint32_t rows, cols, tiles_c;
  uint32_t stride, slots;  // record slots per tile (0: one per island, in order), per buffer
  uint32_t by_cols;        // consecutive blocks take the tiles of a column, not of a row
};

struct ResidentPlan {
  ResidentTile tile{0, 0, 1, 0, 0, 0};
  int blocks = 0;          // one per tile
  int threads = 0;
  uint32_t smem = 0;       // dynamic shared memory per block
  bool one_block = false;  // a plain launch of one block that holds the whole grid
  bool warp = false;       // an island per warp in registers (hsga_resident_warp.cu)
};

// Migration moves of a streamed run, worked out ahead of their generation
// (hsga_moves.cuh).  now: this generation's, [island][direction], or NULL: the
// launch derives them.  next: written, from leave_next, for the next
// generation; leave_after: written for the one after it; or NULL.
struct Moves {
  const uint16_t *now = nullptr;
  uint16_t *next = nullptr;
  const uint8_t *leave_next = nullptr;
  uint8_t *leave_after = nullptr;
};

// err: the grid's device error word (bounded waits report timeouts there).
// plan: from stream_plan for the same parameters.
struct StreamPlan {
  int blocks = 0;   // resident blocks of the whole device
  size_t smem = 0;  // dynamic shared memory per block
  int group = 0;    // islands per warp visit
  bool moves_ahead = false;  // launches of a run plan the migration of later ones
  bool back = false;         // odd generations walk the islands from last to first
  bool large = false;        // the flat kernel's instance for large grids
  bool staged = false;       // the staged kernel, else the flat one
};
// aligned: the population planes start on 16-byte boundaries.
bool stream_plan(const RunParams &p, bool aligned, StreamPlan *out);

// Whether parents and children do not fit in L2 together.  Then every other
// generation walks the islands from last to first: it begins with the parents
// that the one before wrote last and finds part of them in L2 (256x512 islands
// of 32 with four surface words: 46.2 us per generation, 54.9 without; grids
// that fit lose 1%).
bool planes_exceed_l2(const RunParams &p);
bool exceeds_l2(uint64_t bytes);
cudaError_t launch_step_streamed(const RunParams &p, const StreamPlan &plan, uint32_t G,
                                 bool do_mig, const Moves &mv, const uint32_t *tin,
                                 const uint64_t *sin, uint32_t *tout, uint64_t *sout, int *err,
                                 cudaStream_t stream);

// The same generation for 32-agent islands with the parents staged in shared
// memory by bulk asynchronous copies (hsga_staged.cu); waits report
// timeouts in err.
bool staged_stream_plan(const RunParams &p, StreamPlan *out);
cudaError_t launch_step_staged(const RunParams &p, const StreamPlan &plan, uint32_t G, bool do_mig,
                               const Moves &mv, const uint32_t *tin, const uint64_t *sin,
                               uint32_t *tout, uint64_t *sout, int *err, cudaStream_t stream);

// The same generation for any island size, fitness model and surface width
// (hsga_flat.cu).
bool flat_stream_plan(const RunParams &p, StreamPlan *out);
cudaError_t launch_step_flat(const RunParams &p, const StreamPlan &plan, uint32_t G, bool do_mig,
                             const Moves &mv, const uint32_t *tin, const uint64_t *sin, uint32_t *tout,
                             uint64_t *sout, int *err, cudaStream_t stream);

// Chooses the resident tiles.  Returns false when the grid does not fit in
// the SMs' shared memory.
bool resident_plan(const RunParams &p, ResidentPlan *out, bool grid_only = false);

cudaError_t launch_step_resident(const RunParams &p, const ResidentPlan &plan, uint32_t G0,
                                 uint32_t ngen, bool premigrated, uint32_t *t, uint64_t *s,
                                 uint64_t *rec, int *err, cudaStream_t stream);

bool resident_warp_plan(const RunParams &p, ResidentPlan *out, bool grid_only);
cudaError_t launch_step_resident_warp(const RunParams &p, const ResidentPlan &plan, uint32_t G0,
                                      uint32_t ngen, bool premigrated, uint32_t *t, uint64_t *s,
                                      uint64_t *rec, int *err, cudaStream_t stream);

cudaError_t launch_migrate(const RunParams &p, uint32_t G, uint32_t *t, uint64_t *s,
                           uint4 *rec, cudaStream_t stream);

// Scratch that launch_sample needs for k genomes (8-byte aligned; may be 0).
size_t sample_scratch_bytes(uint32_t k);
uint32_t sample_launches(uint32_t k);  // kernels that it launches

// T: per-genome deposition counters (free-running grids) written as word 3,
// or NULL to write G.
cudaError_t launch_sample(const RunParams &p, uint32_t G, uint32_t k, const uint32_t *t,
                          const uint64_t *s, uint32_t *out_words, uint32_t *out_is,
                          uint32_t *scratch, cudaStream_t stream, const uint32_t *T = nullptr);

// Wide surfaces (hsga_wide.cu): the field(s) a synchronous generation
// writes (word < 0: none).
struct WideDeposit {
  int word1;
  uint32_t shift1;
  int word2;
  uint32_t shift2;
};
WideDeposit wide_deposit_for(const RunParams &p, uint64_t G);
cudaError_t launch_migrate_wide(const RunParams &p, uint32_t G, uint32_t *t, uint64_t *s,
                                uint64_t *rec, cudaStream_t stream);
cudaError_t launch_gather_wide(const RunParams &p, uint32_t G, uint32_t k, const uint32_t *t,
                               const uint64_t *s, const uint32_t *where, uint32_t *out,
                               cudaStream_t stream);
// Free-running generations (hsga_async.cu).  slice: generations each warp
// advances an island octet by per visit (1: the whole grid one generation at
// a time).
cudaError_t launch_step_buffered(const RunParams &p, uint32_t G0, uint32_t ngen, uint32_t slice,
                                 uint32_t *t, uint64_t *s, uint32_t *T, uint64_t *mail,
                                 uint32_t *ack, uint4 *inbuf, uint4 *chst, uint32_t *log,
                                 uint32_t log_G0, uint32_t log_gens, cudaStream_t stream);
cudaError_t launch_step_async(const RunParams &p, uint32_t G0, uint32_t ngen, uint32_t slice,
                              uint32_t *t, uint64_t *s, uint32_t *T, uint64_t *rec,
                              uint32_t *seen, uint32_t *log, uint32_t log_G0, uint32_t log_gens,
                              cudaStream_t stream);

// Device memory through the registered allocator hooks (hsga_capi.cu).
struct AllocHooks {
  hsga_alloc_fn alloc;
  hsga_free_fn free_fn;
  void *ctx;
};
AllocHooks current_allocator();
void *device_alloc(const AllocHooks &h, size_t bytes, cudaStream_t s);
void *device_alloc16(const AllocHooks &h, size_t bytes, cudaStream_t s, void **held);
void device_free(const AllocHooks &h, void *ptr, cudaStream_t s);
bool device_pointer(const void *ptr);

// Whether `s` is being captured into a CUDA graph (calls that wait for their
// stream return HSGA_ERR_NOT_CAPTURABLE then; defined in hsga_capi.cu).
bool stream_capturing(cudaStream_t s);

// Configuration checks and kernel parameters (defined in hsga_capi.cu).
int validate_config(const hsga_config *c);
RunParams params_from_config(const hsga_config *c);

cudaError_t launch_wait_probe(const uint64_t *record, uint32_t seq, uint64_t limit_ns, int *err,
                              uint64_t *out, cudaStream_t stream);
cudaError_t launch_philox_sweep(uint64_t seed, uint32_t c0, uint32_t count, uint32_t c1,
                                uint32_t c2, uint32_t c3, uint32_t *out, cudaStream_t stream);
cudaError_t launch_philox_throughput(uint64_t seed, uint32_t threads, uint32_t m, uint32_t c2,
                                     uint32_t c3, uint32_t *out, cudaStream_t stream);
cudaError_t launch_sites(uint32_t policy, uint32_t S, uint32_t W, uint64_t T0, uint64_t count,
                         uint32_t *out, cudaStream_t stream);

}  // namespace hsga
