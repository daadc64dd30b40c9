// hsga_internal.h -- kernel launch interface between the C-ABI runtime
// (hsga_capi.cu) and the kernel translation units.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "hsga_device.cuh"

namespace hsga {

constexpr int kStagedThreads = 256;     // staged streamed kernel (n = 32) block: 8 warps
// 24 resident warps per SM (<= 80 registers), each with one group staged:
// us per generation at 16.8M agents / on 256x256 / 128x128 islands of 32, 24
// warps and 1 stage 72.1 / 11.9 / 4.9, 24 and 2 72.6 / 12.2 / 5.1, 16 and 2
// 72.4 / 11.9 / 6.3, 16 and 3 74.2 / 12.1 / 6.3, 32 and 1 72.1 / 11.2 / 5.6
// (but tournament 5 on 500x500 69.7 against 65.1: 64 registers spill).
constexpr int kStagedBlocksPerSM = 3;
constexpr uint32_t kStagedStages = 1;   // groups in flight per warp
constexpr int kResidentThreads = 128;   // free-running, float and wide kernels: 4 warps
constexpr uint64_t kWaitNs = 1000000000ull; // bounded device wait: 1 s

// The resident kernel cuts the torus into tiles of rows x cols islands (the
// last tile of a row or column may be smaller), tiles_c to a row of tiles.
struct ResidentTile {
  uint32_t rows, cols, tiles_c;
};

struct ResidentPlan {
  ResidentTile tile{0, 0, 1};
  int blocks = 0;          // one per tile
  int threads = 0;
  uint32_t smem = 0;       // dynamic shared memory per block
  bool one_block = false;  // a plain launch of one block that holds the whole grid
};

// err: the grid's device error word (bounded waits report timeouts there).
// plan: from stream_plan for the same parameters.
struct StreamPlan {
  int blocks = 0;   // resident blocks of the whole device
  size_t smem = 0;  // dynamic shared memory per block
  int group = 0;    // islands per warp visit
};
bool stream_plan(const RunParams &p, StreamPlan *out);
cudaError_t launch_step_streamed(const RunParams &p, const StreamPlan &plan, uint32_t G,
                                 bool do_mig, const uint32_t *tin, const uint64_t *sin,
                                 uint32_t *tout, uint64_t *sout, int *err, cudaStream_t stream);

// The same generation for 32-agent islands with the parents staged in shared
// memory by bulk asynchronous copies (hsga_staged.cu); waits report
// timeouts in err.
cudaError_t launch_step_staged(const RunParams &p, uint32_t G, bool do_mig, const uint32_t *tin,
                               const uint64_t *sin, uint32_t *tout, uint64_t *sout, int *err,
                               cudaStream_t stream);

// The same generation for any island size, fitness model and surface width
// (hsga_flat.cu).
bool flat_stream_plan(const RunParams &p, StreamPlan *out);
cudaError_t launch_step_flat(const RunParams &p, const StreamPlan &plan, uint32_t G, bool do_mig,
                             const uint32_t *tin, const uint64_t *sin, uint32_t *tout,
                             uint64_t *sout, int *err, cudaStream_t stream);

// Chooses the resident tiles.  Returns false when the grid does not fit in
// the SMs' shared memory.
bool resident_plan(const RunParams &p, ResidentPlan *out, bool grid_only = false);

cudaError_t launch_step_resident(const RunParams &p, const ResidentPlan &plan, uint32_t G0,
                                 uint32_t ngen, bool premigrated, uint32_t *t, uint64_t *s,
                                 uint64_t *rec, int *err, cudaStream_t stream);

cudaError_t launch_migrate(const RunParams &p, uint32_t G, uint32_t *t, uint64_t *s,
                           uint4 *rec, cudaStream_t stream);

// Scratch that launch_sample needs for k genomes (8-byte aligned; may be 0).
size_t sample_scratch_bytes(uint32_t k);

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
