// hsga_batch.cu -- many independent runs advanced together.
//
// A batch holds runs of uneven size and configuration (grid shape, agents
// per island, policy, mutation rates, seed, generation budget).  One "tick"
// advances every active run by one synchronous generation: a single launch
// covers all of them, so small runs that could not fill the GPU alone share
// it.  The work list is a flat array of (run, first island) items of up to
// kFlatGroup islands each, which warps advance as hsga_flat.cuh describes;
// each run's parameters, planes and start tick live in a device descriptor,
// and the current tick lives in device memory so that a CUDA graph of many
// ticks can be captured once per active set and replayed.  Runs are admitted
// and retired between calls, which is what the serving loop builds on.
// Consecutive ticks overlap by programmatic dependent launch.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <new>
#include <vector>

#include "hsga.h"
#include "hsga_internal.h"
#include "hsga_flat.cuh"

namespace hsga {
namespace {

struct BatchRun {  // device descriptor of one run
  RunParams p;
  uint32_t *trait[2];
  uint64_t *surf[2];
  uint32_t start_tick;  // the run is at generation 0 at this tick
  uint32_t pad;
};

struct WorkItem {
  uint32_t run : 28, group : 4;  // group: islands, up to kFlatGroup
  uint32_t isl0;
};

// 16 warps (<= 128 registers, the runs' round keys among them): 104 ms for a
// 16-run mix; 20 warps, where they spill, 111; 12 warps 110.
constexpr int kBatchBlocksPerSM = 4;

__global__ void __launch_bounds__(kFlatThreads, kBatchBlocksPerSM)
    batch_step_kernel(const BatchRun *__restrict__ runs, const WorkItem *__restrict__ items,
                      uint32_t n_items, const uint32_t *__restrict__ tick_base,
                      uint32_t tick_off, uint32_t stage_bytes, uint32_t may_back,
                      int *__restrict__ err) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[kFlatWarps];
  const uint32_t lane = threadIdx.x & 31u, wib = __shfl_sync(kFull, threadIdx.x >> 5, 0);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (lane == 0) {
    mbar_init(&s_bar[wib], 1);
    mbar_init_fence();
  }
  __syncwarp();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const uint32_t tick = *tick_base + tick_off, par = tick & 1u;
  // Items are strided over the warps, which so sweep the list together and find
  // migrants in L2 (a contiguous share of the list per warp: 123 against 108 ms
  // for a 16-run mix); a run's descriptor is read, and its generator heads and
  // deposit evaluated, only where a warp's next item belongs to another run.
  const uint32_t nwarps = gridDim.x * kFlatWarps;
  uint32_t i = blockIdx.x * kFlatWarps + wib;
  uint32_t phase = 0;
  // odd ticks walk the list backwards where the planes exceed L2: the last
  // children written are the first parents read
  const bool back = may_back != 0u && par != 0u;
  const auto item = [&](uint32_t k) { return items[back ? n_items - 1u - k : k]; };
  WorkItem w = i < n_items ? item(i) : WorkItem{0u, 0u, 0u};
  while (i < n_items) {
    const uint32_t run = w.run;
    const BatchRun &R = runs[run];
    const RunParams &p = R.p;  // read in place (a copy would live in local memory)
    const uint32_t G = tick - R.start_tick;
    const uint32_t *tin = R.trait[par];
    const uint64_t *sin = R.surf[par];
    uint32_t *tout = R.trait[par ^ 1u];
    uint64_t *sout = R.surf[par ^ 1u];
    const bool bulk = (((uintptr_t)tin | (uintptr_t)sin) & 15u) == 0u;
    const FlatDeposit<1> dep = flat_deposit<1>(p, G);
    // 32-bit test, every-generation case first (a 64-bit modulo otherwise)
    const bool do_mig = p.interval == 1u || (p.interval != 0u && G % p.interval == 0u);
    const bool t2 = p.tournament == 2u;
    RoundKeys keys;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
      keys.rk0[r] = p.rk0[r];
      keys.rk1[r] = p.rk1[r];
    }
    FlatStage st = flat_stage(smem + wib * stage_bytes, &s_bar[wib], p.n, 1);
    st.phase = phase;
    flat_heads(keys, p.n, G, st);
    __syncwarp();
    do {
      const uint32_t isl0 = w.isl0, group = w.group;
      i += nwarps;
      if (i < n_items) w = item(i);
      const bool ok = t2 ? flat_group<1, true, 0, false>(p, keys, dep, do_mig, bulk, isl0,
                                                         group, G, false, 0u, false, tin, sin, tout, sout, st)
                         : flat_group<1, false, 0, false>(p, keys, dep, do_mig, bulk, isl0,
                                                          group, G, false, 0u, false, tin, sin, tout, sout, st);
      if (!ok) {
        // give up: record the timeout, wait (bounded) for the copy, leave
        if (lane == 0) {
          atomicCAS(err, 0, kDevErrWaitTimeout);
          mbar_wait(st.bar, st.phase);
        }
        __syncwarp();
        return;
      }
    } while (i < n_items && w.run == run);
    phase = st.phase;
  }
}

__global__ void advance_tick_kernel(uint32_t *tick, uint32_t by) { *tick += by; }

struct HostRun {
  hsga_config cfg;
  RunParams p;
  uint64_t budget = 0;
  uint64_t start_tick = 0;
  uint32_t *trait[2] = {nullptr, nullptr};
  uint64_t *surf[2] = {nullptr, nullptr};
  uint64_t agents = 0;
  bool live = false;
};

constexpr uint64_t kMaxTick = 0xFFFFFFFFull - 64;
constexpr uint32_t kGraphTicks = 64;

}  // namespace
}  // namespace hsga

using namespace hsga;

struct hsga_batch {
  cudaStream_t stream = nullptr;
  bool own_stream = false;  // graphs cannot be captured on the legacy default stream
  AllocHooks alloc{};
  std::vector<HostRun> runs;
  BatchRun *d_runs = nullptr;
  size_t d_runs_cap = 0;
  bool runs_dirty = true;
  WorkItem *d_items = nullptr;
  size_t items_cap = 0;
  uint32_t n_items = 0;
  std::vector<WorkItem> h_items;
  bool items_dirty = true;
  // runs in the work list are ordered by finishing tick, latest first, so
  // the runs still active at any later tick are a prefix of the list:
  // (finishing tick, items up to and including that run)
  std::vector<std::pair<uint64_t, uint32_t>> prefix;
  uint32_t stage_bytes = 0;  // shared memory per warp for the largest island in the list
  uint32_t least = kFlatGroup;  // islands per item (group_of)
  uint32_t back = 0;         // odd ticks walk the list backwards
  int most_per_sm = 1;       // blocks that an SM keeps resident with it
  int per_sm = 0;            // blocks per SM that ticks are launched with
  std::map<int, int> tuned;  // per_sm by log4 of the item count
  uint32_t *d_tick = nullptr;  // the tick, then the kernels' error word
  uint64_t tick = 0;
  cudaGraphExec_t graph = nullptr;
  bool graph_valid = false;
  int sms = 0;
  uint64_t launches = 0, replications = 0, phases = 0;
  int broken = HSGA_OK;  // the first error of a tick that the host has read
};

namespace {

bool active_at(const HostRun &r, uint64_t t) {
  return r.live && r.start_tick <= t && t < r.start_tick + r.budget;
}

void drop_graph(hsga_batch *b) {
  if (b->graph) cudaGraphExecDestroy(b->graph);
  b->graph = nullptr;
  b->graph_valid = false;
}

cudaError_t upload_runs(hsga_batch *b) {
  if (!b->runs_dirty) return cudaSuccess;
  const size_t n = std::max<size_t>(b->runs.size(), 1);
  if (n > b->d_runs_cap) {
    device_free(b->alloc, b->d_runs, b->stream);
    size_t cap = std::max<size_t>(n, 2 * b->d_runs_cap);
    b->d_runs = (BatchRun *)device_alloc(b->alloc, sizeof(BatchRun) * cap, b->stream);
    if (!b->d_runs) {
      b->d_runs_cap = 0;
      return cudaErrorMemoryAllocation;
    }
    b->d_runs_cap = cap;
  }
  std::vector<BatchRun> h(b->runs.size());
  for (size_t i = 0; i < b->runs.size(); ++i) {
    memset(&h[i], 0, sizeof(BatchRun));
    h[i].p = b->runs[i].p;
    for (int j = 0; j < 2; ++j) {
      h[i].trait[j] = b->runs[i].trait[j];
      h[i].surf[j] = b->runs[i].surf[j];
    }
    h[i].start_tick = (uint32_t)b->runs[i].start_tick;
  }
  cudaError_t e = cudaSuccess;
  if (!h.empty())
    e = cudaMemcpyAsync(b->d_runs, h.data(), sizeof(BatchRun) * h.size(),
                        cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);  // h is a local
  b->runs_dirty = false;
  drop_graph(b);
  return e;
}

// Islands per item of a run: a multiple of what starts on 16-byte boundaries.
uint32_t group_of(const HostRun &R, uint32_t least) {
  const uint32_t step = (R.p.n & 3u) == 0u ? 1u : (R.p.n & 1u) == 0u ? 2u : 4u;
  return (least + step - 1u) / step * step;
}

// The fewest islands per item, two at least, that leave every item of the active
// runs a warp of its own, so that a tick is one item's latency; eight if none do.
// One run of 64x64 islands of 32 3.95 us per tick, in items of four 4.60, of eight
// 5.39, with a tournament of 5 4.63, 5.79 and 7.79; 100x100 in items of five 4.98
// and 6.58, of eight 5.91 and 8.51.
uint32_t fewest_islands(const hsga_batch *b) {
  const uint64_t warps = (uint64_t)b->sms * (uint64_t)b->most_per_sm * kFlatWarps;
  for (uint32_t least = 2; least < kFlatGroup; ++least) {
    uint64_t items = 0;
    for (const HostRun &R : b->runs)
      if (active_at(R, b->tick))
        items += (R.p.islands + group_of(R, least) - 1u) / group_of(R, least);
    if (items <= warps) return least;
  }
  return kFlatGroup;
}

// Work list of the runs active at the current tick, ordered by finishing tick,
// latest first.
cudaError_t rebuild_items(hsga_batch *b) {
  std::vector<uint32_t> order;
  for (size_t r = 0; r < b->runs.size(); ++r)
    if (active_at(b->runs[r], b->tick)) order.push_back((uint32_t)r);
  std::stable_sort(order.begin(), order.end(), [&](uint32_t x, uint32_t y) {
    return b->runs[x].start_tick + b->runs[x].budget > b->runs[y].start_tick + b->runs[y].budget;
  });
  b->h_items.clear();
  b->prefix.clear();
  uint32_t n_max = 1;
  uint64_t agents = 0;
  for (uint32_t r : order) {
    agents += b->runs[r].agents;
    n_max = std::max(n_max, b->runs[r].p.n);
  }
  b->stage_bytes = flat_stage_bytes(n_max, 1);
  b->back = exceeds_l2(24u * agents) ? 1u : 0u;  // both planes of 12-byte genomes
  int per_sm = 0;
  cudaError_t e = cudaFuncSetAttribute(batch_step_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_step_kernel, kFlatThreads,
                                                      kFlatWarps * b->stage_bytes);
  if (e != cudaSuccess) return e;
  b->most_per_sm = std::max(per_sm, 1);
  b->least = fewest_islands(b);
  for (uint32_t r : order) {
    const HostRun &R = b->runs[r];
    const uint32_t group = group_of(R, b->least);
    for (uint32_t i0 = 0; i0 < R.p.islands; i0 += group)
      b->h_items.push_back(WorkItem{r, group, i0});
    b->prefix.push_back({R.start_tick + R.budget, (uint32_t)b->h_items.size()});
  }
  const size_t n = b->h_items.size();
  if (n > b->items_cap) {
    device_free(b->alloc, b->d_items, b->stream);
    const size_t cap = std::max(n, 2 * b->items_cap);
    b->d_items = (WorkItem *)device_alloc(b->alloc, sizeof(WorkItem) * cap, b->stream);
    if (!b->d_items) {
      b->items_cap = 0;
      return cudaErrorMemoryAllocation;
    }
    b->items_cap = cap;
  }
  if (n)
    e = cudaMemcpyAsync(b->d_items, b->h_items.data(), sizeof(WorkItem) * n,
                        cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  b->items_dirty = false;
  b->n_items = 0xFFFFFFFFu;  // force a prefix update
  return e;
}

// Items of the runs still active at the current tick (a prefix of the list).
void select_active_prefix(hsga_batch *b) {
  uint32_t n = 0;
  for (const auto &pe : b->prefix) {
    if (pe.first > b->tick) n = pe.second;
    else break;
  }
  if (n != b->n_items) {
    b->n_items = n;
    drop_graph(b);
  }
}

int tick_blocks(const hsga_batch *b) {
  const uint64_t need = ((uint64_t)b->n_items + kFlatWarps - 1) / kFlatWarps;
  const uint64_t most = (uint64_t)b->sms * (uint64_t)std::max(b->per_sm, 1);
  return (int)std::max<uint64_t>(1, std::min<uint64_t>(need, most));
}

cudaError_t launch_tick(hsga_batch *b, uint32_t off) {
  if (!b->n_items) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)tick_blocks(b));
  cfg.blockDim = dim3(kFlatThreads);
  cfg.dynamicSmemBytes = kFlatWarps * b->stage_bytes;
  cfg.stream = b->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, batch_step_kernel, (const BatchRun *)b->d_runs,
                            (const WorkItem *)b->d_items, b->n_items,
                            (const uint32_t *)b->d_tick, off, b->stage_bytes, b->back,
                            (int *)(b->d_tick + 1));
}

// Launch-shape autotuner: each candidate number of resident blocks per SM
// advances the batch by a few real ticks (results do not depend on the shape)
// and the fastest is kept per work-list size class.
cudaError_t autotune(hsga_batch *b, uint64_t *ticks_left) {
  int bucket = 0;
  for (uint32_t x = b->n_items; x > 3; x >>= 2) ++bucket;
  const int before = b->per_sm;
  const auto it = b->tuned.find(bucket);
  if (it != b->tuned.end()) {
    b->per_sm = std::min(it->second, b->most_per_sm);
    if (b->per_sm != before) drop_graph(b);
    return cudaSuccess;
  }
  const uint32_t per_cand = 4;
  const int candidates = std::min(3, b->most_per_sm);
  float best = 1e30f;
  int best_per_sm = b->most_per_sm, tried = 0;
  cudaEvent_t e0, e1;
  cudaError_t e = cudaEventCreate(&e0);
  if (e != cudaSuccess) return e;
  e = cudaEventCreate(&e1);
  if (e != cudaSuccess) {
    cudaEventDestroy(e0);
    return e;
  }
  for (int c = 0; c < candidates && *ticks_left >= per_cand && e == cudaSuccess; ++c) {
    b->per_sm = b->most_per_sm - c;
    e = cudaEventRecord(e0, b->stream);
    for (uint32_t k = 0; k < per_cand && e == cudaSuccess; ++k) e = launch_tick(b, k);
    if (e != cudaSuccess) break;
    advance_tick_kernel<<<1, 1, 0, b->stream>>>(b->d_tick, per_cand);
    cudaEventRecord(e1, b->stream);
    e = cudaEventSynchronize(e1);
    if (e != cudaSuccess) break;
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    b->tick += per_cand;
    *ticks_left -= per_cand;
    b->launches += per_cand + 1;
    ++tried;
    if (ms < best) {
      best = ms;
      best_per_sm = b->per_sm;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  b->per_sm = best_per_sm;
  if (b->per_sm != before) drop_graph(b);
  if (e == cudaSuccess && tried == candidates) b->tuned[bucket] = best_per_sm;
  return e;
}

cudaError_t run_ticks(hsga_batch *b, uint64_t L) {
  cudaError_t e = cudaSuccess;
  if (L >= kGraphTicks) {
    if (!b->graph_valid) {
      cudaGraph_t g = nullptr;
      e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
      if (e != cudaSuccess) return e;
      for (uint32_t k = 0; k < kGraphTicks && e == cudaSuccess; ++k) e = launch_tick(b, k);
      advance_tick_kernel<<<1, 1, 0, b->stream>>>(b->d_tick, kGraphTicks);
      const cudaError_t end = cudaStreamEndCapture(b->stream, &g);
      if (e == cudaSuccess) e = end;
      if (e == cudaSuccess) e = cudaGraphInstantiate(&b->graph, g, 0);
      if (g) cudaGraphDestroy(g);
      if (e != cudaSuccess) return e;
      b->graph_valid = true;
    }
    while (L >= kGraphTicks && e == cudaSuccess) {
      e = cudaGraphLaunch(b->graph, b->stream);
      L -= kGraphTicks;
      b->tick += kGraphTicks;
      b->launches += (uint64_t)kGraphTicks + 1;
    }
  }
  if (e == cudaSuccess && L > 0) {
    for (uint32_t k = 0; k < L && e == cudaSuccess; ++k) e = launch_tick(b, k);
    advance_tick_kernel<<<1, 1, 0, b->stream>>>(b->d_tick, (uint32_t)L);
    b->tick += L;
    b->launches += L + 1;
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  return e;
}

// Waits for the batch's stream, into which the calls before may have put copies
// to the caller, and reads the ticks' error word: a tick whose bounded wait for
// a copy ran out has left islands behind, and no population is valid any more.
int finish(hsga_batch *b) {
  int err = 0;
  cudaError_t e = cudaMemcpyAsync(&err, b->d_tick + 1, sizeof(int), cudaMemcpyDeviceToHost,
                                  b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return HSGA_ERR_CUDA;
  if (err != 0) b->broken = err == kDevErrWaitTimeout ? HSGA_ERR_WAIT_TIMEOUT : HSGA_ERR_DEVICE;
  return b->broken;
}

int free_run(hsga_batch *b, HostRun &R) {
  for (int j = 0; j < 2; ++j) {
    device_free(b->alloc, R.trait[j], b->stream);
    device_free(b->alloc, R.surf[j], b->stream);
    R.trait[j] = nullptr;
    R.surf[j] = nullptr;
  }
  R.live = false;
  b->runs_dirty = true;
  b->items_dirty = true;
  return HSGA_OK;
}

// generation reached by run R at the batch's current tick, and its plane
uint64_t run_generation(const hsga_batch *b, const HostRun &R) {
  const uint64_t t = std::min(b->tick, R.start_tick + R.budget);
  return t - R.start_tick;
}

}  // namespace

extern "C" {

int hsga_batch_create(void *cuda_stream, hsga_batch **out) {
  if (!out) return HSGA_ERR_INVALID_ARG;
  *out = nullptr;
  hsga_batch *b = new (std::nothrow) hsga_batch();
  if (!b) return HSGA_ERR_OOM;
  b->stream = (cudaStream_t)cuda_stream;
  if (!b->stream) {
    if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) {
      delete b;
      return HSGA_ERR_CUDA;
    }
    b->own_stream = true;
  }
  b->alloc = current_allocator();
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev);
  b->d_tick = (uint32_t *)device_alloc(b->alloc, 2 * sizeof(uint32_t), b->stream);
  if (!b->d_tick) {
    if (b->own_stream) cudaStreamDestroy(b->stream);
    delete b;
    return HSGA_ERR_OOM;
  }
  if (cudaMemsetAsync(b->d_tick, 0, 2 * sizeof(uint32_t), b->stream) != cudaSuccess) {
    device_free(b->alloc, b->d_tick, b->stream);
    delete b;
    return HSGA_ERR_CUDA;
  }
  *out = b;
  return HSGA_OK;
}

int hsga_batch_add(hsga_batch *b, const hsga_config *cfg, uint64_t generations,
                   uint32_t *run_id) {
  if (!b || !run_id) return HSGA_ERR_INVALID_ARG;
  const int v = validate_config(cfg);
  if (v != HSGA_OK) return v;
  if (cfg->migration_mode != HSGA_MIGRATION_SYNC || cfg->fitness != HSGA_FITNESS_TRAIT ||
      cfg->surface_words > 1)
    return HSGA_ERR_UNSUPPORTED;
  if (b->tick + generations > kMaxTick) return HSGA_ERR_INVALID_ARG;
  HostRun R;
  R.cfg = *cfg;
  R.p = params_from_config(cfg);
  R.budget = generations;
  R.start_tick = b->tick;
  R.agents = (uint64_t)R.p.islands * R.p.n;
  bool ok = true;
  for (int j = 0; j < 2; ++j) {
    R.trait[j] = (uint32_t *)device_alloc(b->alloc, sizeof(uint32_t) * R.agents, b->stream);
    R.surf[j] = (uint64_t *)device_alloc(b->alloc, sizeof(uint64_t) * R.agents, b->stream);
    ok = ok && R.trait[j] && R.surf[j];
  }
  R.live = true;
  if (!ok) {
    free_run(b, R);
    return HSGA_ERR_OOM;
  }
  // founders in the plane the run starts from
  const int par = (int)(b->tick & 1);
  cudaError_t e = cudaMemsetAsync(R.trait[par], 0, sizeof(uint32_t) * R.agents, b->stream);
  if (e == cudaSuccess)
    e = cudaMemsetAsync(R.surf[par], 0, sizeof(uint64_t) * R.agents, b->stream);
  if (e != cudaSuccess) {
    free_run(b, R);
    return HSGA_ERR_CUDA;
  }
  b->runs.push_back(R);
  b->runs_dirty = true;
  b->items_dirty = true;
  *run_id = (uint32_t)(b->runs.size() - 1);
  return HSGA_OK;
}

int hsga_batch_run(hsga_batch *b, uint64_t ticks) {
  if (!b) return HSGA_ERR_INVALID_ARG;
  if (stream_capturing(b->stream)) return HSGA_ERR_NOT_CAPTURABLE;
  if (b->broken != HSGA_OK) return b->broken;
  cudaError_t e = upload_runs(b);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? HSGA_ERR_OOM : HSGA_ERR_CUDA;
  uint64_t left = ticks;
  while (left > 0) {
    uint64_t phase_end = b->tick + left;
    bool any = false;
    for (const HostRun &R : b->runs)
      if (active_at(R, b->tick)) {
        any = true;
        phase_end = std::min(phase_end, R.start_tick + R.budget);
      }
    if (!any) break;
    // (the runs that others have left behind may do with smaller items)
    if (b->items_dirty || fewest_islands(b) < b->least) {
      e = rebuild_items(b);
      if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? HSGA_ERR_OOM : HSGA_ERR_CUDA;
    }
    select_active_prefix(b);
    b->phases++;
    for (const HostRun &R : b->runs)
      if (active_at(R, b->tick))
        b->replications += R.agents * (phase_end - b->tick);
    uint64_t L = phase_end - b->tick;
    left -= L;
    e = autotune(b, &L);
    if (e == cudaSuccess) e = run_ticks(b, L);
    if (e != cudaSuccess) return HSGA_ERR_CUDA;
  }
  return HSGA_OK;
}

int hsga_batch_info(const hsga_batch *b, uint32_t run, hsga_batch_run_info *out) {
  if (!b || !out || run >= b->runs.size()) return HSGA_ERR_INVALID_ARG;
  const HostRun &R = b->runs[run];
  memset(out, 0, sizeof(*out));
  out->generation = run_generation(b, R);
  out->budget = R.budget;
  out->agents = R.agents;
  out->done = out->generation >= R.budget ? 1u : 0u;
  out->live = R.live ? 1u : 0u;
  return HSGA_OK;
}

int hsga_batch_get_population(hsga_batch *b, uint32_t run, uint32_t *trait, uint64_t *surf) {
  if (!b || !trait || run >= b->runs.size() || !b->runs[run].live) return HSGA_ERR_INVALID_ARG;
  if (stream_capturing(b->stream)) return HSGA_ERR_NOT_CAPTURABLE;
  const HostRun &R = b->runs[run];
  const int par = (int)((R.start_tick + run_generation(b, R)) & 1);
  cudaError_t e = cudaMemcpyAsync(trait, R.trait[par], sizeof(uint32_t) * R.agents,
                                  cudaMemcpyDefault, b->stream);
  if (e == cudaSuccess && surf)
    e = cudaMemcpyAsync(surf, R.surf[par], sizeof(uint64_t) * R.agents, cudaMemcpyDefault,
                        b->stream);
  return e == cudaSuccess ? finish(b) : HSGA_ERR_CUDA;
}

int hsga_batch_sample(hsga_batch *b, uint32_t run, uint32_t k, uint32_t *out_words,
                      uint32_t *out_island_slot) {
  if (!b || run >= b->runs.size() || !b->runs[run].live || (k > 0 && !out_words))
    return HSGA_ERR_INVALID_ARG;
  const HostRun &R = b->runs[run];
  if (k > R.p.islands) return HSGA_ERR_INVALID_ARG;
  if (k == 0) return HSGA_OK;
  if (stream_capturing(b->stream)) return HSGA_ERR_NOT_CAPTURABLE;
  const uint64_t G = run_generation(b, R);
  const int par = (int)((R.start_tick + G) & 1);
  const size_t scratch_bytes = sample_scratch_bytes(k);
  uint32_t *scratch = scratch_bytes
                          ? (uint32_t *)device_alloc(b->alloc, scratch_bytes, b->stream)
                          : nullptr;
  void *held = nullptr;
  uint32_t *staging =
      (uint32_t *)device_alloc16(b->alloc, sizeof(uint32_t) * 6 * k, b->stream, &held);
  if ((scratch_bytes && !scratch) || !staging) {
    device_free(b->alloc, scratch, b->stream);
    device_free(b->alloc, held, b->stream);
    return HSGA_ERR_OOM;
  }
  cudaError_t e = launch_sample(R.p, (uint32_t)G, k, R.trait[par], R.surf[par], staging,
                                staging + 4 * (size_t)k, scratch, b->stream);
  b->launches += sample_launches(k);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(out_words, staging, sizeof(uint32_t) * 4 * k, cudaMemcpyDefault,
                        b->stream);
  if (e == cudaSuccess && out_island_slot)
    e = cudaMemcpyAsync(out_island_slot, staging + 4 * (size_t)k, sizeof(uint32_t) * 2 * k,
                        cudaMemcpyDefault, b->stream);
  device_free(b->alloc, scratch, b->stream);
  device_free(b->alloc, held, b->stream);
  return e == cudaSuccess ? finish(b) : HSGA_ERR_CUDA;
}

int hsga_batch_remove(hsga_batch *b, uint32_t run) {
  if (!b || run >= b->runs.size() || !b->runs[run].live) return HSGA_ERR_INVALID_ARG;
  return free_run(b, b->runs[run]);
}

int hsga_batch_get_stats(const hsga_batch *b, hsga_batch_stats *out) {
  if (!b || !out) return HSGA_ERR_INVALID_ARG;
  memset(out, 0, sizeof(*out));
  out->tick = b->tick;
  out->replications = b->replications;
  out->kernel_launches = b->launches;
  out->phases = b->phases;
  out->threads_per_block = (uint32_t)kFlatThreads;
  out->blocks = b->d_items && !b->items_dirty && b->n_items != 0xFFFFFFFFu
                    ? (uint32_t)tick_blocks(b)
                    : 0u;
  for (const HostRun &R : b->runs) {
    if (R.live) {
      out->live_runs++;
      out->device_bytes += R.agents * 24;
    }
    if (active_at(R, b->tick)) out->active_runs++;
  }
  return HSGA_OK;
}

int hsga_run_footprint(const hsga_config *cfg, uint64_t *bytes) {
  if (!bytes) return HSGA_ERR_INVALID_ARG;
  const int v = validate_config(cfg);
  if (v != HSGA_OK) return v;
  const uint64_t agents = (uint64_t)cfg->rows * cfg->cols * cfg->agents_per_island;
  *bytes = agents * 24 + sizeof(BatchRun) +
           sizeof(WorkItem) * ((uint64_t)cfg->rows * cfg->cols / kFlatGroup + 1);
  return HSGA_OK;
}

int hsga_batch_synchronize(hsga_batch *b) {
  if (!b) return HSGA_ERR_INVALID_ARG;
  if (stream_capturing(b->stream)) return HSGA_ERR_NOT_CAPTURABLE;
  return finish(b);
}

void hsga_batch_destroy(hsga_batch *b) {
  if (!b) return;
  cudaStreamSynchronize(b->stream);
  drop_graph(b);
  for (HostRun &R : b->runs)
    if (R.live) free_run(b, R);
  device_free(b->alloc, b->d_runs, b->stream);
  device_free(b->alloc, b->d_items, b->stream);
  device_free(b->alloc, b->d_tick, b->stream);
  cudaStreamSynchronize(b->stream);
  if (b->own_stream) cudaStreamDestroy(b->stream);
  delete b;
}

}  // extern "C"
