// hsga_flat.cu -- streamed generation kernel for every island size, fitness
// model, surface width and alignment that the staged kernel (32-agent integer
// islands with one surface word) does not serve: one launch advances one synchronous
// generation of the whole grid, steps a1-a6, a warp taking groups of eight
// islands (hsga_flat.cuh).  Consecutive launches overlap by programmatic
// dependent launch, as in the staged kernel.
#include <cuda_runtime.h>

#include "hsga_flat.cuh"

namespace hsga {
namespace {

constexpr int kFlatMaxSmem = 160 * 1024;  // limit set on the kernels; one block uses far less

// LARGE: the instance for grids that a launch takes long over.  Integer fitness
// with at most one surface word is bound by issue and has later generations'
// migration worked out ahead (hsga_moves.cuh; 500x500 islands of 8 24.1 us
// against 28.0, 512x1024 of 24 69.6 against 73.3); binary32 fitness and wide
// surfaces gain nothing from that (256x512 of 32 with two words 29.9 against
// 28.9).
template <int K, bool FLT>
constexpr bool kFlatAhead = K <= 1 && !FLT;

// Warps per SM: 28 fit by themselves where a tournament of 2 and narrow surfaces
// leave the registers, and planning must not take them away; 16 for larger
// tournaments and binary32 (hsga_flat.cuh has the alternatives' times).
template <int K, bool T2, bool FLT, bool LARGE>
constexpr int kFlatBlocksPerSM = LARGE && T2 && !FLT && K <= 2 ? 7 : T2 || (K >= 2 && !FLT) ? 5 : 4;

template <int K, bool T2, int NN, bool FLT, bool LARGE>
__global__ void __launch_bounds__(kFlatThreads, (kFlatBlocksPerSM<K, T2, FLT, LARGE>))
    step_flat_kernel(RunParams p, FlatDeposit<K> dep, uint32_t G, uint32_t group, int migrate,
                     int bulk, int back, Moves mv, const uint32_t *__restrict__ tin,
                     const uint64_t *__restrict__ sin, uint32_t *__restrict__ tout,
                     uint64_t *__restrict__ sout, int *__restrict__ err) {
  constexpr bool AHEAD = LARGE && kFlatAhead<K, FLT>;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[kFlatWarps];
  const uint32_t lane = threadIdx.x & 31u, wib = __shfl_sync(kFull, threadIdx.x >> 5, 0);
  // the next launch may be scheduled now; it waits below for this one
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (lane == 0) {
    mbar_init(&s_bar[wib], 1);
    mbar_init_fence();
  }
  __syncwarp();
  const uint32_t n = NN ? (uint32_t)NN : p.n;
  FlatStage st = flat_stage(smem + wib * flat_stage_bytes(n, K), &s_bar[wib], n, K);
  flat_heads(p, n, G, st);
  __syncwarp();
  const uint32_t groups = (p.islands + group - 1) / group;
  // On small grids the first group's draws come before the wait and overlap the
  // launch before: 20x20 islands of 32, binary32 2.5 us, 3.1 with the wait first;
  // 64x64 with four words 4.2 and 5.0; 128x256 of 48 8.0 and 8.7; 20x20 of 17 2.1
  // and 2.6.  (Large ones lose 2% to the second copy of the loads.)
  if constexpr (LARGE) asm volatile("griddepcontrol.wait;" ::: "memory");
  const uint32_t warp = blockIdx.x * kFlatWarps + wib, nwarps = gridDim.x * kFlatWarps;
  const bool planned = AHEAD && mv.now != nullptr;
  const auto first_of = [&](uint32_t grp) { 
    return (LARGE && back ? groups - 1u - grp : grp) * group;
  };
  const auto move_of = [&](uint32_t grp) {
    return planned && grp < groups
               ? load_move(mv, first_of(grp), min(group, p.islands - first_of(grp)))
               : 0u;
  };
  uint32_t next = move_of(warp);
  [[maybe_unused]] Planner planner(p, mv, warp, nwarps);
  for (uint32_t grp = warp; grp < groups; grp += nwarps) {
    const uint32_t move = next;
    next = move_of(grp + nwarps);
    if (!flat_group<K, T2, NN, FLT, LARGE>(p, p, dep, migrate != 0, bulk != 0, first_of(grp),
                                           group, G, planned, move, !LARGE && grp == warp, tin,
                                           sin, tout, sout, st)) {
      // give up: record the timeout, wait (bounded) for the copy, leave (once
      // the moves that later launches read are written)
      if (lane == 0) {
        atomicCAS(err, 0, kDevErrWaitTimeout);
        mbar_wait(st.bar, st.phase);
      }
      __syncwarp();
      break;
    }
    if constexpr (AHEAD) planner.template visit<NN>(p, p, mv, G, group);
  }
  if constexpr (AHEAD) planner.template rest<NN>(p, p, mv, G);
}

// Resident blocks and the shared memory to ask for per block: padded so that
// no further block fits on an SM, since the next launch, scheduled early,
// would park one there beside the running ones.
template <int K, bool T2, int NN, bool FLT, bool LARGE>
bool flat_plan(const RunParams &p, StreamPlan *out) {
  const size_t need = kFlatWarps * flat_stage_bytes(p.n, K);
  int dev = 0, sms = 0, per_sm = 0, sm_smem = 0, reserved = 0;
  const auto fn = step_flat_kernel<K, T2, NN, FLT, LARGE>;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kFlatMaxSmem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kFlatThreads, need) !=
          cudaSuccess ||
      per_sm < 1)
    return false;
  const size_t pad = ((size_t)sm_smem / (per_sm + 1) + 255u) & ~(size_t)127;
  const size_t used = need + (size_t)reserved;  // as the SM counts it
  // Islands per group: the size (whose groups all start on a 16-byte boundary)
  // that takes the warps the least work, ceil(groups / warps) rounds of a
  // group each, counting 1.2 islands' worth for a group's migration draws and
  // staging.  4,096 groups of 8 on 3,040 warps take two rounds of 8; groups of
  // 6 two rounds of 6.
  const uint32_t warps = (uint32_t)(sms * per_sm) * kFlatWarps;
  const uint32_t step = (p.n & 3u) == 0u ? 1u : (p.n & 1u) == 0u ? 2u : 4u;
  double best = 1e30;
  for (uint32_t g = 4; g <= kFlatGroup; g += step) {
    const uint32_t groups = (p.islands + g - 1) / g;
    const double cost = (double)((groups + warps - 1) / warps) * (g + 1.2);
    if (cost <= best) {
      best = cost;
      out->group = (int)g;
    }
  }
  out->blocks = sms * per_sm;
  out->back = LARGE && planes_exceed_l2(p);
  // ahead only if the warps take at least two groups each (one: 128x256 of 48)
  out->moves_ahead =
      LARGE && kFlatAhead<K, FLT> && p.islands / (uint32_t)out->group >= 2u * warps;
  out->large = kFlatAhead<K, FLT> ? out->moves_ahead : out->back;
  out->smem = pad > used && pad * per_sm <= (size_t)sm_smem && pad <= kFlatMaxSmem
                  ? pad - (size_t)reserved
                  : need;
  return true;
}

template <int K, bool T2, int NN, bool FLT>
cudaError_t launch_flat_t(const RunParams &p, const StreamPlan &plan, const FlatDeposit<K> &dep,
                          uint32_t G, bool do_mig, const Moves &mv, const uint32_t *tin,
                          const uint64_t *sin, uint32_t *tout, uint64_t *sout, int *err,
                          cudaStream_t stream) {
  const uint32_t groups = (p.islands + plan.group - 1) / plan.group;
  const uint32_t need = (groups + kFlatWarps - 1) / kFlatWarps;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(need < (uint32_t)plan.blocks ? need : (uint32_t)plan.blocks);
  cfg.blockDim = dim3(kFlatThreads);
  cfg.dynamicSmemBytes = plan.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const int bulk = (((uintptr_t)tin | (uintptr_t)sin | (uintptr_t)sout) & 15u) == 0 ? 1 : 0;
  const int back = plan.back && (G & 1u) ? 1 : 0;
  return cudaLaunchKernelEx(&cfg,
                            plan.large ? step_flat_kernel<K, T2, NN, FLT, true>
                                       : step_flat_kernel<K, T2, NN, FLT, false>,
                            p, dep, G, (uint32_t)plan.group, do_mig ? 1 : 0, bulk, back, mv, tin,
                            sin, tout, sout, err);
}

// Calls F::run<K, T2, NN, FLT>(args...) for a configuration.
template <class F, int K, class... A>
auto flat_pick(const RunParams &p, A &&...args) {
  const bool t2 = p.tournament == 2, n32 = p.n == 32;
  if (p.flt)  // general tournament path only
    return n32 ? F::template run<K, false, 32, true>(p, args...)
               : F::template run<K, false, 0, true>(p, args...);
  if constexpr (K > 1) {  // aligned 32-agent islands with at most one word: the staged kernel
    if (n32)
      return t2 ? F::template run<K, true, 32, false>(p, args...)
                : F::template run<K, false, 32, false>(p, args...);
  }
  return t2 ? F::template run<K, true, 0, false>(p, args...)
            : F::template run<K, false, 0, false>(p, args...);
}

template <class F, class... A>
auto flat_pick_words(const RunParams &p, A &&...args) {
  if (p.policy == HSGA_NONE) return flat_pick<F, 0>(p, args...);
  if (p.words == 4) return flat_pick<F, 4>(p, args...);
  if (p.words == 2) return flat_pick<F, 2>(p, args...);
  return flat_pick<F, 1>(p, args...);
}

struct Plan {
  template <int K, bool T2, int NN, bool FLT>
  static bool run(const RunParams &p, StreamPlan *out) {
    return flat_plan<K, T2, NN, FLT, true>(p, out) &&
           (out->large || flat_plan<K, T2, NN, FLT, false>(p, out));
  }
};

struct Launch {
  template <int K, bool T2, int NN, bool FLT>
  static cudaError_t run(const RunParams &p, const StreamPlan &plan, uint32_t G, bool do_mig,
                         const Moves &mv, const uint32_t *tin, const uint64_t *sin, uint32_t *tout, uint64_t *sout,
                         int *err, cudaStream_t stream) {
    return launch_flat_t<K, T2, NN, FLT>(p, plan, flat_deposit<K>(p, G), G, do_mig, mv, tin, sin,
                                         tout, sout, err, stream);
  }
};

}  // namespace

bool flat_stream_plan(const RunParams &p, StreamPlan *out) {
  return flat_pick_words<Plan>(p, out);
}

cudaError_t launch_step_flat(const RunParams &p, const StreamPlan &plan, uint32_t G, bool do_mig,
                             const Moves &mv, const uint32_t *tin, const uint64_t *sin,
                             uint32_t *tout, uint64_t *sout, int *err, cudaStream_t stream) {
  return flat_pick_words<Launch>(p, plan, G, do_mig, mv, tin, sin, tout, sout, err, stream);
}

}  // namespace hsga
