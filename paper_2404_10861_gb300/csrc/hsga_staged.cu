// hsga_staged.cu -- streamed generation kernel for 32-agent islands with the
// parents staged in shared memory by bulk asynchronous copies.
//
// One launch advances one synchronous generation of the whole grid (steps
// a1-a6 of the paper's cycle, section "Asynchronous Island-model Genetic
// Algorithm": migration, then evaluation, tournament selection, mutation and
// the surface update).  A persistent grid of warps walks the islands in groups
// of eight (four directions of eight islands fill a warp's lanes).  Each warp
// stages a group's parents in shared memory; one lane copies them in with
// cp.async.bulk (1,024 bytes of traits and 2,048 bytes of surfaces, both
// contiguous in the island-major planes), completing on the stage's mbarrier,
// while the group's replication draws are evaluated.  The bytes in flight
// cost no registers, and the tournament reads the parents from shared memory:
// two 4-byte loads for the candidates' fitness and one 8-byte load for the
// winner's surface per child (warp shuffles of the fitness in their place:
// 70.4 against 65.6 us with a tournament of 5).  Immigrants are gathered from
// the neighbours' parent planes one group ahead and land with one shared-memory
// store each.  Children go straight to the child planes with streaming stores.
//
// Of the replication blocks' first three rounds only two products depend on
// the island, one of them the same on every lane (lane_head).  Where warps take
// several groups, a launch works out the migration of the two generations after
// it between its groups and finds its own worked out (hsga_moves.cuh).
//
// What bounds it, per generation at 16.8M agents: 64.9 us, of which 59.4 are
// its 24 bytes per agent at the measured copy bandwidth; half of the issue
// slots are taken.  Groups of six, each deriving its own migration: 71.7, and 69
// without any load or store; before the reads of a group came ahead of its
// stores: 75.2.  Tournament 5 on 500x500 islands 59.8 (65.7, 71.8), untracked
// 16.8M 54.2 (60.0), 256x256 islands 10.7 (11.9); these are bound by issue.
//
// Consecutive generations overlap at the launch boundary (programmatic
// dependent launch): a launch lets the next one be scheduled as soon as it
// starts, and the next one initialises its barriers and generator heads and
// draws its first groups, then waits (griddepcontrol.wait) for this launch to complete and its
// writes to be visible before it touches either population plane.
//
// Waits on a stage are bounded (1 s of %globaltimer): on expiry the warp
// records HSGA_ERR_WAIT_TIMEOUT in the grid's error word, waits (bounded
// again) for its own copies still in flight, and leaves.
#include <cuda_runtime.h>

#include "hsga_stage.cuh"

namespace hsga {
namespace {

struct StagedLaunch {
  uint32_t G;
  uint32_t back;    // walk the groups from the last to the first
  uint32_t stages;  // groups staged per warp, 1 .. kStagedStages
  Moves mv;
};

template <bool TRACKED, bool T2, bool TWO, bool DEL, bool MIG, uint32_t GR>
__global__ void __launch_bounds__(kStagedThreads, (kStagedBlocks<GR>))
    step_staged_kernel(RunParams p, Deposit dep, StagedLaunch l, const uint32_t *__restrict__ tin,
                       const uint64_t *__restrict__ sin, uint32_t *__restrict__ tout,
                       uint64_t *__restrict__ sout, int *__restrict__ err) {
  const uint32_t G = l.G, stages = l.stages;
  const Moves &mv = l.mv;
  extern __shared__ __align__(128) unsigned char s_ring[];  // the ring (kRingBytes), padded
  __shared__ __align__(8) uint64_t s_bar[kStagedWarps][kStagedStages];
  const uint32_t lane = threadIdx.x & 31u, wib = __shfl_sync(kFull, threadIdx.x >> 5, 0);
  const uint32_t warp = blockIdx.x * kStagedWarps + wib;
  const uint32_t nwarps = gridDim.x * kStagedWarps;
  const uint32_t nfull = p.islands / GR;
  unsigned char *ring = s_ring + (size_t)wib * kStagedStages * kStageBytes<GR>;
  uint64_t *bar = s_bar[wib];
  constexpr uint32_t kTx = kTraitBytes<GR> + (TRACKED ? kSurfBytes<GR> : 0u);

  // stage st holds a group's traits (1,024 B) then its surfaces (2,048 B)
  auto issue = [&](uint32_t isl0, uint32_t st) {  // one lane
    unsigned char *dst = ring + st * kStageBytes<GR>;
    proxy_fence();
    mbar_expect_tx(&bar[st], kTx);
    bulk_load(dst, tin + (size_t)isl0 * 32u, kTraitBytes<GR>, &bar[st]);
    if constexpr (TRACKED)
      bulk_load(dst + kTraitBytes<GR>, sin + (size_t)isl0 * 32u, kSurfBytes<GR>, &bar[st]);
  };

  // the next launch may be scheduled now; it waits below for this one
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (lane == 0) {
#pragma unroll
    for (uint32_t st = 0; st < stages; ++st) mbar_init(&bar[st], 1);
    mbar_init_fence();
  }
  const uint32_t first = (l.back ? nfull - 1u - warp : warp) * GR;
  const uint32_t skip = l.back ? 0u - nwarps * GR : nwarps * GR;
  const LaneHead head = lane_head(p, lane, G, kPurposeReplicate);
  [[maybe_unused]] LaneHead head2;  // candidates 2-5
  if constexpr (!T2) head2 = lane_head(p, lane, G, kPurposeReplicate + 1u);
  // Only groups of eight plan ahead: a round of smaller ones is too short.  The
  // first group's draws come before the wait, beside the launch before: 16x16
  // islands 2.0 us, 2.5 after it, 64x64 2.3 and 3.9 (tournament 5 4.2 and 5.6),
  // 256x256 10.7 and 11.2, 16.8M agents 64.9 and 66.0.
  constexpr bool PLAN = GR == kStageGroup;
  const bool planned = PLAN && mv.now != nullptr;
  const auto move_of = [&](uint32_t isl) {
    return planned ? (uint32_t)mv.now[(size_t)isl * 4u + lane] : derive_move<GR>(p, isl, G);
  };
  uint32_t move = 0;  // the lane's in the next group to gather for
  Words4 w[GR];
  if (warp < nfull) {
    if constexpr (MIG && !PLAN) move = move_of(first);
#pragma unroll
    for (uint32_t i = 0; i < GR; ++i) w[i] = lane_tail(p, head, first + i);
  }
  // the previous launch (which wrote this launch's parents and read the
  // plane this one writes) has completed and its writes are visible
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (lane == 0) {
#pragma unroll
    for (uint32_t st = 0; st < stages; ++st)
      if (warp + st * nwarps < nfull) issue(first + st * skip, st);
  }
  __syncwarp();

  // The immigrants of a group are gathered while the group before it is
  // replicated: the gather's latency, with nothing to hide it, made up a
  // third of a generation on L2-resident grids.
  Arrival next{kNoArrival, 0u, 0ull};
  if constexpr (MIG) {
    if (warp < nfull) {
      if constexpr (PLAN) move = move_of(first);
      next = arrival_of<TRACKED>(p, move, first, tin, sin);
      if (planned && warp + nwarps < nfull) move = move_of(first + skip);
    }
  }
  [[maybe_unused]] Planner planner(p, mv, warp, nwarps);
  uint32_t st = 0, phase = 0;  // ring position of the k-th group and its phase parity
  uint32_t isl0 = first;
  for (uint32_t grp = warp; grp < nfull; grp += nwarps, isl0 += skip) {
    const Arrival in = next;
    if constexpr (MIG) {
      if (grp + nwarps < nfull) {
        if (!planned) move = move_of(isl0 + skip);
        next = arrival_of<TRACKED>(p, move, isl0 + skip, tin, sin);
        if (planned && grp + 2u * nwarps < nfull) move = move_of(isl0 + 2u * skip);
      }
    }
    if (grp != warp) {
#pragma unroll
      for (uint32_t i = 0; i < GR; ++i) w[i] = lane_tail(p, head, isl0 + i);
    }
    if (!__all_sync(kFull, mbar_wait(&bar[st], phase))) {
      // give up: record the timeout, wait (bounded) for this warp's copies
      // still in flight (the groups issued into the ring from this one on),
      // leave (once the moves that later launches read are written)
      if (lane == 0) {
        atomicCAS(err, 0, kDevErrWaitTimeout);
        uint32_t s2 = st, ph2 = phase;
        for (uint32_t j = 0; j < stages && grp + j * nwarps < nfull; ++j) {
          mbar_wait(&bar[s2], ph2);
          if (++s2 == stages) {
            s2 = 0;
            ph2 ^= 1u;
          }
        }
      }
      __syncwarp();
      break;
    }
    uint32_t *tr = (uint32_t *)(ring + st * kStageBytes<GR>);
    uint64_t *sr = (uint64_t *)(ring + st * kStageBytes<GR> + kTraitBytes<GR>);
    if constexpr (MIG) {
      if (in.at != kNoArrival) {
        tr[in.at] = in.it;
        if constexpr (TRACKED) sr[in.at] = in.is;
      }
      __syncwarp();
    }
    uint32_t *to = tout + (size_t)isl0 * 32u + lane;
    uint64_t *so = TRACKED ? sout + (size_t)isl0 * 32u + lane : sout;
    replicate_group<TRACKED, T2, TWO, DEL, GR>(
        p, dep, w, tr, sr, to, so, [&](uint32_t i, uint32_t q) {
          return q == 0 ? lane_tail(p, head2, isl0 + i)
                        : philox_rk(p, lane, isl0 + i, G, kPurposeReplicate + 1 + q);
        });
    __syncwarp();  // every lane is done with this stage before it is refilled
    if (lane == 0 && grp + stages * nwarps < nfull) issue(isl0 + stages * skip, st);
    if constexpr (PLAN) planner.visit<32>(p, p, mv, G, GR);
    if (++st == stages) {
      st = 0;
      phase ^= 1u;
    }
  }
  if constexpr (PLAN) planner.rest<32>(p, p, mv, G);
  // the last islands, too few for a group, on the register path, one to a warp
  // (333x337 islands 16.2 us; all of them on one warp 18.5)
  const uint32_t rest = nfull * GR + (nwarps - 1u - warp);
  if (rest < p.islands) single_island<TRACKED, T2, MIG>(p, dep, G, rest, tin, sin, tout, sout);
}

template <bool TRACKED, bool T2, bool TWO, bool DEL, bool MIG, uint32_t GR>
int staged_blocks() {
  static int blocks = 0;
  if (blocks == 0) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t smem = staged_smem_bytes<GR>();
    cudaFuncSetAttribute(step_staged_kernel<TRACKED, T2, TWO, DEL, MIG, GR>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, step_staged_kernel<TRACKED, T2, TWO, DEL, MIG, GR>, kStagedThreads, smem);
    if (per_sm > kStagedBlocks<GR>) per_sm = kStagedBlocks<GR>;
    blocks = sms * (per_sm > 0 ? per_sm : 1);
  }
  return blocks;
}

template <bool TRACKED, bool T2, bool TWO, bool DEL, bool MIG, uint32_t GR>
void launch_staged_t(const RunParams &p, const Deposit &dep, const StagedLaunch &l,
                     const uint32_t *tin, const uint64_t *sin, uint32_t *tout, uint64_t *sout,
                     int *err, cudaStream_t stream) {
  const uint32_t groups = (p.islands + GR - 1) / GR;
  const uint32_t need = (groups + kStagedWarps - 1) / kStagedWarps;
  int b = staged_blocks<TRACKED, T2, TWO, DEL, MIG, GR>();
  if ((uint32_t)b > need) b = (int)need;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)b);
  cfg.blockDim = dim3(kStagedThreads);
  cfg.dynamicSmemBytes = staged_smem_bytes<GR>();
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, step_staged_kernel<TRACKED, T2, TWO, DEL, MIG, GR>, p, dep, l, tin, sin,
                     tout, sout, err);
}

template <bool TRACKED, bool T2, uint32_t GR>
void launch_staged_m(const RunParams &p, const Deposit &dep, const StagedLaunch &l, bool mig,
                     const uint32_t *tin, const uint64_t *sin, uint32_t *tout, uint64_t *sout,
                     int *err, cudaStream_t stream) {
#define HSGA_STAGED(TWO_, DEL_)                                                               \
  if (mig)                                                                                    \
    launch_staged_t<TRACKED, T2, TWO_, DEL_, true, GR>(p, dep, l, tin, sin, tout, sout, err,  \
                                                       stream);                               \
  else                                                                                        \
    launch_staged_t<TRACKED, T2, TWO_, DEL_, false, GR>(p, dep, l, tin, sin, tout, sout, err, \
                                                        stream);
  if (TRACKED && dep.two) {
    HSGA_STAGED(true, true)
  } else if (p.has_del) {
    HSGA_STAGED(false, true)
  } else {
    HSGA_STAGED(false, false)
  }
#undef HSGA_STAGED
}

template <uint32_t GR>
void launch_staged_g(const RunParams &p, const Deposit &dep, const StagedLaunch &l, bool mig,
                     const uint32_t *tin, const uint64_t *sin, uint32_t *tout, uint64_t *sout,
                     int *err, cudaStream_t stream) {
  const bool t2 = p.tournament == 2;
  if (p.policy != HSGA_NONE) {
    if (t2) launch_staged_m<true, true, GR>(p, dep, l, mig, tin, sin, tout, sout, err, stream);
    else launch_staged_m<true, false, GR>(p, dep, l, mig, tin, sin, tout, sout, err, stream);
  } else {
    if (t2) launch_staged_m<false, true, GR>(p, dep, l, mig, tin, sin, tout, sout, err, stream);
    else launch_staged_m<false, false, GR>(p, dep, l, mig, tin, sin, tout, sout, err, stream);
  }
}

}  // namespace

// Launches plan ahead where a warp takes at least two groups: with one, planning
// would lengthen every warp's only visit.
bool staged_stream_plan(const RunParams &p, StreamPlan *out) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  out->moves_ahead =
      p.islands / kStageGroup >= 2u * kStagedWarps * kStagedBlocksPerSM * (uint32_t)sms;
  out->back = planes_exceed_l2(p);
  // groups of four where they take one round of the warps: the generation is
  // then one group's latency (16x16 islands 2.5 us against 3.0 with groups of
  // eight, both with their draws after the wait)
  const uint32_t one_round =
      kSmallStageGroup * kStagedWarps * kSmallStagedBlocksPerSM * (uint32_t)sms;
  // two rounds of them, too, are faster than one full round of eights and a
  // partial one (with larger tournaments only where that one gives a scheduler
  // more than one more warp): 24,000 islands 5.50 us against 6.22, 28,000 5.71
  // and 6.39, tournament 5 9.32 and 8.21, 9.27 and 11.26; 20,500 5.35 and 5.62,
  // 9.22 and 8.02; three rounds, 31,000, 6.12 and 6.46, but 33,000 6.66 and 6.48
  const uint32_t eights = kStageGroup * kStagedWarps * kStagedBlocksPerSM * (uint32_t)sms;
  const uint32_t least = p.tournament == 2u ? eights : eights + eights / 4u;
  const bool small = p.islands <= one_round || (p.islands > least && p.islands <= 2u * one_round);
  out->group = (int)(small ? kSmallStageGroup : kStageGroup);
  return true;
}

cudaError_t launch_step_staged(const RunParams &p, const StreamPlan &plan, uint32_t G,
                               bool do_mig, const Moves &mv, const uint32_t *tin,
                               const uint64_t *sin, uint32_t *tout, uint64_t *sout, int *err,
                               cudaStream_t stream) {
  if (p.n != 32) return cudaErrorInvalidValue;
  const Deposit dep = deposit_for(p, G);
  const bool tracked = p.policy != HSGA_NONE, t2 = p.tournament == 2;
  // a second group staged ahead pays where memory is the limit: 16.8M agents
  // 66.0 against 67.3 us, but untracked 54.5 against 52.7, tournament 5 on
  // 500x500 islands 61.6 against 60.8, 256x256 islands 11.5 against 11.2
  const StagedLaunch l{G, plan.back && (G & 1u) ? 1u : 0u, tracked && t2 && plan.back ? 2u : 1u,
                       mv};
  if (plan.group == (int)kSmallStageGroup)
    launch_staged_g<kSmallStageGroup>(p, dep, l, do_mig, tin, sin, tout, sout, err, stream);
  else
    launch_staged_g<kStageGroup>(p, dep, l, do_mig, tin, sin, tout, sout, err, stream);
  return cudaGetLastError();
}

}  // namespace hsga
