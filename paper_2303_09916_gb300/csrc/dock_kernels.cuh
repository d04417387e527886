// Chain and scoring kernels, instantiated once per map format by the
// dock_fmt*.cu translation units (compiled in parallel).
#pragma once
#include "chain_device.cuh"
#include "launch.h"

namespace dsdp {

// Register budgets of the chain kernel: variant 0 caps at 128 registers (16
// warps per SM, no spills), variant 1 at 96 (20 warps), 2 at 80 (24 warps) and
// 3 at 72 (28 warps), each with a few more bytes spilled; the autotuner picks
// per plan by measurement.  Variants 2 and 3 are compiled for the
// one-atom-per-lane tiles only (two atoms per lane and mixed tiles take
// variants 0 and 1; a plan asking for more falls back to the 96-register
// kernel).  The bounds are stated for CTAs of up to 4 warps (chains); CTAs of
// 1 or 2 warps get the same register cap.
constexpr int kMaxChainWarps = 4;
template <int VAR>
struct ChainOcc;
template <>
struct ChainOcc<0> {
  static constexpr int kMinBlocks = 4;  // 65536 / (128 * 4) = 128 registers
};
template <>
struct ChainOcc<1> {
  static constexpr int kMinBlocks = 5;  // 102 -> 96 registers
};
template <>
struct ChainOcc<2> {
  static constexpr int kMinBlocks = 6;  // 85 -> 80 registers
};
template <>
struct ChainOcc<3> {
  static constexpr int kMinBlocks = 7;  // 73 -> 72 registers
};
// Chains: a CTA runs one tile of up to W chains of one job; W = blockDim / 32.
// The job's ligand blob is staged into shared memory once per tile; ligands of
// up to 32 atoms run one atom per lane, larger ones two, whatever else the
// launch holds (a chain's arithmetic depends on its own job only).  APLS: the
// tiles compiled in (1 or 2; 3 = both, for launches that mix them -- each
// single-tile kernel keeps its register allocation to itself).
// n_items = 0: CTA b runs tile b.  Else the CTAs pull items from a work queue
// until none are left: item i is tile i (n_blocks = 0), or, time-sliced, one
// slice of a tile (the blocks say which).
//
// Why slices: a chain's length (evaluations until its last local optimisation
// ends) varies by a factor of two around the mean and is not known before.  Run
// to the end one after the other, the long chains that start last leave most SMs
// idle: 6,144 typical-4k chains kept an SM busy for 72 % of the launch (37.1 ms;
// 29.4 sliced).  In slices every chain starts early, and a slow one never waits:
// an item of a tile that is still running is left to the CTA that runs it
// (tickets), which goes on with the tile's next slice.  The slices come in the
// order of the work that their chains have left, most first (plan_tiles).
//
// The queue runs dry while the slowest chains still have slices to go: in the end a
// few of them decide how long the launch takes.  Once no more than team_when CTAs
// are left, they leave their chains in the records, and dock_team_kernel finishes
// those, several warps to a chain.
struct ChainQueue {
  int* counter;              // the next item
  int* exited;               // CTAs that found nothing left to do
  int* tickets;              // [n_tiles] items taken and not finished
  int* next_step;            // [n_tiles][W] the step each chain stands at
  const SliceBlock* blocks;  // by item_begin
  int n_blocks, n_items;
  int team_when;             // 0: every chain is finished here
};

// The next tile for this CTA, n_tiles when none is left (one thread).  The first
// taker of an idle tile runs it; an item of a running tile stays with its CTA.
__device__ __forceinline__ int queue_next(const ChainQueue& q, int n_tiles) {
  for (;;) {
    const int item = atomicAdd(q.counter, 1);
    if (item >= q.n_items) return n_tiles;
    int t = item;
    if (q.n_blocks) {
      int lo = 0, hi = q.n_blocks;  // blocks[lo].item_begin <= item < blocks[hi].item_begin
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(&q.blocks[mid].item_begin) <= item) lo = mid;
        else hi = mid;
      }
      t = __ldg(&q.blocks[lo].tile_begin) + item - __ldg(&q.blocks[lo].item_begin);
    }
    if (atomicAdd(q.tickets + t, 1) == 0) {
      __threadfence();  // the records of the tile's last slice, written before its ticket was given back
      return t;
    }
  }
}

template <int FMT, int APLS, int IU, bool REVIEW, bool FLAT>
__device__ __forceinline__ void chain_cta(const DevJob* __restrict__ jobs, const Tile* __restrict__ tiles, int n_tiles,
                                          const ChainQueue& queue, int blob_smem, const ScratchLayout& lay) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ int s_tile;
  __shared__ int s_job;
  const int warp = threadIdx.x >> 5;
  // the plan's next group of chains depends on nothing here: its CTAs may take
  // the places this launch's CTAs leave (no effect without such a launch)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x == 0) {
    s_job = -1;
    s_tile = queue.n_items ? queue_next(queue, n_tiles) : (int)blockIdx.x;
    if (queue.n_items && s_tile >= n_tiles) atomicAdd(queue.exited, 1);
  }
  __syncthreads();
  for (;;) {
    const int t = s_tile;
    if (t >= n_tiles) break;
    const Tile tile = tiles[t];
    const DevJob& J = jobs[tile.job];
    if (s_job != tile.job) {  // uniform: s_job only changes between barriers
      __syncthreads();
      stage_blob(smem, J.blob, reinterpret_cast<const BlobHeader*>(J.blob)->stage_bytes);
      if (threadIdx.x == 0) s_job = tile.job;
    }
    if (warp < tile.count) {
      const WarpScratch W = warp_scratch_at(smem + blob_smem + warp * lay.bytes, lay);
      const LigView L = view_blob(smem);
      const int chain = tile.chain0 + warp;
      ChainSlice sl{nullptr, nullptr, 0};
      if (queue.n_blocks) {
        sl.rec = chain_record(J, chain);
        sl.next_step = queue.next_step + (size_t)t * (blockDim.x >> 5) + warp;
        sl.steps = J.slice_steps;
      }
      if (APLS == 1 || (APLS == 3 && L.n_atoms <= 32)) run_chain<1, FMT, IU, REVIEW, FLAT>(J, L, W, chain, sl);
      else run_chain<2, FMT, IU, REVIEW, FLAT>(J, L, W, chain, sl);
    }
    if (!queue.n_items) break;
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();  // this slice's records, before the ticket is given back
      if (atomicSub(queue.tickets + s_tile, 1) == 1) {
        s_tile = queue_next(queue, n_tiles);
      } else if (queue.team_when && jobs[s_job].optimizer == DSDP_OPT_BFGS &&
                 *(volatile int*)queue.counter >= queue.n_items &&
                 (int)gridDim.x - *(volatile int*)queue.exited <= queue.team_when) {
        s_tile = n_tiles;
      }
      if (s_tile >= n_tiles) atomicAdd(queue.exited, 1);
    }
    __syncthreads();
  }
  // what follows on the stream follows this launch: it ends after the group before it
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int FMT, int VAR, int APLS>
__global__ void __launch_bounds__(32 * kMaxChainWarps, ChainOcc<VAR>::kMinBlocks)
    dock_chains_kernel(const DevJob* __restrict__ jobs, const Tile* __restrict__ tiles, int n_tiles, ChainQueue queue,
                       int blob_smem, ScratchLayout lay) {
  constexpr bool kReview = VAR == 1 && (APLS == 3 || (APLS == 1 && fmt_channels(FMT) == 1));
  chain_cta<FMT, APLS, APLS == 3 ? 1 : 2, kReview, VAR == 0 && APLS == 1>(jobs, tiles, n_tiles, queue, blob_smem, lay);
}

// Teams (run_team): CTA b runs tile b, a single chain, with all its warps.  MB: CTAs
// of kMaxTeam warps the registers must allow per SM; with one chain per SM at most,
// one (64 plain-2k chains take 5 % less time than with two), else two, which is 128
// registers and four teams of 4 per SM (384 typical-4k chains 6.1 ms against 7.5 with
// one).  next_step: the
// chains that a time-sliced launch left unfinished (ChainQueue), from their records;
// null: whole chains.  APLS as in dock_chains_kernel; two atoms per lane alone run the
// kernel of both (384 chains of 45 atoms, 20 steps: 6.11 ms; by itself that kernel
// spills 44 bytes at 128 registers, 6.32), one atom per lane its own (Eq. 3 maps 6.93
// ms, with both 7.07; Eq. 4 3.24).
template <int FMT, int MB, int APLS>
__global__ void __launch_bounds__(32 * kMaxTeam, MB)
    dock_team_kernel(const DevJob* __restrict__ jobs, const Tile* __restrict__ tiles, const int* next_step,
                     int blob_smem, ScratchLayout lay) {
  extern __shared__ __align__(16) uint8_t smem[];
  // as in dock_chains_kernel: a next group may start where this one leaves room
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const Tile tile = tiles[blockIdx.x];
  const DevJob& J = jobs[tile.job];
  const int first = next_step ? __ldcg(next_step + blockIdx.x) : 0;
  if (first > J.n_steps) return;
  stage_blob(smem, J.blob, reinterpret_cast<const BlobHeader*>(J.blob)->stage_bytes);
  const LigView L = view_blob(smem);
  uint8_t* const scratch = smem + blob_smem;
  const WarpScratch W = warp_scratch_at(scratch + (threadIdx.x >> 5) * lay.bytes, lay);
  TeamSlot* const ex = reinterpret_cast<TeamSlot*>(scratch + (blockDim.x >> 5) * lay.bytes);
  if (APLS == 1 || (APLS == 3 && L.n_atoms <= 32)) run_team<1, FMT>(J, L, W, ex, tile.chain0, first);
  else run_team<2, FMT>(J, L, W, ex, tile.chain0, first);
}

// Score + gradient of a batch of conformations: one warp per conformation,
// warps striding over the batch (the ligand is staged once per CTA, while the first
// conformation is on its way).  FLAT (score_placed): a batch of at most one warp
// per scheduler, which takes as long as one evaluation does.  Registers: no spills.
// FLAT has a CTA per SM and takes up to 128 (600 conformations of 30 / 45 / 64 atoms on
// FP32 maps 4.6 / 6.8 / 9.4 us, at 80 registers 4.9 / 8.2 / 11.9); of many conformations
// one atom per lane takes 96, 20 warps per SM (100,003 of 30 atoms 182 us, Eq. 3 maps
// 166; at 80, 24 warps, 184 and 197) and unrolls the passes with hydrophobic and H-bond
// pairs too (180 and 164), two take the 80 that they need.
template <int APL, int FMT, bool FLAT>
__global__ void __launch_bounds__(128, FLAT ? 4 : APL == 1 ? 5 : 6)
    score_eval_kernel(MapView M, const uint8_t* __restrict__ blob, const float* __restrict__ conf, int n_conf, int T,
                      float* __restrict__ energy, float* __restrict__ grad, uint32_t flags, int blob_smem,
                      ScratchLayout lay) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int warps = gridDim.x * (blockDim.x >> 5);
  int c = blockIdx.x * (blockDim.x >> 5) + warp;
  Conf x = load_conf(conf + (size_t)(c < n_conf ? c : 0) * (7 + T), T);
  stage_blob(smem, blob, blob_smem);
  const LigView L = view_blob(smem);
  const WarpScratch W = warp_scratch_at(smem + blob_smem + warp * lay.bytes, lay);
  LaneLig<APL> R;
  load_lane_lig<APL>(L, R);
  const int n_ramp = ramp_steps(L);
  while (c < n_conf) {  // warp-uniform loop
    x.q = qnormalize(x.q);
    float g;
    Placed<APL> P;
    place_atoms<APL>(L, x, P);
    const float e = score_placed<APL, FMT, 2, FLAT, FLAT || APL == 1 ? 2 : 1>(M, L, R, n_ramp, W, x, P, g, flags);
    if (lane == 0 && energy) energy[c] = e;
    if (grad && lane < 6 + T) grad[(size_t)c * (6 + T) + lane] = g;
    c += warps;
    if (c < n_conf) x = load_conf(conf + (size_t)c * (7 + T), T);
  }
}

template <int FMT, int VAR, int APLS>
cudaError_t launch_chains_var(const ChainLaunch& a, cudaStream_t st) {
  const dim3 block(32 * a.warps_per_cta);
  const size_t smem = (size_t)a.blob_smem + (size_t)a.warps_per_cta * a.scratch.bytes;
  auto k = dock_chains_kernel<FMT, VAR, APLS>;
  cudaError_t e = allow_smem((const void*)k, smem);
  if (e != cudaSuccess) return e;
  const int cached = kChainSmemPerSm / (int)(smem + 1024);  // CTAs per SM (1 KB each is the system's)
  const bool carve = APLS == 1 && cached * a.warps_per_cta >= kChainSmemWarps;
  int grid = a.n_tiles;
  ChainQueue q{a.counter, a.exited, a.tickets, a.next_step, a.blocks, 0, 0, a.team_when};
  if (a.queue != kNoQueue) {
    int per_sm = 0;
    const int sms = device_sms();
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 32 * a.warps_per_cta, smem);
    if (e != cudaSuccess) return e;
    const int slots = per_sm * sms > 1 ? per_sm * sms : 1;
    if (a.n_tiles > slots || a.team_when) {
      grid = a.n_tiles < slots ? a.n_tiles : slots;
      q.n_blocks = a.n_blocks;
      q.n_items = a.n_items;
    } else if (a.queue == kQueue) {
      q.n_items = a.n_tiles;  // every tile has a slot of its own: nothing to slice
    }
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2]{};
  cfg.attrs = attr;
  if (a.overlap) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (carve) {
    attr[cfg.numAttrs].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[cfg.numAttrs++].val.sharedMemCarveout = a.more_smem ? kChainSmemPercentMore : kChainSmemPercent;
  }
  return cudaLaunchKernelEx(&cfg, k, reinterpret_cast<const DevJob*>(a.jobs), reinterpret_cast<const Tile*>(a.tiles),
                            a.n_tiles, q, a.blob_smem, a.scratch);
}

template <int FMT, int APLS>
cudaError_t launch_team(const ChainLaunch& a, cudaStream_t st) {
  const size_t smem = (size_t)a.blob_smem + (size_t)a.team * (a.scratch.bytes + 2 * sizeof(TeamSlot));
  auto k = a.team == kMaxTeam ? dock_team_kernel<FMT, 1, APLS> : dock_team_kernel<FMT, 2, APLS>;
  const cudaError_t e = allow_smem((const void*)k, smem);
  if (e != cudaSuccess) return e;
  k<<<a.n_tiles, 32 * a.team, smem, st>>>(reinterpret_cast<const DevJob*>(a.jobs),
                                          reinterpret_cast<const Tile*>(a.tiles),
                                          a.team_resumes ? a.next_step : nullptr, a.blob_smem, a.scratch);
  return cudaGetLastError();
}

template <int FMT>
cudaError_t launch_chains_impl(const ChainLaunch& a, cudaStream_t st) {
  if (a.team > 1) return a.apl_mask == 1 ? launch_team<FMT, 1>(a, st) : launch_team<FMT, 3>(a, st);
  if (a.warps_per_cta != 1 && a.warps_per_cta != 2 && a.warps_per_cta != kMaxChainWarps) return cudaErrorInvalidValue;
  if (a.apl_mask == 1) {
    switch (a.variant) {
      case 0: return launch_chains_var<FMT, 0, 1>(a, st);
      case 1: return launch_chains_var<FMT, 1, 1>(a, st);
      case 2: return launch_chains_var<FMT, 2, 1>(a, st);
      default: return launch_chains_var<FMT, 3, 1>(a, st);
    }
  }
  if (a.apl_mask == 2) return a.variant ? launch_chains_var<FMT, 1, 2>(a, st) : launch_chains_var<FMT, 0, 2>(a, st);
  // mixed tiles: the 128- and 96-register budgets
  return a.variant ? launch_chains_var<FMT, 1, 3>(a, st) : launch_chains_var<FMT, 0, 3>(a, st);
}

template <int FMT>
cudaError_t launch_score_impl(const ScoreLaunch& a, cudaStream_t st) {
  const int wpc = 4;
  const int sms = device_sms();
  const int want = (a.n_conf + wpc - 1) / wpc, cap = sms * 8;  // warps stride over the conformations
  const dim3 block(32 * wpc), grid(want < cap ? want : cap);
  const size_t smem = (size_t)a.blob_smem + (size_t)wpc * a.scratch.bytes;
  const bool flat = a.n_conf <= 4 * sms;
  auto k = a.apl == 1 ? (flat ? score_eval_kernel<1, FMT, true> : score_eval_kernel<1, FMT, false>)
                      : (flat ? score_eval_kernel<2, FMT, true> : score_eval_kernel<2, FMT, false>);
  const cudaError_t e = allow_smem((const void*)k, smem);
  if (e != cudaSuccess) return e;
  k<<<grid, block, smem, st>>>(a.map, a.blob, a.conf, a.n_conf, a.n_torsions, a.energy, a.grad, a.flags, a.blob_smem,
                               a.scratch);
  return cudaGetLastError();
}

}  // namespace dsdp

#define DSDP_INSTANTIATE_FMT(F)                                                                   \
  namespace dsdp {                                                                                \
  cudaError_t launch_chains_fmt##F(const ChainLaunch& a, cudaStream_t st) {                       \
    return launch_chains_impl<F>(a, st);                                                          \
  }                                                                                               \
  cudaError_t launch_score_fmt##F(const ScoreLaunch& a, cudaStream_t st) {                        \
    return launch_score_impl<F>(a, st);                                                           \
  }                                                                                               \
  }
