// Host-side launch descriptions of the kernels (included by the .cu files only).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "chain_device.cuh"

namespace dsdp {

// Whether a chain launch takes its tiles from the work queue (ChainQueue): never,
// always, or when there are more tiles than CTAs fit on the GPU at once.
enum ChainQueueMode { kNoQueue, kQueue, kQueueIfMany };

constexpr int kMaxTeam = 8;  // warps of a chain (dock_team_kernel)

struct ChainLaunch {
  const void* jobs;   // DevJob[] (device)
  const void* tiles;  // Tile[] (device)
  int n_tiles;
  ChainQueueMode queue;
  int* counter;       // the queue's device arrays (ChainQueue), zeroed before the launch
  int* exited;
  int* tickets;
  int* next_step;
  const SliceBlock* blocks;  // device; the items of a time-sliced launch
  int n_blocks, n_items;
  bool overlap;       // independent of the launch before it on the stream: its CTAs may start as that one's leave
  int warps_per_cta;
  int team;           // warps of a chain (dock_team_kernel); 1: none of it
  bool team_resumes;  // the team finishes what a time-sliced launch left
  int team_when;      // CTAs left when a time-sliced launch leaves the rest to a team; 0: never
  int apl;            // largest atoms-per-lane tile present
  int apl_mask;       // tiles present: bit 0 one atom per lane (<= 32 atoms), bit 1 two (<= 64)
  bool more_smem;     // kChainSmemPercentMore
  int blob_smem;      // bytes reserved for the largest staged blob prefix
  ScratchLayout scratch;  // per-warp scratch, sized for the group's largest ligand
  int variant;        // register budget of the chain kernel (0: 128, 1: 96)
};

struct ScoreLaunch {
  MapView map;
  const uint8_t* blob;  // device
  const float* conf;
  int n_conf;
  float* energy;
  float* grad;
  uint32_t flags;
  int apl;
  int n_torsions;
  int blob_smem;
  ScratchLayout scratch;
};

#define DSDP_DECLARE_FMT(F)                                               \
  cudaError_t launch_chains_fmt##F(const ChainLaunch& a, cudaStream_t st); \
  cudaError_t launch_score_fmt##F(const ScoreLaunch& a, cudaStream_t st);
DSDP_DECLARE_FMT(0)
DSDP_DECLARE_FMT(1)
DSDP_DECLARE_FMT(2)
DSDP_DECLARE_FMT(3)
DSDP_DECLARE_FMT(4)
DSDP_DECLARE_FMT(5)
#undef DSDP_DECLARE_FMT

// SMs of the current device (asked for once per device).
int device_sms();
// Lets a kernel use `smem` bytes of dynamic shared memory; below 48 KB it may anyway,
// and the call would cost a fifth of a launch.
cudaError_t raise_smem(const void* kernel, size_t smem);
inline cudaError_t allow_smem(const void* kernel, size_t smem) {
  return smem <= 47 * 1024 ? cudaSuccess : raise_smem(kernel, smem);
}

constexpr int kSmemPerSm = 228 * 1024;
// What a chain launch of one-atom-per-lane tiles asks the SMs to set aside as shared
// memory, in percent: what is left of an SM's 256 KB caches the corners of the atoms'
// cells, which successive evaluations of a chain mostly share.  Unasked, the driver
// leaves an SM that never drains with the split of whichever kernel it ran before: four
// steps of 32 typical-4k systems in flight, grid builds and rescoring between them, ran
// 418 systems/s, at 59 % 597 (one at a time 539 and 574).  59 % is the rule; 73 %
// (more chains, less cache) for a launch that fills the GPU by itself and misses less:
//   of maps of up to 4 times the L2 cache (32 ligands on one FP32 receptor, 20 steps,
//     25.0 ms, at 59 % 25.6 and at 80 % 27.4; of 12 torsions 26.5, 28.3, 26.5; 6 receptors
//     20.2, 20.4; but 24 receptors 22.2 ms at 73 %, 21.1 at 59, 22.8 at 52, 34.2 at 80);
//   of Barzilai-Borwein chains alone (32 receptors, 10 steps, 24.1 ms, at 59 % 24.8).
// Not beside another group of its plan or chains under way on other streams, with which
// it shares the SMs (64 ligands of 10-60 atoms 63.7 ms, at 73 % 65.3), nor for a context's
// jobs, whose next batch starts before an SM drains and finds the last one's split
// (saturated serving 492 requests/s, 478), and not up to 16 chains per SM, which need
// no more (1,024 Barzilai-Borwein chains 6.16 ms, 6.21).  Measured for chains of up to 9.2 KB (16 in
// 164 KB); larger ones keep what the driver gives.  (The split that a percentage stands
// for is the driver's and not shown anywhere: 66 % ran like 59, 71 like 73, 87 like 100.)
constexpr int kChainSmemPerSm = 164 * 1024, kChainSmemWarps = 16;
constexpr int kChainSmemPercent = 59, kChainSmemPercentMore = 73, kNearL2s = 4;

MapView map_view_of(const dsdp_grid_view* g);
cudaError_t launch_rescore(const void* jobs, const void* tiles, int n_tiles, cudaStream_t st);
int rescore_tile_chains();
cudaError_t launch_topk(const void* jobs, int n_jobs, int max_chains, cudaStream_t st);

}  // namespace dsdp
