// Device-resident entry points of the C ABI: scoring a batch of
// conformations, and docking plans (chain kernels, FP64 rescoring, top-k)
// that can be enqueued repeatedly or captured into CUDA graphs.
#include <string.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "launch.h"

constexpr int kMaxGroups = 12;  // map formats x atoms per lane

struct dsdp_plan {
  dsdp_ctx* ctx = nullptr;
  int n_jobs = 0;
  uint32_t flags = 0;
  int warps_per_cta = 1;
  int variant = 0;        // chain kernel register budget (0: 128, 1: 96)
  uint64_t tune_key = 0;  // shape key for the autotuner's choice
  int max_chains = 0;
  // one device arena holding job table, tiles, counters and scratch
  void* arena = nullptr;
  size_t arena_bytes = 0;
  struct Group {
    int fmt, apl, first_tile, n_tiles, blob_smem, max_atoms, max_torsions, apl_mask;
    int first_block, n_blocks, n_items;  // time-sliced queue (SliceBlock)
    int first_chain, n_chains;           // tiles of one chain each (teams)
    bool misses_less;                    // of near maps or Barzilai-Borwein alone (kChainSmemPercent)
  };
  std::vector<Group> groups;
  void* d_jobs = nullptr;
  void* d_tiles = nullptr;
  void* d_singles = nullptr;  // room for the same chains in tiles of one; null if teams are never taken
  void* d_rtiles = nullptr;
  // work queue: [kMaxGroups counters, one per group][kMaxGroups exit counts][tickets per tile]
  // [next step per tile and warp]; zeroed by each launch
  int* d_queue = nullptr;
  size_t queue_bytes = 0;
  size_t queue_next_off = 0;  // of the next steps, in ints
  // What runs the chains without a fixed choice: the register budget, chains per CTA,
  // warps of each chain (dock_team_kernel), and whether a group with more tiles than fit
  // at once takes the queue.
  struct Arrangement {
    int variant, warps, team;
    bool queue;
  };
  Arrangement automatic{0, 1, 1, false};  // by the plan's size, whatever it runs now
  bool auto_queue = false;    // as it runs now (variant, warps_per_cta): the queue, teams
  int team = 1;
  int last_team = 0;          // of the last launch (chains in flight elsewhere may take its teams)
  bool any_bfgs = false;
  bool resident = false;      // 16 chains per SM or fewer
  int apl_max = 1;            // atoms per lane of the largest ligand
  void* d_blocks = nullptr;
  int n_rtiles = 0;
  // per job, to lay groups and tiles out again for another configuration
  struct Shape {
    int fmt, apl, blob, atoms, torsions, chains;
    double cost;  // length of a chain, relative
    int slices;   // of each of its chains
    const void* maps;
    size_t map_bytes;
    bool bfgs;
  };
  std::vector<Shape> shape;
  std::vector<int> job_order;  // jobs by chain length, longest first
  int sms = 148;
  size_t l2_bytes = 0;
  // The plan's last chain launch, among those of the process's other plans (ChainsInFlight).
  struct Flight {
    cudaEvent_t done = nullptr;  // null: not tracked
    int device = 0, chains = 0;
    cudaStream_t stream = nullptr;
    bool busy = false;  // launched and not seen to have ended
  } flight;
};

namespace dsdp {

dsdp_status normalize_params(const dsdp_dock_params* in, dsdp_dock_params* out) {
  if (!in) return set_error(DSDP_ERR_INVALID_ARG, "dock params NULL");
  *out = *in;
  if (out->n_chains == 0) out->n_chains = 384;
  if (out->n_mc_steps == 0) out->n_mc_steps = 40;
  if (out->n_opt_iters == 0) out->n_opt_iters = 100;
  if (out->temperature == 0.0) out->temperature = 1.2;
  if (out->top_k == 0) out->top_k = 9;
  if (out->rmsd_dedup == 0.0) out->rmsd_dedup = 1.0;
  if (out->site_radius == 0.f) out->site_radius = 7.0f;
  if (out->n_chains < 1 || out->n_chains > DSDP_MAX_CHAINS)
    return set_error(DSDP_ERR_INVALID_ARG, "n_chains %d outside 1..%d", out->n_chains, DSDP_MAX_CHAINS);
  if (out->n_mc_steps < 0 || out->n_mc_steps > 100000) return set_error(DSDP_ERR_INVALID_ARG, "n_mc_steps out of range");
  if (out->trace < 0 || out->trace > 2) return set_error(DSDP_ERR_INVALID_ARG, "trace must be 0, 1 or 2");
  if (out->n_opt_iters < 0 || out->n_opt_iters > 100000)
    return set_error(DSDP_ERR_INVALID_ARG, "n_opt_iters out of range");
  if (out->optimizer != DSDP_OPT_BFGS && out->optimizer != DSDP_OPT_BB)
    return set_error(DSDP_ERR_INVALID_ARG, "unknown optimizer %d", out->optimizer);
  if (!(out->temperature > 0.0)) return set_error(DSDP_ERR_INVALID_ARG, "temperature must be positive");
  if (out->top_k < 1 || out->top_k > DSDP_MAX_TOP_K)
    return set_error(DSDP_ERR_INVALID_ARG, "top_k %d outside 1..%d", out->top_k, DSDP_MAX_TOP_K);
  if (!(out->rmsd_dedup >= 0.0)) return set_error(DSDP_ERR_INVALID_ARG, "rmsd_dedup must be >= 0");
  if (out->n_site_points < 0 || out->n_site_points > DSDP_MAX_SITE_POINTS)
    return set_error(DSDP_ERR_INVALID_ARG, "n_site_points %d outside 0..%d", out->n_site_points,
                     DSDP_MAX_SITE_POINTS);
  if (!(out->site_radius > 0.f) || !isfinite(out->site_radius))
    return set_error(DSDP_ERR_INVALID_ARG, "site_radius must be positive");
  return DSDP_OK;
}

static cudaError_t launch_chains_dispatch(int fmt, const ChainLaunch& a, cudaStream_t st) {
  switch (fmt) {
    case 0: return launch_chains_fmt0(a, st);
    case 1: return launch_chains_fmt1(a, st);
    case 2: return launch_chains_fmt2(a, st);
    case 3: return launch_chains_fmt3(a, st);
    case 4: return launch_chains_fmt4(a, st);
    default: return launch_chains_fmt5(a, st);
  }
}

static cudaError_t launch_score_dispatch(int fmt, const ScoreLaunch& a, cudaStream_t st) {
  switch (fmt) {
    case 0: return launch_score_fmt0(a, st);
    case 1: return launch_score_fmt1(a, st);
    case 2: return launch_score_fmt2(a, st);
    case 3: return launch_score_fmt3(a, st);
    case 4: return launch_score_fmt4(a, st);
    default: return launch_score_fmt5(a, st);
  }
}

static dsdp_status check_view(const dsdp_grid_view* g) {
  if (!g || !g->d_maps) return set_error(DSDP_ERR_INVALID_ARG, "grid view or maps NULL");
  if (g->dtype < 0 || g->dtype > 2 || g->mode < 0 || g->mode > 1)
    return set_error(DSDP_ERR_INVALID_ARG, "grid view dtype/mode invalid");
  for (int a = 0; a < 3; ++a)
    if (g->n[a] < 2) return set_error(DSDP_ERR_INVALID_ARG, "grid needs >= 2 vertices per axis");
  if (!(g->spacing > 0.0)) return set_error(DSDP_ERR_INVALID_ARG, "grid spacing must be positive");
  if ((double)DSDP_NUM_MAP_TYPES * g->n[0] * g->n[1] * g->n[2] >= 2147483648.0)
    return set_error(DSDP_ERR_INVALID_ARG, "grid exceeds 2^31 nodes (32-bit map indices)");
  return DSDP_OK;
}

static int device_attribute(cudaDeviceAttr attr, std::atomic<int>* known) {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && (v = known[dev].load(std::memory_order_relaxed)) > 0) return v;
  cudaDeviceGetAttribute(&v, attr, dev);
  if (dev >= 0 && dev < 64) known[dev].store(v, std::memory_order_relaxed);
  return v;
}

int device_sms() {
  static std::atomic<int> known[64];
  return device_attribute(cudaDevAttrMultiProcessorCount, known);
}

static size_t device_l2_bytes() {
  static std::atomic<int> known[64];
  return (size_t)device_attribute(cudaDevAttrL2CacheSize, known);
}

// A kernel has one limit per device, which every thread's launches share: it only ever
// grows, so that a launch cannot lower it between another thread's call and launch.
cudaError_t raise_smem(const void* kernel, size_t smem) {
  struct Limit {
    const void* kernel;
    int device;
    size_t bytes;
  };
  static std::mutex mu;
  static std::vector<Limit> limits;
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  Limit* l = nullptr;
  for (Limit& x : limits)
    if (x.kernel == kernel && x.device == dev) l = &x;
  const size_t most = l ? std::max(l->bytes, smem) : smem;
  const cudaError_t set = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (set != cudaSuccess) return set;
  if (l) l->bytes = most;
  else limits.push_back(Limit{kernel, dev, most});
  return cudaSuccess;
}

static size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// A job's coordinate scratch: FP64 coordinates while rescoring, the chains' records
// (ChainRecord) while a time-sliced launch runs them.
static size_t coord_bytes(int n_chains, int n_atoms, int n_torsions) {
  return (size_t)n_chains * std::max(sizeof(double) * 3 * n_atoms, (size_t)slice_record_bytes(n_torsions));
}

// Autotuner choices by plan shape (tune_key): (variant, persistent, warps).  Written
// by dsdp_plan_autotune, read by plans created with tile_config 0.
struct TuneEntry {
  uint64_t key;
  int variant, persistent, warps;
};
static std::mutex g_tune_mu;
static std::vector<TuneEntry> g_tune;

// Format mask, atoms per lane, log2 of the chain count, the optimisers, and what the
// choice stands in for: a fixed configuration that beats one automatic arrangement says
// nothing of another (one warp a chain is the fastest for 384 Barzilai-Borwein chains
// and takes twice a team's time for BFGS).
static uint64_t tune_key(uint32_t fmt_mask, int apl, size_t chains, bool all_bfgs, bool any_bfgs,
                         const dsdp_plan::Arrangement& automatic, int sms) {
  int lg = 0;
  while ((size_t(1) << lg) < chains) ++lg;
  return (uint64_t)lg | ((uint64_t)apl << 8) | ((uint64_t)fmt_mask << 16) | ((uint64_t)all_bfgs << 24) |
         ((uint64_t)any_bfgs << 25) | ((uint64_t)automatic.queue << 26) | ((uint64_t)automatic.variant << 27) |
         ((uint64_t)automatic.team << 28) | ((uint64_t)sms << 32);
}

static bool tune_lookup(uint64_t key, int* variant, int* persistent, int* warps) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  for (const TuneEntry& t : g_tune)
    if (t.key == key) {
      *variant = t.variant;
      *persistent = t.persistent;
      *warps = t.warps;
      return true;
    }
  return false;
}

static void tune_store(uint64_t key, int variant, int persistent, int warps) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  for (TuneEntry& t : g_tune)
    if (t.key == key) {
      t.variant = variant;
      t.persistent = persistent;
      t.warps = warps;
      return;
    }
  g_tune.push_back(TuneEntry{key, variant, persistent, warps});
}

static void tune_erase(uint64_t key) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  for (size_t i = 0; i < g_tune.size(); ++i)
    if (g_tune[i].key == key) {
      g_tune.erase(g_tune.begin() + i);
      return;
    }
}

// Slices of the launch's longest chains when it time-slices (ChainQueue): enough
// that the last slices are a small part of the launch, few enough that a slice
// (a few MC steps, hundreds of evaluations) hides its record's load and store.  Up to
// 16 chains per SM (most or all have a place at once) they seldom move and what counts
// is how soon the slowest reach the teams: 64 slices, of one MC step for jobs of up to
// 63 (1,536 chains as above: 11.6 ms, in 16 slices 12.8).  The limit goes by chains and
// not by the places that shared memory leaves: 2,280 chains of 10-60 atoms 27.8 ms,
// with their 10 places per SM as the limit 36.9; 2,400 of 60 atoms 38.6 and 39.7.
constexpr int kSliceRounds = 16, kSliceRoundsResident = 64;

static ChainQueueMode queue_mode(const dsdp_plan* P) {
  return (P->flags & DSDP_PLAN_PERSISTENT) ? kQueue : P->auto_queue ? kQueueIfMany : kNoQueue;
}

// Chain tiles of W chains of one job in groups of one launch each, and the items
// of a time-sliced launch.  A fixed configuration has one group per map format
// (the kernel that holds both tiles when it mixes them).  With the queue the
// ligands of up to and above 32 atoms are groups of their own: each runs its own
// kernel with its own shared memory (22 KB a chain at 60 atoms, 8 KB at 30), and
// the next group's CTAs start as the last one's leave (launch_chains_var).
// Jobs whose chains take longest come first (what starts last decides how long
// the launch's tail is), and of the slices those whose chains have the most work
// left, a job's slices side by side.
static void plan_tiles(dsdp_plan* P, int W, std::vector<Tile>& tiles, std::vector<SliceBlock>& blocks) {
  tiles.clear();
  blocks.clear();
  int n_chains = 0;
  P->groups.clear();
  const bool split = queue_mode(P) != kNoQueue;
  struct Item {
    double left;
    int tile, n;
  };
  std::vector<Item> items;
  std::vector<std::pair<const void*, size_t>> maps;
  for (int f = 0; f < 6; ++f)
    for (int apl = split ? 2 : 0; apl >= (split ? 1 : 0); --apl) {  // 0: both
      dsdp_plan::Group g{};
      g.fmt = f;
      g.first_tile = (int)tiles.size();
      items.clear();
      maps.clear();
      bool bfgs = false;
      for (int j : P->job_order) {
        const dsdp_plan::Shape& s = P->shape[j];
        if (s.fmt != f || (apl && s.apl != apl)) continue;
        g.apl = std::max(g.apl, s.apl);
        g.apl_mask |= s.apl;
        g.blob_smem = std::max(g.blob_smem, s.blob);
        g.max_atoms = std::max(g.max_atoms, s.atoms);
        g.max_torsions = std::max(g.max_torsions, s.torsions);
        maps.emplace_back(s.maps, s.map_bytes);
        bfgs = bfgs || s.bfgs;
        const int first = (int)tiles.size() - g.first_tile;
        for (int c = 0; c < s.chains; c += W) tiles.push_back(Tile{j, c, std::min(W, s.chains - c), 0});
        const int n = (int)tiles.size() - g.first_tile - first;
        for (int r = 0; r < s.slices; ++r) items.push_back(Item{s.cost * (s.slices - r) / s.slices, first, n});
      }
      g.n_tiles = (int)tiles.size() - g.first_tile;
      g.first_chain = n_chains;
      for (int t = g.first_tile; t < (int)tiles.size(); ++t) g.n_chains += tiles[t].count;
      n_chains += g.n_chains;
      std::sort(maps.begin(), maps.end());
      size_t map_bytes = 0;
      for (size_t k = 0; k < maps.size(); ++k)
        if (k + 1 == maps.size() || maps[k].first != maps[k + 1].first) map_bytes += maps[k].second;
      g.misses_less = map_bytes <= kNearL2s * P->l2_bytes || !bfgs;
      if (!g.n_tiles) continue;
      std::stable_sort(items.begin(), items.end(), [](const Item& a, const Item& b) { return a.left > b.left; });
      g.first_block = (int)blocks.size();
      for (const Item& it : items) {
        blocks.push_back(SliceBlock{g.n_items, it.tile});
        g.n_items += it.n;
      }
      g.n_blocks = (int)blocks.size() - g.first_block;
      P->groups.push_back(g);
    }
}

// Chains per SM that a time-sliced launch leaves to teams of 4 (chain stage of 1,536
// chains of 20-36 atoms: never 17.1 ms, from 4 per SM on 13.7, from 8 on 11.6; 2,000
// typical-4k chains 8.25, 8.0, 7.3).  Not when a group's chains outnumber their places
// and another group waits for these: the teams must wait for the whole group, and the
// other starts behind them (64 ligands of 10-60 atoms: never 60.5 ms, from 8 on 62).
constexpr int kTailTeams = 8;

// Warps of a chain (dock_team_kernel) when the plan's chains leave most of the GPU
// idle; 1 when they do not.  Up to one chain per SM a team of 8 (64 plain-2k chains
// take 6 % less time than in teams of 4, 200 typical-4k chains 7 % more), up to 8
// per SM teams of 4 (1,200 chains 6.9 ms, one warp each 8.1; 1,536 chains 9.7 against
// 8.3): beyond, the trial points that a line search does not come to cost more than
// the shorter way saves.  Teams are a warp per SM sub-partition or two: 5 and 6 warps
// measured slower than 4.
static int team_warps(size_t chains, int sms) {
  if (chains <= (size_t)sms) return kMaxTeam;
  return chains <= (size_t)(8 * sms) ? 4 : 1;
}

// Chain launches on their way.  Which way is the fastest for a plan of few chains
// depends on all the chains that run at the same time, so each plan marks the end of
// its last chain launch with an event, and a plan that could take teams counts what
// other streams have under way on its device.  The count only chooses between ways that
// give the same bits.  A launch under stream capture neither counts nor is counted: when
// and beside what it will run is not known.
static std::mutex g_flight_mu;
static std::vector<dsdp_plan::Flight*> g_flights;

static void track_flight(dsdp_plan::Flight* f, int chains) {
  f->chains = chains;
  if (cudaGetDevice(&f->device) != cudaSuccess ||
      cudaEventCreateWithFlags(&f->done, cudaEventDisableTiming) != cudaSuccess) {
    f->done = nullptr;
    cudaGetLastError();
    return;
  }
  std::lock_guard<std::mutex> lk(g_flight_mu);
  g_flights.push_back(f);
}

static void untrack_flight(dsdp_plan::Flight* f) {
  if (!f->done) return;
  {
    std::lock_guard<std::mutex> lk(g_flight_mu);
    g_flights.erase(std::remove(g_flights.begin(), g_flights.end(), f), g_flights.end());
  }
  cudaEventDestroy(f->done);
}

static void mark_flight(dsdp_plan::Flight* f, cudaStream_t st) {
  if (!f->done) return;
  std::lock_guard<std::mutex> lk(g_flight_mu);
  f->stream = st;
  f->busy = cudaEventRecord(f->done, st) == cudaSuccess;
  if (!f->busy) cudaGetLastError();
}

// Chains that other streams of the plan's device have under way: of each stream its
// largest launch (a stream's launches run one after the other), of the streams the
// seven largest (beside its own, a device runs eight unless the environment says more).
static size_t chains_in_flight(const dsdp_plan::Flight& own, cudaStream_t st) {
  constexpr int kStreams = 7;
  cudaStream_t stream[kStreams];
  int chains[kStreams], n = 0;
  // another thread's capture must not be ended by a query of this one
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  const bool swapped = cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess;
  {
    std::lock_guard<std::mutex> lk(g_flight_mu);
    for (dsdp_plan::Flight* f : g_flights) {
      if (!f->busy || f == &own || f->device != own.device || f->stream == st) continue;
      if (cudaEventQuery(f->done) != cudaErrorNotReady) {
        f->busy = false;
        continue;
      }
      int k = 0;
      while (k < n && stream[k] != f->stream) ++k;
      if (k == n && n < kStreams) chains[n++] = 0;
      if (k == kStreams) k = (int)(std::min_element(chains, chains + n) - chains);
      if (f->chains > chains[k]) chains[k] = f->chains, stream[k] = f->stream;
    }
  }
  if (cudaPeekAtLastError() == cudaErrorNotReady) cudaGetLastError();  // no error
  if (swapped) cudaThreadExchangeStreamCaptureMode(&mode);
  size_t sum = 0;
  for (int k = 0; k < n; ++k) sum += chains[k];
  return sum;
}

// Warps of a chain of a plan of `chains` that would take teams of `team` alone (1: it
// would not), with `others` under way beside them (round of launches of 10 steps,
// typical-4k, ms with one warp a chain / teams of 4 / of 8): streams x chains 2 x 128
// 3.7 / 1.94 / 1.80, 4 x 128 4.4 / 2.5 / 2.9, 8 x 128 4.7 / 3.2 / 5.3;
// 4 x 384 5.1 / 4.1 / 7.9, 5 x 5.0 / 4.8, 6 x 5.7 / 5.7, 7 x 5.6 / 6.8, 8 x 6.5 / 7.5.
// Two atoms per lane (45): 4 x 128 9.3 / 4.3 / 4.1, 8 x 128 10.1 / 5.4 / 7.7; 8 x 384 10.7
// in tiles of 4 chains / 12.4.  (One launch alone loses its teams' gain earlier,
// team_warps: its chains keep step.)
static int shared_team_warps(int team, size_t chains, size_t others, int apl_max, int sms) {
  if (team == 1) return 1;
  const size_t all = chains + others;
  if (chains <= (size_t)sms && all <= (size_t)((apl_max == 2 ? 4 : 2) * sms)) return kMaxTeam;
  return all <= (size_t)((apl_max == 2 ? 18 : 16) * sms) ? 4 : 1;
}

static cudaError_t plan_use_warps(dsdp_plan* P, int W) {
  std::vector<Tile> tiles;
  std::vector<SliceBlock> blocks;
  plan_tiles(P, W, tiles, blocks);
  P->warps_per_cta = W;
  cudaError_t e = cudaSuccess;
  if (!tiles.empty())
    e = cudaMemcpy(P->d_tiles, tiles.data(), sizeof(Tile) * tiles.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess && !blocks.empty())
    e = cudaMemcpy(P->d_blocks, blocks.data(), sizeof(SliceBlock) * blocks.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess && P->d_singles) {
    std::vector<Tile> singles;
    for (const Tile& t : tiles)
      for (int c = 0; c < t.count; ++c) singles.push_back(Tile{t.job, t.chain0 + c, 1, 0});
    e = cudaMemcpy(P->d_singles, singles.data(), sizeof(Tile) * singles.size(), cudaMemcpyHostToDevice);
  }
  return e;
}

}  // namespace dsdp

using namespace dsdp;

extern "C" dsdp_status dsdp_score_eval_device(const dsdp_grid_view* grid, const void* h_blob, const void* d_blob,
                                              const float* d_conf, int32_t n_conf, float* d_energy, float* d_grad,
                                              uint32_t flags, void* stream) {
  dsdp_status s = check_view(grid);
  if (s != DSDP_OK) return s;
  int32_t n_atoms = 0, T = 0, P = 0, B = 0;
  s = dsdp_ligand_blob_info(h_blob, &n_atoms, &T, &P, &B);
  if (s != DSDP_OK) return s;
  if (!d_blob || !d_conf || n_conf < 0) return set_error(DSDP_ERR_INVALID_ARG, "score_eval_device arguments");
  if (n_conf == 0) return DSDP_OK;
  if ((flags & DSDP_TERM_ALL) == 0 || (flags & ~(uint32_t)DSDP_TERM_ALL))
    return set_error(DSDP_ERR_INVALID_ARG, "flags must select DSDP_TERM_INTER and/or DSDP_TERM_INTRA");
  ScoreLaunch a;
  a.map = map_view_of(grid);
  a.blob = (const uint8_t*)d_blob;
  a.conf = d_conf;
  a.n_conf = n_conf;
  a.energy = d_energy;
  a.grad = d_grad;
  a.flags = flags;
  a.apl = n_atoms <= 32 ? 1 : 2;
  a.n_torsions = T;
  a.blob_smem = (int)((const BlobHeader*)h_blob)->stage_bytes;
  // an evaluation uses the prefix sums alone; the rest of a chain's scratch would take
  // the cache of the maps' corners (100,003 poses of 64 atoms 557 us, with it 604)
  a.scratch = scratch_layout(n_atoms, T);
  a.scratch.bytes = a.scratch.H;
  return check_cuda(launch_score_dispatch(map_fmt(grid->dtype, grid->mode), a, (cudaStream_t)stream),
                    "score_eval_kernel launch");
}

extern "C" dsdp_status dsdp_plan_create(dsdp_ctx* ctx, int32_t n_jobs, const dsdp_job_device* jobs, uint32_t flags,
                                        int32_t tile_config, dsdp_plan** out) {
  return plan_create(ctx, n_jobs, jobs, flags, tile_config, true, out);
}

dsdp_status dsdp::plan_create(dsdp_ctx* ctx, int n_jobs, const dsdp_job_device* jobs, uint32_t flags, int tile_config,
                              bool alone, dsdp_plan** out) {
  if (!out) return set_error(DSDP_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (n_jobs < 1 || !jobs) return set_error(DSDP_ERR_INVALID_ARG, "plan needs >= 1 job");
  if (tile_config < 0 || tile_config > 12) return set_error(DSDP_ERR_INVALID_ARG, "tile_config outside 0..12");
  std::vector<DevJob> dj(n_jobs);
  std::vector<int> fmt(n_jobs), apl(n_jobs), blob_bytes(n_jobs), pairs(n_jobs), atoms(n_jobs), tors(n_jobs);
  size_t scratch = 0;
  int max_chains = 0;
  for (int j = 0; j < n_jobs; ++j) {
    const dsdp_job_device& J = jobs[j];
    dsdp_status s = check_view(&J.grid);
    if (s != DSDP_OK) return s;
    s = dsdp_ligand_blob_info(J.h_blob, &atoms[j], &tors[j], &pairs[j], nullptr);
    if (s != DSDP_OK) return s;
    if (!J.d_blob) return set_error(DSDP_ERR_INVALID_ARG, "job %d: d_blob NULL", j);
    dsdp_dock_params p;
    s = normalize_params(&J.params, &p);
    if (s != DSDP_OK) return s;
    if (!(flags & DSDP_PLAN_NO_RESCORE) && (J.receptor.n < 1 || !J.receptor.xyz || !J.receptor.xs_type))
      return set_error(DSDP_ERR_INVALID_ARG, "job %d: rescoring needs the receptor's device arrays", j);
    for (int a = 0; a < 3; ++a)
      if (!(J.box_size[a] >= 0.0) || !isfinite(J.box_lo[a]))
        return set_error(DSDP_ERR_INVALID_ARG, "job %d: search box invalid", j);
    if (p.trace && !J.d_trace) return set_error(DSDP_ERR_INVALID_ARG, "job %d: trace requested without d_trace", j);
    if (p.n_site_points > 0 && !J.d_site_points)
      return set_error(DSDP_ERR_INVALID_ARG, "job %d: n_site_points > 0 without d_site_points", j);
    fmt[j] = map_fmt(J.grid.dtype, J.grid.mode);
    apl[j] = atoms[j] <= 32 ? 1 : 2;
    blob_bytes[j] = (int)((const BlobHeader*)J.h_blob)->stage_bytes;
    max_chains = std::max(max_chains, p.n_chains);
    const int nx = 7 + tors[j];
    if (!J.d_chain_best_conf) scratch += up256(sizeof(float) * (size_t)p.n_chains * nx);
    if (!J.d_chain_best_e) scratch += up256(sizeof(float) * (size_t)p.n_chains);
    if (!J.d_chain_evals) scratch += up256(sizeof(uint32_t) * (size_t)p.n_chains);
    scratch += 3 * up256(sizeof(double) * (size_t)p.n_chains);
    scratch += up256(coord_bytes(p.n_chains, atoms[j], tors[j]));
    DevJob& d = dj[j];
    memset(&d, 0, sizeof(d));
    d.blob = (const uint8_t*)J.d_blob;
    d.maps = J.grid.d_maps;
    for (int a = 0; a < 3; ++a) {
      d.n[a] = J.grid.n[a];
      d.origin[a] = (float)J.grid.origin[a];
      d.box_lo[a] = (float)J.box_lo[a];
      d.box_size[a] = (float)J.box_size[a];
    }
    d.spacing = (float)J.grid.spacing;
    d.inv_spacing = (float)(1.0 / J.grid.spacing);
    d.dtype = J.grid.dtype;
    d.mode = J.grid.mode;
    d.n_chains = p.n_chains;
    d.n_steps = p.n_mc_steps;
    d.n_opt_iters = p.n_opt_iters;
    d.optimizer = p.optimizer;
    d.temperature = (float)p.temperature;
    d.seed_lo = (uint32_t)(p.seed & 0xffffffffu);
    d.seed_hi = (uint32_t)(p.seed >> 32);
    d.chain_best_conf = J.d_chain_best_conf;
    d.chain_best_e = J.d_chain_best_e;
    d.chain_evals = J.d_chain_evals;
    d.trace = p.trace ? J.d_trace : nullptr;
    d.trace_starts = p.trace == 2;
    d.sites = p.n_site_points > 0 ? J.d_site_points : nullptr;
    d.n_sites = p.n_site_points;
    d.site_r2 = p.site_radius * p.site_radius;
    d.n_rec = J.receptor.n;
    d.rec_xyz = J.receptor.xyz;
    d.rec_type = J.receptor.xs_type;
    d.top_k = p.top_k;
    d.rmsd_dedup = (float)p.rmsd_dedup;
    d.out_n = J.d_out_n;
    d.out_chain = J.d_out_chain;
    d.out_score = J.d_out_score;
    d.out_inter = J.d_out_inter;
    d.out_intra = J.d_out_intra;
    d.out_conf = J.d_out_conf;
    d.out_coords = J.d_out_coords;
  }
  dsdp_plan* P = new dsdp_plan();
  P->ctx = ctx;
  P->n_jobs = n_jobs;
  P->flags = flags;
  P->max_chains = max_chains;
  P->sms = ctx_sm_count(ctx);
  P->l2_bytes = device_l2_bytes();
  size_t total_chains = 0, max_blocks = 0;
  bool all_bfgs = true, any_bfgs = false;
  {
    // Length of a job's chains, relative: evaluations (MC steps; Barzilai-Borwein
    // runs all its iterations, BFGS about 60 of 100) times the cost of one (the
    // intra pair steps are half of a 30-atom evaluation, the rest does not depend
    // on the ligand much beyond its tile).
    double longest = 1e-9;
    P->shape.resize(n_jobs);
    for (int j = 0; j < n_jobs; ++j) {
      const BlobHeader* h = (const BlobHeader*)jobs[j].h_blob;
      const double cost = (dj[j].n_steps + 1.0) * (dj[j].optimizer == DSDP_OPT_BB ? 1.6 : 1.0) *
                          (dj[j].n_opt_iters + 1.0) * (14.0 * apl[j] + h->n_steps);
      const size_t map_bytes = (size_t)DSDP_NUM_MAP_TYPES * dj[j].n[0] * dj[j].n[1] * dj[j].n[2] *
                               fmt_channels(fmt[j]) * fmt_elem_bytes(fmt[j]);
      const bool bfgs = dj[j].optimizer == DSDP_OPT_BFGS;
      P->shape[j] = dsdp_plan::Shape{fmt[j], apl[j], blob_bytes[j], atoms[j], tors[j], dj[j].n_chains,
                                     cost,   0,      dj[j].maps,    map_bytes, bfgs};
      longest = std::max(longest, cost);
      total_chains += (size_t)dj[j].n_chains;
    }
    for (int j = 0; j < n_jobs; ++j) {
      const bool bfgs = dj[j].optimizer == DSDP_OPT_BFGS;
      all_bfgs = all_bfgs && bfgs;
      any_bfgs = any_bfgs || bfgs;
    }
    P->any_bfgs = any_bfgs;
    P->resident = total_chains <= (size_t)16 * P->sms;
    P->job_order.resize(n_jobs);
    for (int j = 0; j < n_jobs; ++j) {
      P->job_order[j] = j;
      // slices of about the same length whatever the job
      const int steps = dj[j].n_steps + 1, rounds = P->resident ? kSliceRoundsResident : kSliceRounds;
      const int want = (int)ceil(rounds * P->shape[j].cost / longest);
      dj[j].slice_steps = (steps + want - 1) / want;
      P->shape[j].slices = (steps + dj[j].slice_steps - 1) / dj[j].slice_steps;
      max_blocks += P->shape[j].slices;
    }
    std::stable_sort(P->job_order.begin(), P->job_order.end(),
                     [&](int a, int b) { return P->shape[a].cost > P->shape[b].cost; });
  }
  int W = 1;
  {
    uint32_t fmt_mask = 0;
    int apl_max = 1;
    for (const dsdp_plan::Shape& g : P->shape) {
      fmt_mask |= 1u << g.fmt;
      apl_max = std::max(apl_max, g.apl);
    }
    // By the number of chains.  Up to 8 per SM: teams, or (Barzilai-Borwein has no line
    // search) one warp per chain, ligands above 32 atoms, whose staged blobs are large, in
    // tiles of 4 chains.  More: the time-sliced queue, one chain per CTA (16 typical-4k
    // systems 29.6 ms, in tiles of 2 and 4 31.0 and 33).  From two waves of 16 per SM on
    // the 96-register kernel, whose 20 resident warps per SM issue more per cycle, below
    // the 128-register kernel, whose fewer instructions per evaluation win on a
    // part-filled GPU.
    P->apl_max = apl_max;
    const size_t wave = (size_t)16 * P->sms;
    const bool many = total_chains > wave / 2;
    dsdp_plan::Arrangement& A = P->automatic;
    A.variant = total_chains >= 2 * wave ? 1 : 0;
    A.queue = many;
    A.team = all_bfgs && alone ? team_warps(total_chains, P->sms) : 1;
    A.warps = apl_max == 2 && !many ? 4 : 1;
    P->tune_key = tune_key(fmt_mask, apl_max, total_chains, all_bfgs, any_bfgs, A, P->sms);
    int var = A.variant, pers = (flags & DSDP_PLAN_PERSISTENT) ? 1 : 0;
    if (tile_config == 0) {
      W = A.warps;
      if (tune_lookup(P->tune_key, &var, &pers, &W)) {
        if (pers) P->flags |= DSDP_PLAN_PERSISTENT;
      } else {
        P->auto_queue = A.queue;
        P->team = pers ? 1 : A.team;
      }
    } else {
      var = (tile_config - 1) % 4;
      W = 1 << ((tile_config - 1) / 4);
    }
    P->variant = var;
  }
  std::vector<Tile> rtiles;
  const int rw = rescore_tile_chains();
  for (int j = 0; j < n_jobs; ++j)
    for (int c = 0; c < dj[j].n_chains; c += rw) rtiles.push_back(Tile{j, c, std::min(rw, dj[j].n_chains - c), 0});
  P->n_rtiles = (int)rtiles.size();
  const size_t b_jobs = up256(sizeof(DevJob) * n_jobs),
               b_tiles = up256(sizeof(Tile) * total_chains) * (P->automatic.team > 1 ? 2 : 1),
               b_rtiles = up256(sizeof(Tile) * rtiles.size()), b_blocks = up256(sizeof(SliceBlock) * max_blocks);
  P->queue_next_off = 2 * kMaxGroups + total_chains;
  // (tiles of W <= 4 may be part filled)
  P->queue_bytes = sizeof(int) * (2 * kMaxGroups + 2 * total_chains + 4 * (size_t)n_jobs);
  const size_t b_cnt = up256(P->queue_bytes);
  P->arena_bytes = b_jobs + b_tiles + b_rtiles + b_blocks + b_cnt + scratch;
  P->arena = ctx_alloc(ctx, P->arena_bytes, nullptr);
  if (!P->arena) {
    const size_t bytes = P->arena_bytes;
    delete P;
    return set_error(DSDP_ERR_OUT_OF_MEMORY, "plan arena of %zu bytes", bytes);
  }
  uint8_t* a = (uint8_t*)P->arena;
  P->d_jobs = a;
  P->d_tiles = a + b_jobs;
  if (P->automatic.team > 1) P->d_singles = a + b_jobs + b_tiles / 2;
  P->d_rtiles = a + b_jobs + b_tiles;
  P->d_blocks = a + b_jobs + b_tiles + b_rtiles;
  P->d_queue = (int*)(a + b_jobs + b_tiles + b_rtiles + b_blocks);
  uint8_t* sc = a + b_jobs + b_tiles + b_rtiles + b_blocks + b_cnt;
  for (int j = 0; j < n_jobs; ++j) {
    DevJob& d = dj[j];
    const int nx = 7 + tors[j];
    auto take = [&](size_t bytes) {
      uint8_t* p = sc;
      sc += up256(bytes);
      return p;
    };
    if (!d.chain_best_conf) d.chain_best_conf = (float*)take(sizeof(float) * (size_t)d.n_chains * nx);
    if (!d.chain_best_e) d.chain_best_e = (float*)take(sizeof(float) * (size_t)d.n_chains);
    if (!d.chain_evals) d.chain_evals = (uint32_t*)take(sizeof(uint32_t) * (size_t)d.n_chains);
    d.chain_score = (double*)take(sizeof(double) * (size_t)d.n_chains);
    d.chain_inter = (double*)take(sizeof(double) * (size_t)d.n_chains);
    d.chain_intra = (double*)take(sizeof(double) * (size_t)d.n_chains);
    d.record_bytes = slice_record_bytes(tors[j]);
    d.chain_coords = (double*)take(coord_bytes(d.n_chains, atoms[j], tors[j]));
  }
  cudaError_t e = cudaMemcpy(P->d_jobs, dj.data(), sizeof(DevJob) * n_jobs, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = plan_use_warps(P, W);
  if (e == cudaSuccess && !rtiles.empty())
    e = cudaMemcpy(P->d_rtiles, rtiles.data(), sizeof(Tile) * rtiles.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    ctx_free(ctx, P->arena, P->arena_bytes, nullptr);
    delete P;
    return check_cuda(e, "plan upload");
  }
  track_flight(&P->flight, (int)total_chains);
  *out = P;
  return DSDP_OK;
}

extern "C" int32_t dsdp_plan_kernel_count(const dsdp_plan* P) {
  if (!P) return 0;
  int n = (int)P->groups.size();
  if (P->auto_queue && P->any_bfgs && (P->resident || n == 1)) n *= 2;  // teams for the chains left over
  if (!(P->flags & DSDP_PLAN_NO_RESCORE)) n += 2;
  return n;
}

extern "C" int32_t dsdp_plan_team(const dsdp_plan* P) { return P ? P->last_team : 0; }

static int config_number(int variant, int warps, bool persistent) {
  return 1 + variant + 4 * (warps == 4 ? 2 : warps - 1) + (persistent ? 12 : 0);
}

extern "C" int32_t dsdp_plan_config(const dsdp_plan* P) {
  if (!P || P->auto_queue || P->team > 1) return 0;
  return config_number(P->variant, P->warps_per_cta, P->flags & DSDP_PLAN_PERSISTENT);
}

extern "C" dsdp_status dsdp_plan_launch_stage(dsdp_plan* P, uint32_t stages, void* stream) {
  if (!P) return set_error(DSDP_ERR_INVALID_ARG, "plan is NULL");
  if (stages == 0 || (stages & ~(uint32_t)DSDP_STAGE_ALL)) return set_error(DSDP_ERR_INVALID_ARG, "bad stages");
  const cudaStream_t st = (cudaStream_t)stream;
  const ChainQueueMode queue = queue_mode(P);
  int team = P->team;
  const bool lone = !P->ctx && P->groups.size() == 1 && !P->resident;
  size_t others = 0;  // chains under way on other streams
  bool track = false;
  if (stages & DSDP_STAGE_CHAINS) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(st, &capture);
    if (e != cudaSuccess) cudaGetLastError();
    track = e == cudaSuccess && capture == cudaStreamCaptureStatusNone;
    if (track && P->flight.done && (team > 1 || (lone && P->groups[0].misses_less)))
      others = chains_in_flight(P->flight, st);
    if (others) team = shared_team_warps(team, (size_t)P->flight.chains, others, P->apl_max, P->sms);
    P->last_team = team;
  }
  if ((stages & DSDP_STAGE_CHAINS) && queue != kNoQueue) {
    const cudaError_t e = cudaMemsetAsync(P->d_queue, 0, P->queue_bytes, st);
    if (e != cudaSuccess) return check_cuda(e, "plan queue reset");
  }
  for (size_t gi = 0; (stages & DSDP_STAGE_CHAINS) && gi < P->groups.size(); ++gi) {
    const dsdp_plan::Group& g = P->groups[gi];
    ChainLaunch a;
    a.jobs = P->d_jobs;
    a.tiles = (const Tile*)P->d_tiles + g.first_tile;
    a.n_tiles = g.n_tiles;
    a.queue = queue;
    a.counter = P->d_queue + gi;
    a.exited = P->d_queue + kMaxGroups + gi;
    a.tickets = P->d_queue + 2 * kMaxGroups + g.first_tile;
    a.next_step = P->d_queue + P->queue_next_off + (size_t)g.first_tile * P->warps_per_cta;
    a.blocks = (const SliceBlock*)P->d_blocks + g.first_block;
    a.n_blocks = g.n_blocks;
    a.n_items = g.n_items;
    a.warps_per_cta = P->warps_per_cta;
    a.apl = g.apl;
    a.apl_mask = g.apl_mask;
    a.more_smem = g.misses_less && lone && others == 0;
    a.blob_smem = (g.blob_smem + 15) & ~15;
    a.scratch = scratch_layout(g.max_atoms, g.max_torsions);
    a.overlap = gi > 0 && queue != kNoQueue;
    a.variant = P->variant;
    // 96 registers are for more than 16 warps per SM: where the ligands' shared memory
    // allows no more, the 128-register kernel (64 ligands of 10-60 atoms 59.6 against
    // 62.1 ms)
    if (P->auto_queue && a.variant == 1 &&
        kSmemPerSm / (a.blob_smem + a.warps_per_cta * a.scratch.bytes + 1024) * a.warps_per_cta <= 16)
      a.variant = 0;
    a.team = team;
    if (team > 1) {
      a.tiles = (const Tile*)P->d_singles + g.first_chain;
      a.n_tiles = g.n_chains;
    }
    a.team_resumes = false;
    a.team_when = P->auto_queue && P->any_bfgs && (P->resident || P->groups.size() == 1) ? kTailTeams * P->sms : 0;
    cudaError_t e = launch_chains_dispatch(g.fmt, a, st);
    if (e != cudaSuccess) return check_cuda(e, "dock_chains_kernel launch");
    if (a.team_when) {  // the chains it leaves
      a.team = 4;
      a.team_resumes = true;
      e = launch_chains_dispatch(g.fmt, a, st);
      if (e != cudaSuccess) return check_cuda(e, "dock_team_kernel launch");
    }
  }
  if (track) mark_flight(&P->flight, st);
  if ((stages & DSDP_STAGE_RESCORE) && !(P->flags & DSDP_PLAN_NO_RESCORE)) {
    cudaError_t e = launch_rescore(P->d_jobs, P->d_rtiles, P->n_rtiles, st);
    if (e != cudaSuccess) return check_cuda(e, "rescore_kernel launch");
    e = launch_topk(P->d_jobs, P->n_jobs, P->max_chains, st);
    if (e != cudaSuccess) return check_cuda(e, "topk_kernel launch");
  }
  return DSDP_OK;
}

extern "C" dsdp_status dsdp_plan_launch(dsdp_plan* P, void* stream) {
  return dsdp_plan_launch_stage(P, DSDP_STAGE_ALL, stream);
}

extern "C" dsdp_status dsdp_plan_autotune(dsdp_plan* P, void* stream, int32_t repeats, int32_t* chosen,
                                          float* ms_by_config) {
  if (!P) return set_error(DSDP_ERR_INVALID_ARG, "plan is NULL");
  if (ms_by_config)
    for (int i = 0; i < 24; ++i) ms_by_config[i] = -1.f;
  if (repeats < 1) repeats = 1;
  const cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaStreamSynchronize(st);  // a launch before may still read the tiles
  if (e != cudaSuccess) return check_cuda(e, "autotune");
  cudaEvent_t a, b;
  e = cudaEventCreate(&a);
  if (e == cudaSuccess) e = cudaEventCreate(&b);
  if (e != cudaSuccess) return check_cuda(e, "autotune events");
  const uint32_t base_flags = P->flags & ~(uint32_t)DSDP_PLAN_PERSISTENT;
  // the automatic arrangement (queue when needed, teams) first: kept if nothing beats it
  const dsdp_plan::Arrangement& A = P->automatic;
  auto use_automatic = [&] {
    P->flags = base_flags;
    P->variant = A.variant;
    P->auto_queue = A.queue;
    P->team = A.team;
    return plan_use_warps(P, A.warps);
  };
  float auto_ms = 1e30f;
  float best = 1e30f;
  int best_var = P->variant, best_pers = (P->flags & DSDP_PLAN_PERSISTENT) ? 1 : 0, best_w = P->warps_per_cta;
  dsdp_status s = DSDP_OK;
  auto measure = [&](float* ms) {
    dsdp_status r = dsdp_plan_launch_stage(P, DSDP_STAGE_CHAINS, stream);  // warm-up
    if (r != DSDP_OK) return r;
    cudaEventRecord(a, st);
    for (int k = 0; k < repeats && r == DSDP_OK; ++k) r = dsdp_plan_launch_stage(P, DSDP_STAGE_CHAINS, stream);
    cudaEventRecord(b, st);
    const cudaError_t ee = cudaEventSynchronize(b);
    if (ee != cudaSuccess) return check_cuda(ee, "autotune run");
    cudaEventElapsedTime(ms, a, b);
    return r;
  };
  if (A.queue || A.team > 1) {  // else it is one of the fixed ones
    s = check_cuda(use_automatic(), "autotune tiles");
    if (s == DSDP_OK) s = measure(&auto_ms);
  }
  P->auto_queue = false;  // with and without the queue are measured apart
  P->team = 1;
  for (int c = 0; c < 6 && s == DSDP_OK; ++c) {
    const int w = 1 << (c / 2), pers = c % 2;
    P->flags = base_flags | (pers ? DSDP_PLAN_PERSISTENT : 0u);
    e = plan_use_warps(P, w);
    if (e != cudaSuccess) {
      s = check_cuda(e, "autotune tiles");
      break;
    }
    // register budgets compiled: 128, 96, 80, 72 for one atom per lane, 128 and
    // 96 for two and for mixed tiles (launch_chains_impl)
    int n_var = 2;
    for (const dsdp_plan::Group& g : P->groups) n_var = std::max(n_var, g.apl_mask == 1 ? 4 : 2);
    for (int var = 0; var < n_var && s == DSDP_OK; ++var) {
      P->variant = var;
      float ms = 0.f;
      s = measure(&ms);
      if (s != DSDP_OK) break;
      if (ms_by_config) ms_by_config[config_number(var, w, pers) - 1] = ms / repeats;
      if (ms < best) {
        best = ms;
        best_var = var;
        best_pers = pers;
        best_w = w;
      }
    }
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  if (chosen) *chosen = config_number(best_var, best_w, best_pers);
  if (s == DSDP_OK && auto_ms <= best) {  // later plans of this shape find it by themselves
    tune_erase(P->tune_key);
    return check_cuda(use_automatic(), "plan tiles");
  }
  P->variant = best_var;
  P->flags = base_flags | (best_pers ? DSDP_PLAN_PERSISTENT : 0u);
  if (s == DSDP_OK) s = check_cuda(plan_use_warps(P, best_w), "plan tiles");
  if (s != DSDP_OK) return s;
  tune_store(P->tune_key, best_var, best_pers, best_w);
  return DSDP_OK;
}

extern "C" dsdp_status dsdp_plan_destroy(dsdp_ctx* ctx, dsdp_plan* P) {
  if (!P) return DSDP_OK;
  untrack_flight(&P->flight);
  if (P->arena) ctx_free(ctx ? ctx : P->ctx, P->arena, P->arena_bytes, nullptr);
  delete P;
  return DSDP_OK;
}
