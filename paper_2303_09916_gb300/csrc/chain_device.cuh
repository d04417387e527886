// Warp-per-chain score + gradient, local optimisers and Monte Carlo chain.
//
// One warp owns one conformation.  Lanes hold atoms (APL atoms per lane, in
// the blob's depth-first order), rigid bodies (lane b = body b) and the
// components of 6 + T dimensional vectors (lane j = component j: 0..2
// position, 3..5 rotation vector, 6 + k torsion k).  The ligand topology sits
// in shared memory; grid maps are read from L2 through the read-only path.
#pragma once
#include "device_common.cuh"

namespace dsdp {

// Pointers into a staged (shared-memory) blob.
struct LigView {
  const BlobHeader* h;
  const float4* atom;
  const int32_t* atom_user;
  const BodyRec* body;
  const uint2* pair_rec;  // after the staged prefix: read from the global blob only
  const uint2* steps;
  const int32_t* torsion_body;
  const int16_t* lane_map;  // [32][2]: atom in slot s of lane l (-1 empty); lane l holds atom l up to 32 atoms
  int n_atoms, T, n_bodies, n_pairs, n_steps, rounds;
};

__device__ __forceinline__ LigView view_blob(const uint8_t* b) {
  LigView v;
  v.h = reinterpret_cast<const BlobHeader*>(b);
  v.atom = reinterpret_cast<const float4*>(b + v.h->off_atom);
  v.atom_user = reinterpret_cast<const int32_t*>(b + v.h->off_atom_user);
  v.body = reinterpret_cast<const BodyRec*>(b + v.h->off_body);
  v.pair_rec = reinterpret_cast<const uint2*>(b + v.h->off_pairs);
  v.steps = reinterpret_cast<const uint2*>(b + v.h->off_steps);
  v.torsion_body = reinterpret_cast<const int32_t*>(b + v.h->off_torsion_body);
  v.lane_map = reinterpret_cast<const int16_t*>(b + v.h->off_lane_map);
  v.n_atoms = v.h->n_atoms;
  v.T = v.h->n_torsions;
  v.n_bodies = v.h->n_bodies;
  v.n_pairs = v.h->n_pairs;
  v.n_steps = v.h->n_steps;
  v.rounds = v.h->rounds;
  return v;
}

// Stages a ligand's blob into shared memory (all threads of the CTA; no barrier before,
// one after) and notes at each body the lane of its parent's first atom, which one
// atom per lane is that atom's index.
__device__ __forceinline__ void stage_blob(uint8_t* smem, const uint8_t* blob, int bytes) {
  for (int i = threadIdx.x; i < bytes / 16; i += blockDim.x)
    reinterpret_cast<int4*>(smem)[i] = __ldg(reinterpret_cast<const int4*>(blob) + i);
  __syncthreads();
  const BlobHeader* h = reinterpret_cast<const BlobHeader*>(smem);
  BodyRec* body = reinterpret_cast<BodyRec*>(smem + h->off_body);
  if (threadIdx.x < h->n_bodies)
    body[threadIdx.x].parent_lane = body[threadIdx.x].parent >= 0 ? body[body[threadIdx.x].parent].atom_begin : -1;
  __syncthreads();
}

// Per-lane ligand data: the atoms of the lane's slots (atom lane with one atom
// per lane; the blob's lane map with two) and, on lane b < n_bodies, body b's
// record; re-read from the staged blob (shared memory) where used.
template <int APL>
struct LaneLig {
  int n_atoms, nb, T, tbody;
};

// Steps [0, n) may hold hydrophobic or H-bond pairs, [n, n_steps) hold none; n is
// even.  (The steps with such pairs come first; bits 14 / 15 are the same in every lane.)
__device__ __forceinline__ int ramp_steps(const LigView& L) {
  int n = 0;
  while (n < L.n_steps && ((L.steps[32 * n].x | L.steps[32 * n + 32].x) & 0xc000u)) n += 2;
  return n;
}

template <int APL>
__device__ __forceinline__ void load_lane_lig(const LigView& L, LaneLig<APL>& R) {
  const int lane = threadIdx.x & 31;
  R.n_atoms = L.n_atoms;
  R.nb = L.n_bodies;
  R.T = L.T;
  R.tbody = (lane >= 6 && lane < 6 + L.T) ? L.torsion_body[lane - 6] : 0;  // the lane with that body's gradient
  if (APL == 1) R.tbody = L.body[R.tbody].atom_begin;
}

// Conformation held by a warp: p and q replicated in every lane, torsion k in lane 6 + k.
struct Conf {
  float3 p;
  Quat q;
  float th;
};

// Per-warp shared scratch (layout in scratch_layout).
struct WarpScratch {
  float4* pre;     // inclusive prefix sums of (g, (r - p) x g): [n_atoms] (gx, gy, gz, cx), then [n_atoms] (cy, cz)
  float* H;        // [6 + T][kHStride] BFGS inverse Hessian, row j owned by lane j
  float* vec;      // [5][kHStride] + kVarWords: g', s, u broadcast to the H rows (BFGS update);
                   // the chain's g and d; its ChainVars
  float* x;        // [7 + kMaxDim] local optimiser: current iterate (BFGS) / best iterate (BB)
  float* cur;      // [7 + kMaxDim] current conformation of the chain
  float* best;     // [7 + kMaxDim] best conformation of the chain
};

constexpr int kConfFloats = 7 + kMaxDim;
constexpr int kVarWords = 24;  // words of the scratch's ChainVars
// Row stride of H (floats): >= kMaxDim rounded up to float4, and 7 float4 per row
// so that rows j = 0..7 fall on distinct 16-byte bank groups (float4 row reads
// by the lanes need the minimum number of shared-memory wavefronts).
constexpr int kHStride = 28;
static_assert(kHStride >= ((kMaxDim + 3) & ~3) && (kHStride / 4) % 2 == 1, "H row stride");
__host__ __device__ constexpr int align16i(int x) { return (x + 15) & ~15; }
// Per-warp scratch sized for a group's largest ligand (n_atoms, torsions).
struct ScratchLayout {
  int pre, H, vec, x, cur, best, bytes;
};
__host__ __device__ inline ScratchLayout scratch_layout(int n_atoms, int n_torsions) {
  ScratchLayout l;
  const int D = 6 + n_torsions;
  l.pre = 0;
  l.H = l.pre + align16i(24 * n_atoms);
  l.vec = l.H + align16i(4 * kHStride * D);
  l.x = l.vec + align16i(4 * (5 * kHStride + kVarWords));
  l.cur = l.x + align16i(4 * kConfFloats);
  l.best = l.cur + align16i(4 * kConfFloats);
  l.bytes = l.best + align16i(4 * kConfFloats);
  return l;
}
__device__ __forceinline__ WarpScratch warp_scratch_at(uint8_t* base, const ScratchLayout& l) {
  WarpScratch W;
  W.pre = reinterpret_cast<float4*>(base + l.pre);
  W.H = reinterpret_cast<float*>(base + l.H);
  W.vec = reinterpret_cast<float*>(base + l.vec);
  W.x = reinterpret_cast<float*>(base + l.x);
  W.cur = reinterpret_cast<float*>(base + l.cur);
  W.best = reinterpret_cast<float*>(base + l.best);
  return W;
}

// Body frames for a conformation: the lane returns the world rotation Q and origin O
// of body `body`, composed from the local transforms by pointer jumping
// (ceil(log2(depth + 1)) rounds of shuffles).  OF_ATOM: the body of the lane's atom
// (the parent's frame is at the parent's first atom, stage_blob); else body = lane,
// nothing beyond n_bodies.
template <bool OF_ATOM>
__device__ __forceinline__ void body_frames(const LigView& L, const Conf& c, int body, Quat& Q, float3& O) {
  const int lane = threadIdx.x & 31;
  const bool child = body > 0 && (OF_ATOM || lane < L.n_bodies);
  float4 b0 = make_float4(0.f, 0.f, 0.f, 0.f), b1 = b0;
  int parent_lane = -1;
  if (child) {
    const float4* rec = reinterpret_cast<const float4*>(L.body + body);
    b0 = rec[0];  // off xyz, parent
    b1 = rec[1];  // axis xyz, torsion
    parent_lane = OF_ATOM ? L.body[body].parent_lane : __float_as_int(b0.w);
  }
  const int tors = __float_as_int(b1.w);
  const float tb = __shfl_sync(kFull, c.th, child ? 6 + tors : 0);
  int ptr = -1;
  if (child) {
    const float s = sin_ftz(0.5f * tb), co = cos_ftz(0.5f * tb);  // |theta / 2| <= pi / 2: absolute error < 4e-7
    Q = Quat{co, s * b1.x, s * b1.y, s * b1.z};
    O = make_float3(b0.x, b0.y, b0.z);
    ptr = parent_lane;
  } else if (OF_ATOM || lane == 0) {
    Q = c.q;
    O = c.p;
  } else {
    Q = Quat{1.f, 0.f, 0.f, 0.f};
    O = make_float3(0.f, 0.f, 0.f);
  }
  for (int r = 0; r < L.rounds; ++r) {
    const int src = ptr >= 0 ? ptr : lane;
    const Quat Qp = shflq(Q, src);
    const float3 Op = shfl3(O, src);
    const int pp = __shfl_sync(kFull, ptr, src);
    if (ptr >= 0) {
      O = Op + qrot(Qp, O);
      Q = qmul(Qp, Q);
      ptr = pp;
    }
  }
}

// A conformation's atoms and body frames.  Two atoms per lane: lane b < n_bodies holds
// body b's frame.  One: every lane holds the frame of its own atom's body, which
// saves fetching it for the atom (seven shuffles); what is done once per body is
// done on the lane of its first atom.
template <int APL>
struct Placed {
  Quat Q;
  float3 O;
  float3 pos[APL];
  int type[APL];  // map type | body << 8
  int atom[APL];  // the slot's atom, -1 when empty
};

template <int APL>
__device__ __forceinline__ void place_atoms(const LigView& L, const Conf& c, Placed<APL>& P) {
  const int lane = threadIdx.x & 31;
  if (APL == 1) {
    P.atom[0] = lane < L.n_atoms ? lane : -1;
    const float4 a = L.atom[lane < L.n_atoms ? lane : 0];
    P.type[0] = __float_as_int(a.w);
    const int b = P.type[0] >> 8;
    body_frames<true>(L, c, b, P.Q, P.O);
    P.pos[0] = P.O + qrot(P.Q, make_float3(a.x, a.y, a.z));
    return;
  }
  body_frames<false>(L, c, lane, P.Q, P.O);
#pragma unroll
  for (int s = 0; s < APL; ++s) {
    P.atom[s] = (int)L.lane_map[2 * lane + s];
    const int i = P.atom[s];
    const float4 a = L.atom[i >= 0 ? i : 0];
    P.type[s] = __float_as_int(a.w);
    const int b = i >= 0 ? (P.type[s] >> 8) & 0xff : 0;
    const Quat Qb = shflq(P.Q, b);
    const float3 Ob = shfl3(P.O, b);
    P.pos[s] = Ob + qrot(Qb, make_float3(a.x, a.y, a.z));
  }
}

// Energy of a placed conformation (all lanes return the same), without its
// gradient: a BFGS line search rejects three of four trial points and needs
// nothing else of those.  The operations that make up the energy, and their
// order, are score_placed's: both return the same bits.
template <int APL, int FMT, int IU = 2>
__device__ __forceinline__ float energy_placed(const MapView& M, const LigView& L, int n_ramp, const Placed<APL>& P) {
  const int lane = threadIdx.x & 31;
  const uint2* tab = L.steps + lane;
  // One atom a lane: the corners' loads first, on their way while the pairs are
  // computed (two atoms' 16 corners, and the kernel for both tile sizes, have not the
  // registers): 32 typical-4k systems 52.2 -> 51.5 ms.  A slot without an atom reads
  // atom 0's corners.
  constexpr bool kEarly = APL == 1 && IU == 2;
  CornerPairs corners;
  if constexpr (kEarly) corners = load_corner_pairs<FMT>(M, P.type[0] & 0xff, map_cell(M, P.pos[0]).base);
  float2 e_pair = make_float2(0.f, 0.f);
  const float2 px = splat2(P.pos[0].x), py = splat2(P.pos[0].y), pz = splat2(P.pos[0].z);
  auto pass = [&](int st, bool ramp) {
    const uint2 t0 = tab[st * 32], t1 = tab[st * 32 + 32];
    float2 dx, dy, dz;
    if (APL == 1) {
      const float3 b0 = shfl3(P.pos[0], (int)t0.x), b1 = shfl3(P.pos[0], (int)t1.x);
      dx = __ffma2_rn(make_float2(b0.x, b1.x), splat2(-1.f), px);
      dy = __ffma2_rn(make_float2(b0.y, b1.y), splat2(-1.f), py);
      dz = __ffma2_rn(make_float2(b0.z, b1.z), splat2(-1.f), pz);
    } else {
      const float3 lo = P.pos[0], hi = P.pos[APL - 1];
      const float3 a0 = t0.x & (1u << 10) ? hi : lo, a1 = t1.x & (1u << 10) ? hi : lo;
      const float3 s0 = t0.x & (1u << 11) ? hi : lo, s1 = t1.x & (1u << 11) ? hi : lo;
      const float3 b0 = shfl3(s0, (int)t0.x), b1 = shfl3(s1, (int)t1.x);
      dx = make_float2(a0.x - b0.x, a1.x - b1.x);
      dy = make_float2(a0.y - b0.y, a1.y - b1.y);
      dz = make_float2(a0.z - b0.z, a1.z - b1.z);
    }
    const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
    const uint32_t both = t0.x | t1.x;
    e_pair = __fadd2_rn(e_pair, vina_energy_x2(r2, make_float2(__uint_as_float(t0.y), __uint_as_float(t1.y)),
                                               t0.x >> 12, t1.x >> 12, ramp && ((both >> 14) & 1),
                                               ramp && ((both >> 15) & 1)));
  };
  int st = 0;
#pragma unroll 1
  for (; st < n_ramp; st += 2) pass(st, true);
#pragma unroll (APL == 1 ? IU : 1)
  for (; st < L.n_steps; st += 2) pass(st, false);
  float e_lane = 0.f;
  e_lane += e_pair.x + e_pair.y;
#pragma unroll
  for (int s = 0; s < APL; ++s) {
    const MapCell cell = map_cell(M, P.pos[s]);
    if constexpr (!kEarly) corners = load_corner_pairs<FMT>(M, P.type[s] & 0xff, cell.base);
    const float em = map_energy_pairs(cell, corners);
    if (P.atom[s] >= 0) e_lane += em;
  }
  return warp_sum(e_lane);
}

// Score and gradient of a placed conformation c (all lanes return the same E;
// lane j < 6 + T returns gradient component j, other lanes 0).  IU: how many
// step pairs of the one-atom-per-lane intra loop are unrolled.  FLAT: the passes that
// may hold hydrophobic or H-bond pairs compute both terms for all (with weight 0
// where a pair has none: the same bits) instead of branching, and are unrolled too --
// more instructions, a shorter way through them.  RU: how many of those passes.
template <int APL, int FMT, int IU = 2, bool FLAT = false, int RU = FLAT ? 2 : 1>
__device__ __forceinline__ float score_placed(const MapView& M, const LigView& L, const LaneLig<APL>& R,
                                              int n_ramp, const WarpScratch& W, const Conf& c, const Placed<APL>& P,
                                              float& grad, uint32_t flags) {
  const int lane = threadIdx.x & 31;
  const int N = L.n_atoms, nb = L.n_bodies;
  const Quat Q = P.Q;
  const float3 O = P.O;
  float3 pos[APL];
  int type[APL];
  int atom[APL];
#pragma unroll
  for (int s = 0; s < APL; ++s) pos[s] = P.pos[s], type[s] = P.type[s], atom[s] = P.atom[s];
  float e_lane = 0.f;
  float3 g[APL];
#pragma unroll
  for (int s = 0; s < APL; ++s) g[s] = make_float3(0.f, 0.f, 0.f);
  // ---- intra: the pair steps of the blob, two per pass (packed FP32x2 pair
  //      terms).  In a step each lane computes at most one pair -- its active atom
  //      against the passive atom of a partner lane, fetched by shuffle -- and takes
  //      the reaction force of at most one pair back from the lane that computed it.
  if (flags & DSDP_TERM_INTRA) {
    float2 e_pair = make_float2(0.f, 0.f);
    const uint2* tab = L.steps + lane;
    if (APL == 1) {
      // packed accumulators: component .x collects the even steps, .y the odd ones
      const float2 px = splat2(pos[0].x), py = splat2(pos[0].y), pz = splat2(pos[0].z);
      float2 ax = make_float2(0.f, 0.f), ay = ax, az = ax;
      // A pass takes two steps.  The passes with hydrophobic or H-bond pairs come
      // first; the others have no branch, so that unrolled (IU passes) the shuffles of
      // one overlap the arithmetic of the next.
      auto pass = [&](int st, bool ramp) {
        const uint2 t0 = tab[st * 32], t1 = tab[st * 32 + 32];
        // shfl.idx reads the source lane from bits 0-4 only: the entry's partner field
        const float3 b0 = shfl3(pos[0], (int)t0.x), b1 = shfl3(pos[0], (int)t1.x);
        const float2 dx = __ffma2_rn(make_float2(b0.x, b1.x), splat2(-1.f), px);
        const float2 dy = __ffma2_rn(make_float2(b0.y, b1.y), splat2(-1.f), py);
        const float2 dz = __ffma2_rn(make_float2(b0.z, b1.z), splat2(-1.f), pz);
        const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
        const uint32_t both = t0.x | t1.x;  // bits 14 / 15: warp-uniform
        float2 e, sp;
        vina_pair_x2(r2, make_float2(__uint_as_float(t0.y), __uint_as_float(t1.y)), t0.x >> 12, t1.x >> 12,
                     ramp && (FLAT || ((both >> 14) & 1)), ramp && (FLAT || ((both >> 15) & 1)), e, sp);
        e_pair = __fadd2_rn(e_pair, e);
        const float2 fx = __fmul2_rn(sp, dx), fy = __fmul2_rn(sp, dy), fz = __fmul2_rn(sp, dz);
        // reaction forces of the pairs this lane is passive in (source lane: bits 5-9)
        const float3 c0 = shfl3(make_float3(fx.x, fy.x, fz.x), (int)(t0.x >> 5));
        const float3 c1 = shfl3(make_float3(fx.y, fy.y, fz.y), (int)(t1.x >> 5));
        ax = __ffma2_rn(make_float2(c0.x, c1.x), splat2(-1.f), __fadd2_rn(ax, fx));
        ay = __ffma2_rn(make_float2(c0.y, c1.y), splat2(-1.f), __fadd2_rn(ay, fy));
        az = __ffma2_rn(make_float2(c0.z, c1.z), splat2(-1.f), __fadd2_rn(az, fz));
      };
      int st = 0;
#pragma unroll RU
      for (; st < n_ramp; st += 2) pass(st, true);
#pragma unroll IU
      for (; st < L.n_steps; st += 2) pass(st, false);
      g[0].x += ax.x + ax.y;
      g[0].y += ay.x + ay.y;
      g[0].z += az.x + az.y;
    } else {
      auto pass = [&](int st, bool ramp) {
        const uint2 t0 = tab[st * 32], t1 = tab[st * 32 + 32];
        const bool ac0 = t0.x & (1u << 10), ac1 = t1.x & (1u << 10);
        const bool pc0 = t0.x & (1u << 11), pc1 = t1.x & (1u << 11);
        const float3 a0 = ac0 ? pos[APL - 1] : pos[0], a1 = ac1 ? pos[APL - 1] : pos[0];
        const float3 s0 = pc0 ? pos[APL - 1] : pos[0], s1 = pc1 ? pos[APL - 1] : pos[0];
        const float3 b0 = shfl3(s0, (int)t0.x), b1 = shfl3(s1, (int)t1.x);
        const float2 dx = make_float2(a0.x - b0.x, a1.x - b1.x);
        const float2 dy = make_float2(a0.y - b0.y, a1.y - b1.y);
        const float2 dz = make_float2(a0.z - b0.z, a1.z - b1.z);
        const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
        const uint32_t both = t0.x | t1.x;
        float2 e, sp;
        vina_pair_x2(r2, make_float2(__uint_as_float(t0.y), __uint_as_float(t1.y)), t0.x >> 12, t1.x >> 12,
                     ramp && (FLAT || ((both >> 14) & 1)), ramp && (FLAT || ((both >> 15) & 1)), e, sp);
        e_pair = __fadd2_rn(e_pair, e);
        const float2 fx = __fmul2_rn(sp, dx), fy = __fmul2_rn(sp, dy), fz = __fmul2_rn(sp, dz);
        const float3 c0 = shfl3(make_float3(fx.x, fy.x, fz.x), (int)(t0.x >> 5));
        const float3 c1 = shfl3(make_float3(fx.y, fy.y, fz.y), (int)(t1.x >> 5));
        // each force goes to the slot its bit names (per-lane predication, no selects)
        if (ac0) g[APL - 1].x += fx.x, g[APL - 1].y += fy.x, g[APL - 1].z += fz.x;
        else g[0].x += fx.x, g[0].y += fy.x, g[0].z += fz.x;
        if (ac1) g[APL - 1].x += fx.y, g[APL - 1].y += fy.y, g[APL - 1].z += fz.y;
        else g[0].x += fx.y, g[0].y += fy.y, g[0].z += fz.y;
        if (pc0) g[APL - 1].x -= c0.x, g[APL - 1].y -= c0.y, g[APL - 1].z -= c0.z;
        else g[0].x -= c0.x, g[0].y -= c0.y, g[0].z -= c0.z;
        if (pc1) g[APL - 1].x -= c1.x, g[APL - 1].y -= c1.y, g[APL - 1].z -= c1.z;
        else g[0].x -= c1.x, g[0].y -= c1.y, g[0].z -= c1.z;
      };
      int st = 0;
#pragma unroll RU
      for (; st < n_ramp; st += 2) pass(st, true);
#pragma unroll (FLAT ? 2 : 1)
      for (; st < L.n_steps; st += 2) pass(st, false);
    }
    e_lane += e_pair.x + e_pair.y;
  }
  // ---- inter: trilinear score and gradient (Eq. 2, Eq. 4 / Eq. 3)
#pragma unroll
  for (int s = 0; s < APL; ++s) {
    if ((flags & DSDP_TERM_INTER) && atom[s] >= 0) {
      float3 gi;
      // the cell is located here, where it is used, not held across the intra block:
      // it would take eight registers of each atom there
      e_lane += map_interp<FMT>(M, type[s] & 0xff, map_cell(M, pos[s]), gi);
      g[s] = g[s] + gi;
    }
  }
  const float E = warp_sum(e_lane);
  // ---- back-propagation: inclusive prefix sums over atoms (depth-first
  //      order) of (g_i, (r_i - p) x g_i); a subtree is a contiguous range.
  //      With two atoms per lane the lane map is not in atom order: each slot
  //      first parks its raw terms at its atom's place, and lane l then scans
  //      atoms 2l and 2l + 1 of the atom order.
  float2* const pre2 = reinterpret_cast<float2*>(W.pre + N);
  if (APL == 2) {
#pragma unroll
    for (int s = 0; s < APL; ++s) {
      if (atom[s] < 0) continue;
      const float3 t = cross3(pos[s] - c.p, g[s]);
      W.pre[atom[s]] = make_float4(g[s].x, g[s].y, g[s].z, t.x);
      pre2[atom[s]] = make_float2(t.y, t.z);
    }
    __syncwarp();
  }
  float v[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float raw[APL][6];
#pragma unroll
  for (int s = 0; s < APL; ++s) {
    const int i = lane * APL + s;  // atom order
#pragma unroll
    for (int k = 0; k < 6; ++k) raw[s][k] = 0.f;
    if (i >= N) continue;
    if (APL == 1) {
      const float3 t = cross3(pos[s] - c.p, g[s]);
      raw[s][0] = g[s].x, raw[s][1] = g[s].y, raw[s][2] = g[s].z;
      raw[s][3] = t.x, raw[s][4] = t.y, raw[s][5] = t.z;
    } else {
      const float4 h0 = W.pre[i];
      const float2 h1 = pre2[i];
      raw[s][0] = h0.x, raw[s][1] = h0.y, raw[s][2] = h0.z;
      raw[s][3] = h0.w, raw[s][4] = h1.x, raw[s][5] = h1.y;
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] += raw[s][k];
  }
  float inc[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) inc[k] = v[k];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float t = __shfl_up_sync(kFull, inc[k], o);
      if (lane >= o) inc[k] += t;
    }
  }
  if (APL == 2) __syncwarp();  // every raw value read before the prefix overwrites it
  {
    // this lane's atoms (atom order): exclusive prefix of the lane plus its own slots
    float run[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) run[k] = inc[k] - v[k];
#pragma unroll
    for (int s = 0; s < APL; ++s) {
      const int i = lane * APL + s;
      if (i >= N) continue;
#pragma unroll
      for (int k = 0; k < 6; ++k) run[k] += raw[s][k];
      W.pre[i] = make_float4(run[0], run[1], run[2], run[3]);
      pre2[i] = make_float2(run[4], run[5]);
    }
  }
  __syncwarp();
  float tor = 0.f;
  const int body = APL == 1 ? type[0] >> 8 : lane;
  if (body > 0 && (APL == 1 || lane < nb)) {
    const float4* rec = reinterpret_cast<const float4*>(L.body + body);
    const float4 b1 = rec[1];
    const int4 b2 = *reinterpret_cast<const int4*>(rec + 2);  // atom_begin, atom_end, depth, parent_lane
    const float4 h0 = W.pre[b2.y - 1], l0 = W.pre[b2.x - 1];
    const float2 h1 = pre2[b2.y - 1], l1 = pre2[b2.x - 1];
    const float3 G = make_float3(h0.x - l0.x, h0.y - l0.y, h0.z - l0.z);
    const float3 C = make_float3(h0.w - l0.w, h1.x - l1.x, h1.y - l1.y);
    const float3 axis = qrot(Q, make_float3(b1.x, b1.y, b1.z));
    tor = dot3(axis, C - cross3(O - c.p, G));
  }
  const float tv = __shfl_sync(kFull, tor, R.tbody);
  float gl = 0.f;
  if (lane < 6) {
    gl = lane < 4 ? reinterpret_cast<const float*>(W.pre + N - 1)[lane]
                  : reinterpret_cast<const float*>(pre2 + N - 1)[lane - 4];
  } else if (lane < 6 + L.T) {
    gl = tv;
  }
  __syncwarp();  // W.pre is rewritten by the next evaluation
  grad = gl;
  return E;
}

// c (+) s for a step held in lane layout.
__device__ __forceinline__ Conf apply_step(const Conf& c, float s, int T) {
  const int lane = threadIdx.x & 31;
  Conf o;
  o.p = make_float3(c.p.x + __shfl_sync(kFull, s, 0), c.p.y + __shfl_sync(kFull, s, 1),
                    c.p.z + __shfl_sync(kFull, s, 2));
  const Quat dq = quat_from_rotvec(__shfl_sync(kFull, s, 3), __shfl_sync(kFull, s, 4), __shfl_sync(kFull, s, 5));
  o.q = qnormalize(qmul(dq, c.q));
  o.th = (lane >= 6 && lane < 6 + T) ? wrap_angle(c.th + s) : c.th;
  return o;
}

// Four warp sums at once, every lane getting all four.  Transposed butterfly:
// the first two exchanges halve the values each lane carries (lanes with bit 4
// clear keep a, b, the others c, d; then bit 3 picks one of the two), the last
// three sum one value over a group of 8 lanes, and lanes 0, 8, 16, 24 hold a, b,
// c, d: 10 shuffles and 6 adds instead of 20 and 20.
__device__ __forceinline__ void warp_sum4(float& a, float& b, float& c, float& d) {
  const int lane = threadIdx.x & 31;
  const bool hi16 = lane & 16, hi8 = lane & 8;
  float k0 = hi16 ? c : a, k1 = hi16 ? d : b;
  const float s0 = hi16 ? a : c, s1 = hi16 ? b : d;
  k0 += __shfl_xor_sync(kFull, s0, 16);
  k1 += __shfl_xor_sync(kFull, s1, 16);
  float k = hi8 ? k1 : k0;
  k += __shfl_xor_sync(kFull, hi8 ? k0 : k1, 8);
  k += __shfl_xor_sync(kFull, k, 4);
  k += __shfl_xor_sync(kFull, k, 2);
  k += __shfl_xor_sync(kFull, k, 1);
  a = __shfl_sync(kFull, k, 0);
  b = __shfl_sync(kFull, k, 8);
  c = __shfl_sync(kFull, k, 16);
  d = __shfl_sync(kFull, k, 24);
}

// BFGS inverse-Hessian step after an accepted line search (Nocedal & Wright
// Eq. 6.17), lane j holding row j of H and component j of the vectors.  With
// d = -H g and y = g' - g, H y = H g' + d, so one product H g' gives both the
// update and the next direction:
//   H' g' = H g' - rho (s (Hy.g') + Hy (s.g')) + (rho^2 y.Hy + rho) s (s.g').
// H is updated in place as H_jk += s_j u_k - rho Hy_j s_k, u = (rho^2 y.Hy + rho) s
// - rho Hy.  Returns the new direction -H' g' (0 beyond D).
__device__ __forceinline__ float bfgs_update(const WarpScratch& W, int D, float s, float y, float gn, float d) {
  const int lane = threadIdx.x & 31;
  const int D4 = (D + 3) & ~3;
  float* vg = W.vec;
  float* vs = W.vec + kHStride;
  float* vu = W.vec + 2 * kHStride;
  const float4* Hrow = reinterpret_cast<const float4*>(W.H + kHStride * (lane < D ? lane : 0));
  if (lane < D4) vg[lane] = lane < D ? gn : 0.f;
  __syncwarp();
  float hg = 0.f;  // (H g')_lane: four independent partial sums
  if (lane < D) {
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = 0; k < D4; k += 4) {
      const float4 h = Hrow[k >> 2], v = *reinterpret_cast<const float4*>(vg + k);
      acc.x = fmaf(h.x, v.x, acc.x);
      acc.y = fmaf(h.y, v.y, acc.y);
      acc.z = fmaf(h.z, v.z, acc.z);
      acc.w = fmaf(h.w, v.w, acc.w);
    }
    hg = (acc.x + acc.y) + (acc.z + acc.w);
  }
  const float hy = lane < D ? hg + d : 0.f;
  float sy = s * y, yhy = y * hy, hyg = hy * gn, sg = s * gn;
  warp_sum4(sy, yhy, hyg, sg);
  float dn;
  if (sy > kMinCurvature) {
    const float rho = 1.f / sy;
    const float coef = rho * rho * yhy + rho;
    if (lane < D4) {
      vs[lane] = lane < D ? s : 0.f;
      vu[lane] = lane < D ? coef * s - rho * hy : 0.f;
    }
    __syncwarp();
    if (lane < D) {
      float4* Hw = reinterpret_cast<float4*>(W.H + kHStride * lane);
      const float a = -rho * hy;
      for (int k = 0; k < D4; k += 4) {
        float4 h = Hw[k >> 2];
        const float4 u = *reinterpret_cast<const float4*>(vu + k), v = *reinterpret_cast<const float4*>(vs + k);
        h.x = fmaf(s, u.x, fmaf(a, v.x, h.x));
        h.y = fmaf(s, u.y, fmaf(a, v.y, h.y));
        h.z = fmaf(s, u.z, fmaf(a, v.z, h.z));
        h.w = fmaf(s, u.w, fmaf(a, v.w, h.w));
        Hw[k >> 2] = h;
      }
    }
    dn = -(hg - rho * (s * hyg + hy * sg) + coef * s * sg);
  } else {
    dn = -hg;
  }
  __syncwarp();  // vec is rewritten by the next update
  return lane < D ? dn : 0.f;
}

// H = I (rows 0..D-1, columns up to D rounded to float4).
__device__ __forceinline__ void bfgs_reset(const WarpScratch& W, int D) {
  const int lane = threadIdx.x & 31;
  const int D4 = (D + 3) & ~3;
  if (lane < D) {
    float4* Hw = reinterpret_cast<float4*>(W.H + kHStride * lane);
    for (int k = 0; k < D4; k += 4)
      Hw[k >> 2] = make_float4(k == lane ? 1.f : 0.f, k + 1 == lane ? 1.f : 0.f, k + 2 == lane ? 1.f : 0.f,
                               k + 3 == lane ? 1.f : 0.f);
  }
}

// Write conf (7 + T floats) from lane layout: lanes 0..2 p, 3..6 q, 7 + k theta_k.
__device__ __forceinline__ void store_conf(float* out, const Conf& c, int T) {
  const int lane = threadIdx.x & 31;
  const float th = __shfl_sync(kFull, c.th, lane >= 7 ? lane - 1 : 0);
  if (lane < 7 + T) {
    float v;
    if (lane == 0) v = c.p.x;
    else if (lane == 1) v = c.p.y;
    else if (lane == 2) v = c.p.z;
    else if (lane == 3) v = c.q.w;
    else if (lane == 4) v = c.q.x;
    else if (lane == 5) v = c.q.y;
    else if (lane == 6) v = c.q.z;
    else v = th;
    out[lane] = v;
  }
}

// Make the conformation written by store_conf visible to the whole warp, then read it.
__device__ __forceinline__ Conf load_conf(const float* in, int T) {
  const int lane = threadIdx.x & 31;
  Conf c;
  c.p = make_float3(in[0], in[1], in[2]);
  c.q = Quat{in[3], in[4], in[5], in[6]};
  c.th = (lane >= 6 && lane < 6 + T) ? in[lane + 1] : 0.f;
  return c;
}

// Adaptive search space (Sec. 2, third modification; Fig. 3): a start position
// uniform in the box intersected with the union of balls of radius R around the
// predicted binding-site points, by rejection.  Attempt 0 is the box draw p0
// (block 0 of step 0), attempt a >= 1 takes words 0-2 of block 64 + a; a
// candidate is accepted when some point lies within R of it.  The candidate
// (one fused multiply-add per axis) and the squared distances ((dx dx + dy dy)
// + dz dz, no contraction) are FP32 with a fixed operation order, so every
// device and the oracle take the same decisions; the lanes share the points.
// After 64 rejected attempts the start is the first point.
__device__ __forceinline__ float3 site_start(const DevJob& J, const ChainStream& rs, float3 p0) {
  const int lane = threadIdx.x & 31;
  for (int a = 0; a < 64; ++a) {
    float3 c = p0;
    if (a > 0) {
      const uint4 b = rs.block(0, 64u + (uint32_t)a);
      c = make_float3(__fmaf_rn(J.box_size[0], ChainStream::to_uniform(b.x), J.box_lo[0]),
                      __fmaf_rn(J.box_size[1], ChainStream::to_uniform(b.y), J.box_lo[1]),
                      __fmaf_rn(J.box_size[2], ChainStream::to_uniform(b.z), J.box_lo[2]));
    }
    bool inside = false;
    for (int k = lane; k < J.n_sites; k += 32) {
      const float dx = __fsub_rn(c.x, __ldg(J.sites + 3 * k)), dy = __fsub_rn(c.y, __ldg(J.sites + 3 * k + 1)),
                  dz = __fsub_rn(c.z, __ldg(J.sites + 3 * k + 2));
      const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
      inside |= d2 <= J.site_r2;
    }
    if (__any_sync(kFull, inside)) return c;
  }
  return make_float3(__ldg(J.sites), __ldg(J.sites + 1), __ldg(J.sites + 2));
}

// Between two MC steps a chain is its current and best conformations, their
// energies, the evaluation count and the step number: what a time-sliced launch
// (dock_chains_kernel) keeps in global memory while another chain has the warp.
// Another SM may have written it: it is read and written past L1.
struct ChainRecord {
  float e_cur, e_best;
  uint32_t evals;
  uint32_t pad;
  // [7 + T]: component k of the current and of the best conformation
  __device__ __forceinline__ float2* conf() { return reinterpret_cast<float2*>(this + 1); }
};
static_assert(sizeof(ChainRecord) == slice_record_bytes(-7), "a record's size");
__device__ __forceinline__ ChainRecord* chain_record(const DevJob& J, int chain) {
  return reinterpret_cast<ChainRecord*>(reinterpret_cast<uint8_t*>(J.chain_coords) +
                                        (size_t)chain * J.record_bytes);
}
struct ChainSlice {
  ChainRecord* rec;  // null: the call runs the whole chain
  int* next_step;    // the step the chain stands at, 0 before its start
  int steps;         // MC steps of a slice (the start and its optimisation count as one)
};

// Chain and optimiser variables that wait in shared memory while a
// conformation is evaluated (read back through volatile loads, so that none of
// them holds a register during the evaluation).
struct alignas(16) ChainVars {
  // what each evaluation reads and writes, in groups of one 16-byte access
  int phase, trial;
  float alpha;
  uint32_t evals;
  float e, gd, e_opt_best;
  int it;
  int T, bb, max_iters, n_ramp;
  // once per local optimisation
  float e_cur, e_best;
  int step, chain;
  int stop;  // MC step at which this run of the chain ends (n_steps + 1: the chain's end)
  int pad;
  const DevJob* job;
  ChainRecord* rec;  // ChainSlice
  int* next_step;
};
// Volatile 16-byte accesses of a group (its first member).
__device__ __forceinline__ uint4 load_group(const volatile void* p) {
  uint4 v;
  asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"((uint32_t)__cvta_generic_to_shared(const_cast<const void*>(p))));
  return v;
}
__device__ __forceinline__ void store_group(volatile void* p, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.volatile.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(const_cast<void*>(p))),
               "r"(x), "r"(y), "r"(z), "r"(w));
}
static_assert(sizeof(ChainVars) <= 4 * kVarWords, "ChainVars must fit its words of the vec area");

// The drawn start of a chain.
__device__ __forceinline__ Conf draw_start(const DevJob& J, int T, int chain) {
  const int lane = threadIdx.x & 31;
  const ChainStream rs{J.seed_lo, J.seed_hi, (uint32_t)chain};
  Conf xt;
  // initial conformation: uniform word n of step 0 is word n % 4 of block n / 4
  const uint4 b0 = rs.block(0, 0), b1 = rs.block(0, 1);
  xt.p = make_float3(__fmaf_rn(J.box_size[0], ChainStream::to_uniform(b0.x), J.box_lo[0]),
                     __fmaf_rn(J.box_size[1], ChainStream::to_uniform(b0.y), J.box_lo[1]),
                     __fmaf_rn(J.box_size[2], ChainStream::to_uniform(b0.z), J.box_lo[2]));
  if (J.n_sites > 0) xt.p = site_start(J, rs, xt.p);
  const float u1 = ChainStream::to_uniform(b0.w), u2 = ChainStream::to_uniform(b1.x),
              u3 = ChainStream::to_uniform(b1.y);
  float s2, c2, s3, c3;
  sincosf(kTwoPiF * u2, &s2, &c2);
  sincosf(kTwoPiF * u3, &s3, &c3);
  const float a = sqrtf(1.f - u1), b = sqrtf(u1);
  xt.q = Quat{b * c3, a * s2, a * c2, b * s3};
  float th = 0.f;
  if (lane >= 6 && lane < 6 + T) {
    const uint4 bk = rs.block(0, (uint32_t)(lane >> 2));
    th = kPiF - kTwoPiF * ChainStream::to_uniform(pick(bk, lane & 3));
  }
  xt.th = th;
  return xt;
}

// The chain's current conformation (W.cur) mutated for MC step `step`: the start of
// its local optimisation.
__device__ __forceinline__ Conf mutated_conf(const DevJob& job, const LigView& L, const WarpScratch& W, int chain,
                                             uint32_t step, int T) {
  const int lane = threadIdx.x & 31;
  const ChainStream rs{job.seed_lo, job.seed_hi, (uint32_t)chain};
  const uint4 w0 = rs.block(step, 0);
  const int mode = (int)(((unsigned long long)(w0.x >> 8) * (unsigned long long)(2 + T)) >> 24);
  Conf xt = load_conf(W.cur, T);
  if (mode == 0) {
    const float3 b = unit_ball(rs, step);
    xt.p = xt.p + kMutationAmplitude * b;
  } else if (mode == 1) {
    const float3 b = unit_ball(rs, step);
    const float k = kMutationAmplitude * (1.f / L.h->gyration_radius);
    xt.q = qnormalize(qmul(quat_from_rotvec(k * b.x, k * b.y, k * b.z), xt.q));
  } else if (lane == 6 + (mode - 2)) {
    xt.th = kPiF - kTwoPiF * ChainStream::to_uniform(w0.z);
  }
  return xt;
}

// End of MC step `step`: Metropolis test of the optimised conformation W.x with
// energy eo, the chain's current and best conformations, and the trace (by one
// warp of the chain, `writer`).
__device__ __forceinline__ void metropolis_step(const DevJob& job, const WarpScratch& W, int chain, int step, int T,
                                                float eo, float& e_cur, float& e_best, bool writer) {
  const int lane = threadIdx.x & 31;
  const int nx = 7 + T;
  const ChainStream rs{job.seed_lo, job.seed_hi, (uint32_t)chain};
  const size_t trace_stride = (size_t)nx + 4;
  float* const trace =
      job.trace && writer ? job.trace + (size_t)chain * (job.n_steps + 1) * trace_stride : nullptr;
  if (step == 0) {
    e_cur = e_best = eo;
    if (lane < nx) {
      W.cur[lane] = W.x[lane];
      W.best[lane] = W.x[lane];
    }
    if (trace && !job.trace_starts) {
      if (lane < nx) trace[lane] = W.x[lane];
      if (lane == 0) {
        trace[nx + 0] = e_cur;
        trace[nx + 1] = e_cur;
        trace[nx + 2] = -1.f;
        trace[nx + 3] = 1.f;
      }
    }
  } else {
    const uint4 w0 = rs.block((uint32_t)step, 0);
    const int mode = (int)(((unsigned long long)(w0.x >> 8) * (unsigned long long)(2 + T)) >> 24);
    const float u = ChainStream::to_uniform(w0.y);
    const bool accept = (eo < e_cur) || (u < expf(-(eo - e_cur) / job.temperature));
    if (accept) {
      e_cur = eo;
      if (lane < nx) W.cur[lane] = W.x[lane];
      if (eo < e_best) {
        e_best = eo;
        if (lane < nx) W.best[lane] = W.x[lane];
      }
    }
    if (trace) {
      float* t = trace + (size_t)step * trace_stride;
      if (lane < nx) t[lane] = W.cur[lane];
      if (lane == 0) {
        t[nx + 0] = eo;
        t[nx + 1] = e_cur;
        t[nx + 2] = (float)mode;
        t[nx + 3] = accept ? 1.f : 0.f;
      }
    }
  }
}

// Row 0 of a trace that records starts: the drawn one, before any optimisation.
__device__ __forceinline__ void trace_start(const DevJob& J, int chain, const Conf& c, int T) {
  float* t = J.trace + (size_t)chain * (J.n_steps + 1) * ((size_t)7 + T + 4);
  store_conf(t, c, T);
  if ((threadIdx.x & 31) == 0) {
    t[7 + T + 0] = 0.f;
    t[7 + T + 1] = 0.f;
    t[7 + T + 2] = -2.f;
    t[7 + T + 3] = 0.f;
  }
}

// One Monte Carlo chain (Sec. 2: one of many short independent copies; Vina's
// mutation and Metropolis rules) with its local optimisations -- BFGS with
// Armijo backtracking (Vina's optimiser; Nocedal & Wright Alg. 6.1) or
// Barzilai-Borwein (the paper's second modification, Sec. 2 / ref. 37: BB1 step
// s.s / s.y, clamped, no line search, best iterate returned).
//
// The whole chain is one loop around a single score + gradient evaluation: a
// small state machine decides, from each evaluation, the next conformation to
// evaluate.  Only the conformation under evaluation stays in registers across
// an evaluation; the optimiser's vectors g and d, the chain's scalars and the
// iterate / current / best conformations wait in shared memory.
//
// With a record in `sl`, the call runs one slice from the step the chain stands
// at and leaves it in the record; without, the whole chain.
// REVIEW: read the ligand's view from the staged blob at each evaluation instead of
// holding it in registers (the 96-register kernels of mixed tiles and of one-channel maps
// spill otherwise).
template <int APL, int FMT, int IU = 2, bool REVIEW = false, bool FLAT = false>
__device__ void run_chain(const DevJob& J, const LigView& L, const WarpScratch& W, int chain, const ChainSlice& sl) {
  enum : int { kStart = 0, kTrial = 1, kBB = 2 };
  const int lane = threadIdx.x & 31;
  const MapView M = make_map_view(J);
  LaneLig<APL> R;
  load_lane_lig<APL>(L, R);
  volatile float* const Vg = W.vec + 3 * kHStride;  // g, component `lane` (lane < kHStride)
  volatile float* const Vd = W.vec + 4 * kHStride;  // search direction / step
  volatile ChainVars& V = *reinterpret_cast<volatile ChainVars*>(W.vec + 5 * kHStride);
  Conf xt;
  const int first = sl.rec ? __ldcg(sl.next_step) : 0;
  if (first > J.n_steps) return;
  bool mutate = first > 0;  // the next evaluation starts an MC step: mutate the current conformation
  {
    const int T = L.T;
    // every lane writes the same values
    V.phase = kStart;
    V.it = V.trial = 0;
    V.e = V.gd = V.e_opt_best = 0.f;
    V.alpha = 1.f;
    V.T = T;
    V.bb = J.optimizer == DSDP_OPT_BB;
    V.max_iters = J.n_opt_iters;
    V.n_ramp = ramp_steps(L);
    V.chain = chain;
    V.job = &J;
    V.step = first;
    V.stop = sl.rec ? min(first + sl.steps, J.n_steps + 1) : J.n_steps + 1;
    V.rec = sl.rec;
    V.next_step = sl.next_step;
    if (lane < kHStride) Vg[lane] = Vd[lane] = 0.f;
    if (mutate) {
      if (lane < 7 + T) {
        const float2 c = __ldcg(sl.rec->conf() + lane);
        W.cur[lane] = c.x;
        W.best[lane] = c.y;
      }
      V.e_cur = __ldcg(&sl.rec->e_cur);
      V.e_best = __ldcg(&sl.rec->e_best);
      V.evals = __ldcg(&sl.rec->evals);
    } else {
      V.e_cur = V.e_best = 0.f;
      V.evals = 0;
    }
  }
  if (!mutate) {
    const int T = L.T;
    xt = draw_start(J, T, chain);
    if (J.trace && J.trace_starts) trace_start(J, chain, xt, T);
  }
  __syncwarp();
  for (;;) {
    if (__builtin_expect(mutate, 0)) {  // once per MC step: kept out of the evaluations' way
      xt = mutated_conf(*V.job, L, W, V.chain, (uint32_t)V.step, V.T);
      mutate = false;
    }
    bool done = false;  // the local optimisation ends with this evaluation
    Placed<APL> P;
    const LigView Lv = REVIEW ? view_blob(reinterpret_cast<const uint8_t*>(L.h)) : L;
    place_atoms<APL>(Lv, xt, P);
    int phase = V.phase;
    if (phase == kTrial) {
      // BFGS: Armijo test of the trial point x + alpha d on its energy alone; its
      // gradient is evaluated when it is accepted (27 % of first trials, 23 % of all)
      const float en = energy_placed<APL, FMT, IU>(M, Lv, V.n_ramp, P);
      const uint4 v0 = load_group(&V.phase), v1 = load_group(&V.e);
      const float e = __uint_as_float(v1.x), gd = __uint_as_float(v1.y);
      float alpha = __uint_as_float(v0.z);
      if (!(en <= e + kArmijoC1 * alpha * gd)) {
        const int trial = (int)v0.y + 1;
        alpha *= kShrink;
        __syncwarp();
        if (lane == 0) store_group(&V.phase, v0.x, (uint32_t)trial, __float_as_uint(alpha), v0.w + 1u);
        if (trial < kMaxTrials) {
          const float dir = lane < kHStride ? Vd[lane] : 0.f;
          const int T = Lv.T;
          xt = apply_step(load_conf(W.x, T), alpha * dir, T);
          __syncwarp();
          continue;
        }
        done = true;  // no acceptable step: the optimisation ends at the current iterate
      }
    }
    if (!done) {
      float gn;
      const float en = score_placed<APL, FMT, IU, FLAT>(M, Lv, R, V.n_ramp, W, xt, P, gn, DSDP_TERM_ALL);
      const uint4 v0 = load_group(&V.phase), v1 = load_group(&V.e), v2 = load_group(&V.T);
      const int T = (int)v2.x, D = 6 + T, max_iters = (int)v2.z;
      const bool bb = v2.y != 0;
      phase = (int)v0.x;
      int it = (int)v1.w;
      float e_opt_best = __uint_as_float(v1.z);
      float e = __uint_as_float(v1.x), gd = __uint_as_float(v1.y), alpha = __uint_as_float(v0.z);
      float g = lane < kHStride ? Vg[lane] : 0.f, dir = lane < kHStride ? Vd[lane] : 0.f;
      if (phase == kStart) {  // first evaluation of a local optimisation
        e = en;
        g = gn;
        store_conf(W.x, xt, T);
        if (max_iters == 0) {
          done = true;
        } else if (!bb) {
          bfgs_reset(W, D);
          dir = -g;  // H0 = I
          gd = -warp_sum(g * g);
          it = 0;
          alpha = 1.f;
          xt = apply_step(xt, dir, T);
          phase = kTrial;
        } else {
          e_opt_best = e;
          alpha = kBBAlpha0;
          it = 0;
          dir = -alpha * g;
          xt = apply_step(xt, dir, T);
          phase = kBB;
        }
      } else if (phase == kTrial) {  // BFGS: an accepted trial point
        const float s = alpha * dir, y = gn - g;
        g = gn;
        e = en;
        store_conf(W.x, xt, T);
        if (++it == max_iters) {
          done = true;
        } else {
          dir = bfgs_update(W, D, s, y, gn, dir);
          gd = warp_sum(g * dir);  // computed directly: the sufficient-decrease test must see the true slope
          alpha = 1.f;
          xt = apply_step(xt, dir, T);
        }
      } else {  // BB: x_{k+1} = x_k + s_k evaluated; next step length from s.s / s.y
        const float sy = warp_sum(dir * (gn - g));
        const float ss = warp_sum(dir * dir);
        alpha = sy > 0.f ? fminf(fmaxf(ss / sy, kBBAlphaMin), kBBAlphaMax) : kBBAlphaMax;
        g = gn;
        if (en < e_opt_best) {
          e_opt_best = en;
          store_conf(W.x, xt, T);
        }
        if (++it == max_iters) {
          done = true;
        } else {
          dir = -alpha * g;
          xt = apply_step(xt, dir, T);
        }
      }
      __syncwarp();  // the groups are read by every lane
      if (lane == 0) {
        store_group(&V.phase, (uint32_t)phase, 0u, __float_as_uint(alpha), v0.w + 1u);  // the next trial is the first
        store_group(&V.e, __float_as_uint(e), __float_as_uint(gd), __float_as_uint(e_opt_best), (uint32_t)it);
      }
      if (lane < kHStride) {
        Vg[lane] = g;
        Vd[lane] = dir;
      }
      __syncwarp();
    }
    if (__builtin_expect(done, 0)) {
      // ---- local optimisation finished: its result is W.x with energy eo
      __syncwarp();
      const int T = V.T, nx = 7 + T;
      const uint32_t evals = V.evals;
      const float eo = (V.bb && V.max_iters > 0) ? V.e_opt_best : V.e;
      // (the job record is read again here rather than held across the evaluations)
      const DevJob& job = *V.job;
      const int chain_id = V.chain;
      int step = V.step;
      float e_cur = V.e_cur, e_best = V.e_best;
      __syncwarp();
      metropolis_step(job, W, chain_id, step, T, eo, e_cur, e_best, true);
      __syncwarp();
      if (++step > job.n_steps) {
        if (lane < nx) job.chain_best_conf[(size_t)chain_id * nx + lane] = W.best[lane];
        if (lane == 0) {
          job.chain_best_e[chain_id] = e_best;
          job.chain_evals[chain_id] = evals;
          if (V.rec) __stcg(V.next_step, step);  // a further slice finds nothing left
        }
        __syncwarp();
        return;
      }
      if (step == V.stop) {  // end of this slice: the chain waits in its record
        ChainRecord* const rec = V.rec;
        if (lane < nx) __stcg(rec->conf() + lane, make_float2(W.cur[lane], W.best[lane]));
        if (lane == 0) {
          __stcg(&rec->e_cur, e_cur);
          __stcg(&rec->e_best, e_best);
          __stcg(&rec->evals, evals);
          __stcg(V.next_step, step);
        }
        __syncwarp();
        return;
      }
      mutate = true;
      V.phase = kStart;
      V.step = step;
      V.e_cur = e_cur;
      V.e_best = e_best;
      __syncwarp();
    }
  }
}

// What a team's warps tell each other of one round: each warp's trial point and its
// score and gradient.  Two of them, used in turn: a warp writes a round's only after
// the barrier that all pass when they have read the one before the last.
struct TeamSlot {
  float e;
  float x[kConfFloats];
  float g[kHStride];
};

// run_chain's BFGS chain by a team of the CTA's warps, for launches whose chains leave
// most of the GPU idle.  A line search halves its step until the energy falls
// enough: three of four trial points are rejected, and run_chain evaluates them one
// after the other.  Here warp w evaluates trial t0 + w, all at once, and the first
// acceptable one in the search's order is taken: the decisions, and so the chain,
// are run_chain's bit for bit.  Everything between evaluations every warp does for
// itself, in scratch of its own; one barrier per round.  first > 0: from the chain's
// record, which stands at that MC step.
//
// Bound: latency (a round is one evaluation and one update, 3.2 us; energies first and
// the winner's gradient after a second barrier: 8 % slower alone and no faster with
// eight launches at once).  One typical-4k system (384 chains, 2.6 evaluations a round
// with teams of 4) takes 5.9 - 6.2 ms of chain stage against 10.7 - 11.2 with one warp a
// chain, one plain-2k system (64 chains, teams of 8) 5.8 - 6.2 against 13.1 - 14.1.
template <int APL, int FMT>
__device__ void run_team(const DevJob& J, const LigView& L, const WarpScratch& W, TeamSlot* ex, int chain, int first) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, team = blockDim.x >> 5;
  const MapView M = make_map_view(J);
  LaneLig<APL> R;
  load_lane_lig<APL>(L, R);
  const int n_ramp = ramp_steps(L);
  const int T = L.T, nx = 7 + T, D = 6 + T, max_iters = J.n_opt_iters;
  Conf xt;
  float e_cur = 0.f, e_best = 0.f;
  uint32_t evals = 0;
  if (first == 0) {
    xt = draw_start(J, T, chain);
    if (J.trace && J.trace_starts && warp == 0) trace_start(J, chain, xt, T);
  } else {
    ChainRecord* const rec = chain_record(J, chain);
    if (lane < nx) {
      const float2 c = __ldcg(rec->conf() + lane);
      W.cur[lane] = c.x;
      W.best[lane] = c.y;
    }
    e_cur = __ldcg(&rec->e_cur);
    e_best = __ldcg(&rec->e_best);
    evals = __ldcg(&rec->evals);
    __syncwarp();
  }
  int round = 0;
  for (int step = first;; ++step) {
    if (step > 0) xt = mutated_conf(J, L, W, chain, (uint32_t)step, T);
    // ---- the start, evaluated by warp 0
    float e = 0.f, g = 0.f;
    {
      TeamSlot* const s = ex + (round++ & 1) * team;
      if (warp == 0) {
        Placed<APL> P;
        place_atoms<APL>(L, xt, P);
        float gn;
        const float en = score_placed<APL, FMT, 2, true>(M, L, R, n_ramp, W, xt, P, gn, DSDP_TERM_ALL);
        if (lane == 0) s->e = en;
        if (lane < kHStride) s->g[lane] = gn;
      }
      store_conf(W.x, xt, T);
      __syncthreads();
      e = s->e;
      if (lane < kHStride) g = s->g[lane];
      ++evals;
    }
    if (max_iters > 0) {
      bfgs_reset(W, D);
      float dir = -g;  // H0 = I
      float gd = -warp_sum(g * g);
      int it = 0, t0 = 0;
      for (;;) {
        TeamSlot* const slots = ex + (round++ & 1) * team;
        const int trial = t0 + warp;
        const float alpha = __int_as_float((127 - trial) << 23);  // kShrink^trial
        if (trial < kMaxTrials) {
          xt = apply_step(load_conf(W.x, T), alpha * dir, T);
          Placed<APL> P;
          place_atoms<APL>(L, xt, P);
          float gn;
          const float en = score_placed<APL, FMT, 2, true>(M, L, R, n_ramp, W, xt, P, gn, DSDP_TERM_ALL);
          TeamSlot* const s = slots + warp;
          store_conf(s->x, xt, T);
          if (lane == 0) s->e = en;
          if (lane < kHStride) s->g[lane] = gn;
        }
        __syncthreads();
        const int tried = min(team, kMaxTrials - t0);
        const float e_l = lane < tried ? slots[lane].e : 0.f, a_l = __int_as_float((127 - t0 - lane) << 23);
        const unsigned ok = __ballot_sync(kFull, lane < tried && e_l <= e + kArmijoC1 * a_l * gd);
        if (!ok) {
          evals += tried;
          t0 += team;
          if (t0 >= kMaxTrials) break;  // no acceptable step: the optimisation ends at the current iterate
          continue;
        }
        const int k = __ffs(ok) - 1;
        evals += k + 1;
        const TeamSlot& won = slots[k];
        const float ak = __int_as_float((127 - t0 - k) << 23);
        const float gn = lane < kHStride ? won.g[lane] : 0.f;
        const float s = ak * dir, y = gn - g;
        g = gn;
        e = won.e;
        if (lane < nx) W.x[lane] = won.x[lane];
        __syncwarp();
        if (++it == max_iters) break;
        dir = bfgs_update(W, D, s, y, gn, dir);
        gd = warp_sum(g * dir);
        t0 = 0;
      }
    }
    // ---- local optimisation finished: its result is W.x with energy e
    __syncwarp();
    metropolis_step(J, W, chain, step, T, e, e_cur, e_best, warp == 0);
    __syncwarp();
    if (step == J.n_steps) break;
  }
  if (warp == 0) {
    if (lane < nx) J.chain_best_conf[(size_t)chain * nx + lane] = W.best[lane];
    if (lane == 0) {
      J.chain_best_e[chain] = e_best;
      J.chain_evals[chain] = evals;
    }
  }
}

}  // namespace dsdp
