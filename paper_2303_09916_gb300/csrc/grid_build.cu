// Receptor grid maps (Sec. 2 first modification; Appendix Eq. 1 and Eq. 4)
// and the gather microbenchmark that bounds the score path.
//
// A CTA owns a brick of 8 x 8 x 4 SB vertices.  It streams the receptor atoms in
// index order and keeps those within the cutoff of the brick's bounding box
// (ballot compaction into shared memory, order preserved, so the sums are
// deterministic).  A warp owns SB blocks of 4 x 4 x 2 vertices, one per lane; it tests
// the kept atoms 32 at a time against its own box and sums, for every atom within
// the cutoff of the box, the pair score and its gradient for all 8 ligand types.
// The 8 types share 4 atomic radii: the gauss / repulsion terms are summed once
// per radius (packed FP32x2, two radii per operation), and the hydrophobic and
// H-bond terms, which only some receptor atoms carry and only at short range, in
// five sums of their own; each type's map is its radius sum plus its own term at
// the end.
//
// Bound: the FMA pipe (a packed FP32x2 instruction holds it for two cycles).  So an
// atom takes the cheapest of three forms that its least distance to the warp's box
// allows, chosen for the whole warp (no divergence):
//   far  (d >= 2.4 for every radius): gauss2 alone -- there gauss1 is below 1e-9 of
//        gauss2 and its slope below 1e-10 kcal/mol/A (half the atoms in range);
//   mid  (d >= 0): no repulsion, which is exactly 0;
//   near: all terms.
// The slopes' sums run in units of gauss2's, which multiplies once at the end.
// The scan over all receptor atoms is the rest: two blocks a warp (SB = 2) halve it
// and are taken from four waves of CTAs on; below, the smaller bricks fill the SMs
// better.
#include "launch.h"

namespace dsdp {
namespace {

constexpr int kBX = 8, kBY = 8, kBZ = 4, kThreads = kBX * kBY * kBZ;
constexpr int kChunk = 1536;       // kept atoms staged at once
constexpr int kTests = 2;          // atoms a thread tests per barrier
constexpr float kSlack = 0.01f;   // what the boxes' tests allow for rounding, in Angstrom (box_slack)
constexpr float kFarMid = 2.40f + kSlack;  // surface distance from which gauss1 is left out

// 2^(-u^2) = exp(-b^2) for u = kRootLog2E b; b = (d - 3) / 2
constexpr double kRootLog2E = 1.2011224087864498;  // sqrt(1 / ln 2)
constexpr float kU = (float)(0.5 * kRootLog2E);    // u = kU d - 3 kU
// unit of the slopes' sums: -kWGauss2 / kRootLog2E (per u exp(-b^2))
constexpr float kSlopeUnit = -kWGauss2 / (float)kRootLog2E;
constexpr float kS1 = -8.f * kWGauss1 / kSlopeUnit;  // gauss1: -8 d exp(-4 d^2)
constexpr float kS3 = 2.f * kWRepulsion / kSlopeUnit;  // repulsion: 2 m

// hydrophobic term of surface distance d (1 below 0.5, linear to 0 at 1.5),
// added to e and de/dd
__device__ __forceinline__ void hydrophobic(float d, float& e, float& de) {
  if (d < 0.5f) {
    e += kWHydrophobic;
  } else if (d < 1.5f) {
    e += kWHydrophobic * (1.5f - d);
    de -= kWHydrophobic;
  }
}
// H-bond term (1 below -0.7, linear to 0 at 0)
__device__ __forceinline__ void hbond(float d, float& e, float& de) {
  if (d < -0.7f) {
    e += kWHBond;
  } else if (d < 0.f) {
    e += kWHBond * (-d * (1.0f / 0.7f));
    de -= kWHBond * (1.0f / 0.7f);
  }
}

// a (e, de/dd) pair term projected on the unit vector u, added to (E, G)
__device__ __forceinline__ void add_term(float4& acc, float e, float de, float ux, float uy, float uz) {
  acc.x += e;
  acc.y = fmaf(de, ux, acc.y);
  acc.z = fmaf(de, uy, acc.z);
  acc.w = fmaf(de, uz, acc.w);
}

template <int FMT>
__device__ __forceinline__ void store_node(void* maps, size_t idx, float e, float gx, float gy, float gz) {
  if (FMT == 0) {
    reinterpret_cast<float4*>(maps)[idx] = make_float4(e, gx, gy, gz);
  } else if (FMT == 1) {
    __nv_bfloat162 a = __floats2bfloat162_rn(e, gx), b = __floats2bfloat162_rn(gy, gz);
    uint2 raw;
    raw.x = *reinterpret_cast<uint32_t*>(&a);
    raw.y = *reinterpret_cast<uint32_t*>(&b);
    reinterpret_cast<uint2*>(maps)[idx] = raw;
  } else if (FMT == 2) {
    __half2 a = __floats2half2_rn(e, gx), b = __floats2half2_rn(gy, gz);
    uint2 raw;
    raw.x = *reinterpret_cast<uint32_t*>(&a);
    raw.y = *reinterpret_cast<uint32_t*>(&b);
    reinterpret_cast<uint2*>(maps)[idx] = raw;
  } else if (FMT == 3) {
    reinterpret_cast<float*>(maps)[idx] = e;
  } else if (FMT == 4) {
    reinterpret_cast<unsigned short*>(maps)[idx] = __bfloat16_as_ushort(__float2bfloat16_rn(e));
  } else {
    reinterpret_cast<unsigned short*>(maps)[idx] = __half_as_ushort(__float2half_rn(e));
  }
}

// Sums of one vertex: gauss / repulsion per radius, packed (1.9, 1.8) and (1.7,
// 2.0): energy and gradient (in the slopes' unit); hydrophobic term of C_H; H-bond terms of
// N_D (with receptor acceptors), N_A and O_A (with receptor donors), O_DA (with
// donors or acceptors): (e, gx, gy, gz).
struct VertexSums {
  float2 Ea, Eb, Xa, Xb, Ya, Yb, Za, Zb;
  float4 Hch, Hnd, Hna, Hoa, Hoda;
};

enum { kNear, kMid, kFar };

// u = kU (r - R_j - s - 3) is kU (r - 8) plus this, per receptor type and radius s.  The
// distance from the cutoff, not r: the offsets are below 1 then, and their rounding,
// which is the same for every atom of a type and adds up in the sums, is an eighth
// (3e-8 at most; with r it is up to 2.7e-7, and the median energy error of the maps of
// radius 1.8 at 4,000 atoms 4.0e-8 against 3.6e-8).
struct Offsets {
  float2 a[9], b[9];  // radii (1.9, 1.8) and (1.7, 2.0)
};
constexpr Offsets make_offsets() {
  constexpr double R[9] = {1.9, 1.9, 1.8, 1.8, 1.8, 1.7, 1.7, 2.0, 1.8};
  Offsets o{};
  for (int t = 0; t < 9; ++t) {
    o.a[t].x = (float)(kU * (3.1 - R[t])), o.a[t].y = (float)(kU * (3.2 - R[t]));
    o.b[t].x = (float)(kU * (3.3 - R[t])), o.b[t].y = (float)(kU * (3.0 - R[t]));
  }
  return o;
}
__constant__ Offsets c_offset = make_offsets();

// gauss2 at u, and with KIND != kFar gauss1 (and repulsion) at the surface distance d, of two radii
template <int KIND>
__device__ __forceinline__ void add_radii(float2 d, float2 u, float2 ux, float2 uy, float2 uz, float2& E, float2& X,
                                          float2& Y, float2& Z) {
  const float2 uu = __fmul2_rn(u, u);
  const float2 g2 = make_float2(ex2_approx(-uu.x), ex2_approx(-uu.y));
  float2 p = __fmul2_rn(u, g2);
  E = __ffma2_rn(g2, splat2(kWGauss2), E);
  if (KIND != kFar) {
    const float2 dd = __fmul2_rn(d, __fmul2_rn(d, splat2(-4.f * kLog2E)));
    const float2 g1 = make_float2(ex2_approx(dd.x), ex2_approx(dd.y));
    E = __ffma2_rn(g1, splat2(kWGauss1), E);
    p = __ffma2_rn(__fmul2_rn(g1, d), splat2(kS1), p);
  }
  if (KIND == kNear) {
    const float2 m = make_float2(fminf(d.x, 0.f), fminf(d.y, 0.f));
    E = __ffma2_rn(__fmul2_rn(m, m), splat2(kWRepulsion), E);
    p = __ffma2_rn(m, splat2(kS3), p);
  }
  X = __ffma2_rn(p, ux, X);
  Y = __ffma2_rn(p, uy, Y);
  Z = __ffma2_rn(p, uz, Z);
}

// One receptor atom at the vertex (mx, my, mz).  The distance, the cutoff and the
// surface distances of the hydrophobic and H-bond branches are one fixed sequence
// of FP32 operations in every form; beyond the cutoff the distance is set so far
// out that every term is exactly 0.
template <int KIND>
__device__ __forceinline__ void add_atom(VertexSums& S, const float4 a, float mx, float my, float mz) {
  const float dx = mx - a.x, dy = my - a.y, dz = mz - a.z;
  const float r2 = dx * dx + dy * dy + dz * dz;
  const int tj = __float_as_int(a.w);
  const float Rj = c_xs_radius[tj];
  // a vertex on an atom (r = 0) takes no gradient from it: ir is finite there and d* = 0
  const float ir = rsqrt_ftz(fmaxf(r2, 1e-30f));
  const float r = r2 < kCutoff * kCutoff ? r2 * ir : 2.f * kFarD;
  const float2 ux = splat2(dx * ir), uy = splat2(dy * ir), uz = splat2(dz * ir);
  const float2 rc = splat2(r2 < kCutoff * kCutoff ? __fmaf_rn(r2, ir, -kCutoff) : 2.f * kFarD), ku = splat2(kU);
  const float2 ua = __ffma2_rn(rc, ku, c_offset.a[tj]), ub = __ffma2_rn(rc, ku, c_offset.b[tj]);
  if (KIND == kFar) {
    const float2 none = make_float2(0.f, 0.f);
    add_radii<kFar>(none, ua, ux, uy, uz, S.Ea, S.Xa, S.Ya, S.Za);
    add_radii<kFar>(none, ub, ux, uy, uz, S.Eb, S.Xb, S.Yb, S.Zb);
    return;
  }
  const float2 sa = make_float2(r - (1.9f + Rj), r - (1.8f + Rj));
  const float2 sb = make_float2(r - (1.7f + Rj), r - (2.0f + Rj));
  add_radii<KIND>(sa, ua, ux, uy, uz, S.Ea, S.Xa, S.Ya, S.Za);
  add_radii<KIND>(sb, ub, ux, uy, uz, S.Eb, S.Xb, S.Yb, S.Zb);
  const int bj = c_xs_bits[tj];  // the same for every lane: the branches below do not diverge on it
  if ((bj & 1) && sa.x < 1.5f) {  // hydrophobic receptor atom: C_H (radius 1.9)
    float e = 0.f, de = 0.f;
    hydrophobic(sa.x, e, de);
    add_term(S.Hch, e, de, ux.x, uy.x, uz.x);
  }
  if (KIND == kNear && (bj & 6) && sa.y < 0.f) {  // donor and/or acceptor within H-bond range (d of radius 1.8 < 0)
    if (bj & 4) {  // receptor acceptor: N_D (1.8)
      float e = 0.f, de = 0.f;
      hbond(sa.y, e, de);
      add_term(S.Hnd, e, de, ux.x, uy.x, uz.x);
    }
    if (bj & 2) {  // receptor donor: N_A (1.8), O_A (1.7)
      float e = 0.f, de = 0.f;
      hbond(sa.y, e, de);
      add_term(S.Hna, e, de, ux.x, uy.x, uz.x);
      e = de = 0.f;
      hbond(sb.x, e, de);
      add_term(S.Hoa, e, de, ux.x, uy.x, uz.x);
    }
    float e = 0.f, de = 0.f;  // O_DA (1.7) with either
    hbond(sb.x, e, de);
    add_term(S.Hoda, e, de, ux.x, uy.x, uz.x);
  }
}

// squared distance from a point to the box of half sides (ex, ey, ez) around (cx, cy, cz)
__device__ __forceinline__ float box_dist2(float4 a, float cx, float cy, float cz, float ex, float ey, float ez) {
  const float dx = fmaxf(fabsf(a.x - cx) - ex, 0.f), dy = fmaxf(fabsf(a.y - cy) - ey, 0.f),
              dz = fmaxf(fabsf(a.z - cz) - ez, 0.f);
  return dx * dx + dy * dy + dz * dz;
}

template <int FMT, int SB>
__global__ void __launch_bounds__(kThreads, 3) grid_build_kernel(int n_rec, const float* __restrict__ xyz,
                                                                 const uint8_t* __restrict__ type, int nx, int ny,
                                                                 int nz, float ox, float oy, float oz, float h,
                                                                 float reach2, float more_slack,
                                                                 void* __restrict__ maps) {
  constexpr int kWarps = kThreads / 32;
  __shared__ float4 s_atom[kChunk];
  __shared__ int s_count[kTests * kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bx0 = blockIdx.x * kBX, by0 = blockIdx.y * kBY, bz0 = blockIdx.z * kBZ * SB;
  const float bcx = ox + h * ((float)bx0 + 0.5f * (kBX - 1)), bcy = oy + h * ((float)by0 + 0.5f * (kBY - 1)),
              bcz = oz + h * ((float)bz0 + 0.5f * (kBZ * SB - 1));
  int count = 0;
  bool staged = false;  // the kept atoms of the whole receptor are in s_atom
#pragma unroll 1
  for (int sb = 0; sb < SB; ++sb) {
    // the warp's 4 x 4 x 2 vertices
    const int wx0 = bx0 + 4 * (warp & 1), wy0 = by0 + 4 * ((warp >> 1) & 1), wz0 = bz0 + 2 * (warp >> 2) + kBZ * sb;
    const int ix = wx0 + (lane & 3), iy = wy0 + ((lane >> 2) & 3), iz = wz0 + (lane >> 4);
    const bool warp_active = wx0 < nx && wy0 < ny && wz0 < nz;
    const float mx = ox + h * (float)ix, my = oy + h * (float)iy, mz = oz + h * (float)iz;
    const float wcx = ox + h * ((float)wx0 + 1.5f), wcy = oy + h * ((float)wy0 + 1.5f),
                wcz = oz + h * ((float)wz0 + 0.5f);
    VertexSums S;
    S.Ea = S.Eb = S.Xa = S.Xb = S.Ya = S.Yb = S.Za = S.Zb = make_float2(0.f, 0.f);
    S.Hch = S.Hnd = S.Hna = S.Hoa = S.Hoda = make_float4(0.f, 0.f, 0.f, 0.f);
    int base = staged ? n_rec : 0;
    do {
      const bool first = base == 0;
      if (!staged) count = 0;
      while (base < n_rec && count <= kChunk - kTests * kThreads) {
        float4 a[kTests];
        unsigned bal[kTests];
#pragma unroll
        for (int k = 0; k < kTests; ++k) {
          const int j = base + k * kThreads + tid;
          bool keep = false;
          a[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (j < n_rec) {
            a[k].x = __ldg(xyz + 3 * j);
            a[k].y = __ldg(xyz + 3 * j + 1);
            a[k].z = __ldg(xyz + 3 * j + 2);
            a[k].w = __int_as_float(min((int)__ldg(type + j), 8));
            // an atom that is not at a finite place is in no vertex's range
            keep = box_dist2(a[k], bcx, bcy, bcz, 0.5f * (kBX - 1) * h, 0.5f * (kBY - 1) * h,
                             0.5f * (kBZ * SB - 1) * h) < reach2 && isfinite(a[k].x + a[k].y + a[k].z);
          }
          bal[k] = __ballot_sync(kFull, keep);
          if (lane == 0) s_count[k * kWarps + warp] = __popc(bal[k]);
        }
        __syncthreads();
        int total = 0;
#pragma unroll
        for (int k = 0; k < kTests; ++k) {
          int off = count + total;
#pragma unroll
          for (int w = 0; w < kWarps; ++w) {
            const int c = s_count[k * kWarps + w];
            if (w < warp) off += c;
            total += c;
          }
          if ((bal[k] >> lane) & 1) s_atom[off + __popc(bal[k] & ((1u << lane) - 1u))] = a[k];
        }
        count += total;
        base += kTests * kThreads;
        __syncthreads();
      }
      if (first && base >= n_rec) staged = true;  // the same in every thread
      if (warp_active) {
        for (int k0 = 0; k0 < count; k0 += 32) {
          const bool have = k0 + lane < count;
          const float4 a = have ? s_atom[k0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
          const float d2 = have ? box_dist2(a, wcx, wcy, wcz, 1.5f * h, 1.5f * h, 0.5f * h) : reach2;
          const float far = 2.0f + kFarMid + c_xs_radius[__float_as_int(a.w)] + more_slack,
                      mid = far - kFarMid + kSlack;
          unsigned m_far = __ballot_sync(kFull, d2 < reach2 && d2 >= far * far);
          unsigned m_mid = __ballot_sync(kFull, d2 < far * far && d2 >= mid * mid);
          unsigned m_near = __ballot_sync(kFull, d2 < mid * mid);
          for (; m_far; m_far &= m_far - 1) add_atom<kFar>(S, s_atom[k0 + __ffs(m_far) - 1], mx, my, mz);
          for (; m_mid; m_mid &= m_mid - 1) add_atom<kMid>(S, s_atom[k0 + __ffs(m_mid) - 1], mx, my, mz);
          for (; m_near; m_near &= m_near - 1) add_atom<kNear>(S, s_atom[k0 + __ffs(m_near) - 1], mx, my, mz);
        }
      }
      if (!staged) __syncthreads();  // the next atoms replace these
    } while (base < n_rec);
    if (ix >= nx || iy >= ny || iz >= nz) continue;
    const size_t nxyz = (size_t)nx * ny * nz;
    const size_t v = ((size_t)iz * ny + iy) * nx + ix;
    auto store = [&](int t, float e, float x, float y, float z, const float4& H) {
      store_node<FMT>(maps, t * nxyz + v, e + H.x, fmaf(x, kSlopeUnit, H.y), fmaf(y, kSlopeUnit, H.z),
                      fmaf(z, kSlopeUnit, H.w));
    };
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    store(0, S.Ea.x, S.Xa.x, S.Ya.x, S.Za.x, S.Hch);   // C_H
    store(1, S.Ea.x, S.Xa.x, S.Ya.x, S.Za.x, none);    // C_P
    store(2, S.Ea.y, S.Xa.y, S.Ya.y, S.Za.y, none);    // N_P
    store(3, S.Ea.y, S.Xa.y, S.Ya.y, S.Za.y, S.Hnd);   // N_D
    store(4, S.Ea.y, S.Xa.y, S.Ya.y, S.Za.y, S.Hna);   // N_A
    store(5, S.Eb.x, S.Xb.x, S.Yb.x, S.Zb.x, S.Hoa);   // O_A
    store(6, S.Eb.x, S.Xb.x, S.Yb.x, S.Zb.x, S.Hoda);  // O_DA
    store(7, S.Eb.y, S.Xb.y, S.Yb.y, S.Zb.y, none);    // S_P
  }
}

// 32-bit mixing hash (multiply-xorshift; the finaliser of MurmurHash3) for the
// microbenchmark's pseudo-random sample points.
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x ^= x >> 16;
  x *= 0x85ebca6bu;
  x ^= x >> 13;
  x *= 0xc2b2ae35u;
  x ^= x >> 16;
  return x;
}

// Each thread samples `repeats` points: the first is its input point, each later
// one an independent pseudo-random position in the grid (hash of the point
// index and the repeat) with a pseudo-random map type, so that consecutive
// samples share no cell and the corner reads are the random 8-corner gathers of
// the scoring path, with none of its arithmetic.
template <int FMT>
__global__ void __launch_bounds__(256) gather_bench_kernel(MapView M, const float* __restrict__ pts,
                                                           const uint8_t* __restrict__ types, int n, int repeats,
                                                           float* __restrict__ out) {
  const int stride = gridDim.x * blockDim.x;
  const float ex = (M.nx - 1) * M.h, ey = (M.ny - 1) * M.h, ez = (M.nz - 1) * M.h;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    float3 p = make_float3(pts[3 * i], pts[3 * i + 1], pts[3 * i + 2]);
    int t = types[i];
    float acc = 0.f;
    for (int r = 0; r < repeats; ++r) {
      float3 g;
      const float e = sample_map<FMT>(M, t, p, g);
      acc += e + g.x + g.y + g.z;
      const uint32_t h0 = mix32((uint32_t)i * 0x9E3779B9u + (uint32_t)r + 1u);
      const uint32_t h1 = mix32(h0 ^ 0x68E31DA4u), h2 = mix32(h1 ^ 0xB5297A4Du);
      p = make_float3(M.ox + ex * ((h0 >> 8) * (1.f / 16777216.f)), M.oy + ey * ((h1 >> 8) * (1.f / 16777216.f)),
                      M.oz + ez * ((h2 >> 8) * (1.f / 16777216.f)));
      t = (int)(h2 & 7u);
    }
    out[i] = acc;
  }
}

// What the tests of an atom against a brick's or a warp's box allow for rounding: at m
// Angstrom from the origin a vertex and a box's centre are each at most 2^-24 m off
// (twice that unfused) along an axis, 4.2e-7 m of distance for both.
float box_slack(int nx, int ny, int nz, float ox, float oy, float oz, float h) {
  const int n[3] = {nx, ny, nz};
  const float o[3] = {ox, oy, oz};
  double m = 0.0;
  for (int a = 0; a < 3; ++a)
    m = fmax(m, fmax(fabs((double)o[a]), fabs((double)o[a] + (double)h * (n[a] + 2 * kBX))));
  return fmaxf(kSlack, (float)(5e-7 * m));
}

template <int FMT>
cudaError_t launch_grid(const dsdp_receptor* rec, int nx, int ny, int nz, float ox, float oy, float oz, float h,
                        void* maps, cudaStream_t st) {
  const int sms = device_sms();
  dim3 grid((nx + kBX - 1) / kBX, (ny + kBY - 1) / kBY, (nz + 2 * kBZ - 1) / (2 * kBZ));
  const bool two = (long long)grid.x * grid.y * grid.z >= 4ll * 3 * sms;  // 3 CTAs per SM
  if (!two) grid.z = (nz + kBZ - 1) / kBZ;
  auto k = two ? grid_build_kernel<FMT, 2> : grid_build_kernel<FMT, 1>;
  const float slack = box_slack(nx, ny, nz, ox, oy, oz, h);
  k<<<grid, kThreads, 0, st>>>(rec->n, rec->xyz, rec->xs_type, nx, ny, nz, ox, oy, oz, h,
                               (kCutoff + slack) * (kCutoff + slack), slack - kSlack, maps);
  return cudaGetLastError();
}

template <int FMT>
cudaError_t launch_gather(const MapView& M, const float* pts, const uint8_t* types, int n, int repeats, float* out,
                          cudaStream_t st) {
  const int sms = device_sms();
  const int blocks = min((n + 255) / 256, sms * 8);
  gather_bench_kernel<FMT><<<blocks, 256, 0, st>>>(M, pts, types, n, repeats, out);
  return cudaGetLastError();
}

}  // namespace

void grid_geometry(const dsdp_box* box, int n[3], double origin[3]) {
  for (int a = 0; a < 3; ++a) {
    n[a] = (int)ceil(box->size[a] / box->spacing);
    origin[a] = box->center[a] - (n[a] - 1) * box->spacing / 2.0;
  }
}

dsdp_status validate_box(const dsdp_box* box) {
  if (!box) return set_error(DSDP_ERR_INVALID_ARG, "box is NULL");
  if (!(box->spacing > 0.0) || !isfinite(box->spacing))
    return set_error(DSDP_ERR_INVALID_ARG, "box spacing must be positive");
  for (int a = 0; a < 3; ++a) {
    if (!isfinite(box->center[a]) || !isfinite(box->size[a]))
      return set_error(DSDP_ERR_INVALID_ARG, "box center/size not finite");
    if (!(box->size[a] > box->spacing))
      return set_error(DSDP_ERR_INVALID_ARG, "box size %g must exceed the spacing %g", box->size[a], box->spacing);
    if (box->size[a] / box->spacing > 4096.0) return set_error(DSDP_ERR_INVALID_ARG, "box has > 4096 vertices per axis");
  }
  int n[3];
  double o[3];
  grid_geometry(box, n, o);
  if ((double)DSDP_NUM_MAP_TYPES * n[0] * n[1] * n[2] >= 2147483648.0)
    return set_error(DSDP_ERR_INVALID_ARG, "grid of %d x %d x %d x 8 nodes exceeds 2^31 (32-bit map indices)", n[0],
                     n[1], n[2]);
  return DSDP_OK;
}

dsdp_status check_cuda(int err, const char* what) {
  if (err == cudaSuccess) return DSDP_OK;
  return set_error(DSDP_ERR_DEVICE, "%s: %s", what, cudaGetErrorString((cudaError_t)err));
}

}  // namespace dsdp

using namespace dsdp;

extern "C" uint64_t dsdp_grid_map_bytes(const dsdp_box* box, dsdp_map_dtype dtype, dsdp_grid_mode mode) {
  if (validate_box(box) != DSDP_OK || (int)dtype < 0 || (int)dtype > 2 || (int)mode < 0 || (int)mode > 1) return 0;
  int n[3];
  double o[3];
  grid_geometry(box, n, o);
  const int fmt = map_fmt((int)dtype, (int)mode);
  return (uint64_t)DSDP_NUM_MAP_TYPES * n[0] * n[1] * n[2] * fmt_channels(fmt) * fmt_elem_bytes(fmt);
}

extern "C" dsdp_status dsdp_grid_build_device(const dsdp_receptor* rec, const dsdp_box* box, dsdp_map_dtype dtype,
                                              dsdp_grid_mode mode, void* d_maps, uint64_t maps_bytes,
                                              void* stream) {
  dsdp_status s = validate_box(box);
  if (s != DSDP_OK) return s;
  if (!rec || rec->n < 0 || (rec->n > 0 && (!rec->xyz || !rec->xs_type)))
    return set_error(DSDP_ERR_INVALID_ARG, "receptor arrays invalid");
  if ((int)dtype < 0 || (int)dtype > 2 || (int)mode < 0 || (int)mode > 1)
    return set_error(DSDP_ERR_INVALID_ARG, "bad map dtype/mode");
  const uint64_t need = dsdp_grid_map_bytes(box, dtype, mode);
  if (!d_maps || maps_bytes < need)
    return set_error(DSDP_ERR_INVALID_ARG, "maps buffer %llu bytes < %llu", (unsigned long long)maps_bytes,
                     (unsigned long long)need);
  int n[3];
  double o[3];
  grid_geometry(box, n, o);
  const float h = (float)box->spacing;
  const cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e;
  switch (map_fmt((int)dtype, (int)mode)) {
    case 0: e = launch_grid<0>(rec, n[0], n[1], n[2], (float)o[0], (float)o[1], (float)o[2], h, d_maps, st); break;
    case 1: e = launch_grid<1>(rec, n[0], n[1], n[2], (float)o[0], (float)o[1], (float)o[2], h, d_maps, st); break;
    case 2: e = launch_grid<2>(rec, n[0], n[1], n[2], (float)o[0], (float)o[1], (float)o[2], h, d_maps, st); break;
    case 3: e = launch_grid<3>(rec, n[0], n[1], n[2], (float)o[0], (float)o[1], (float)o[2], h, d_maps, st); break;
    case 4: e = launch_grid<4>(rec, n[0], n[1], n[2], (float)o[0], (float)o[1], (float)o[2], h, d_maps, st); break;
    default: e = launch_grid<5>(rec, n[0], n[1], n[2], (float)o[0], (float)o[1], (float)o[2], h, d_maps, st); break;
  }
  return check_cuda(e, "grid_build_kernel launch");
}

MapView dsdp::map_view_of(const dsdp_grid_view* g) {
  MapView M;
  M.maps = g->d_maps;
  M.nx = g->n[0];
  M.ny = g->n[1];
  M.nz = g->n[2];
  M.ox = (float)g->origin[0];
  M.oy = (float)g->origin[1];
  M.oz = (float)g->origin[2];
  M.h = (float)g->spacing;
  M.inv_h = (float)(1.0 / g->spacing);
  return M;
}

extern "C" dsdp_status dsdp_gather_bench_device(const dsdp_grid_view* grid, const float* d_points,
                                                const uint8_t* d_types, int32_t n_points, int32_t repeats,
                                                float* d_out, void* stream) {
  if (!grid || !grid->d_maps || !d_points || !d_types || !d_out || n_points <= 0 || repeats <= 0)
    return set_error(DSDP_ERR_INVALID_ARG, "gather bench arguments invalid");
  if (grid->n[0] < 2 || grid->n[1] < 2 || grid->n[2] < 2) return set_error(DSDP_ERR_INVALID_ARG, "grid too small");
  const MapView M = map_view_of(grid);
  const cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e;
  switch (map_fmt(grid->dtype, grid->mode)) {
    case 0: e = launch_gather<0>(M, d_points, d_types, n_points, repeats, d_out, st); break;
    case 1: e = launch_gather<1>(M, d_points, d_types, n_points, repeats, d_out, st); break;
    case 2: e = launch_gather<2>(M, d_points, d_types, n_points, repeats, d_out, st); break;
    case 3: e = launch_gather<3>(M, d_points, d_types, n_points, repeats, d_out, st); break;
    case 4: e = launch_gather<4>(M, d_points, d_types, n_points, repeats, d_out, st); break;
    default: e = launch_gather<5>(M, d_points, d_types, n_points, repeats, d_out, st); break;
  }
  return check_cuda(e, "gather_bench_kernel launch");
}
