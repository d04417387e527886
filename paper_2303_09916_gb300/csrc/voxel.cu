// Receptor voxel features (Sec. 2, "Protein-ligand binding site prediction"):
// the input of the binding-site network, 36 x 36 x 36 voxels with 18
// channels over a 70 A cube centred on the protein; S and Se share one
// element channel and the freed channel marks the protein surface.
//
//   * voxel k of an axis covers [c - 35 + k 70/36, c - 35 + (k + 1) 70/36); an
//     atom's voxel is floor((x - (c - 35)) * (36/70)), FP32, subtraction then
//     multiplication; atoms outside the cube are dropped;
//   * channels 0..16: sums of the caller's 17 per-atom features over the
//     voxel's atoms; channel 17: the number of its surface atoms;
//   * surface atom (Shrake & Rupley, J. Mol. Biol. 79, 351 (1973)): some test
//     point x_i + (r_i + 1.4) u_k of its solvent-accessible sphere lies outside
//     the sphere of radius r_j + 1.4 of every other atom j; u_k are the 98
//     primitive integer vectors of {-2..2}^3, normalised (FP32, correctly
//     rounded square root and division); every point and distance test is FP32
//     with a fixed operation order (no contraction);
//   * sums are exact and order-free: features are rounded to multiples of 2^-24
//     and accumulated as 64-bit integers; a channel is the sum times 2^-24
//     rounded to FP32.
//
// Three launches.  voxel_bin_kernel sorts the atoms into cells of 4 voxels (one
// CTA, counting sort in shared memory; the others clear the accumulator).
// voxel_atoms_kernel gives an atom a warp, whose lanes hold its 98 test points
// (four per lane): it scans the cells in reach 32 atoms at a time, keeps those
// whose sphere can reach the atom's (a conservative FP32 pre-test), and each lane
// checks its points against them, broadcast by shuffle, until all are buried.
// voxel_finish_kernel writes the channels.
//
// Bound: latency (launches, L2 loads).  Scanning every atom for every atom, as
// receptors of more atoms than the output holds cell lists for still do, took
// 52 us of the call's 59 at 4,000 atoms.  The lists wait in the output array, which
// is written last.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "launch.h"

namespace dsdp {
namespace {

constexpr int kVoxN = DSDP_VOXEL_N;
constexpr int kVoxF = DSDP_VOXEL_FEATURES;
constexpr int kVoxC = DSDP_VOXEL_CHANNELS;
constexpr int kPointsPerLane = 4;  // 128 slots for the 98 directions
constexpr float kProbe = 1.4f;
constexpr float kFix = 16777216.0f;  // 2^24

// The 98 test directions as integer vectors (a, b, c) in {-2..2}^3 with
// gcd(|a|, |b|, |c|) = 1, built at compile time; a lane normalises its own.
struct SasDirs {
  signed char v[98][3];
};
constexpr int gcd_abs(int x, int y) {
  x = x < 0 ? -x : x;
  y = y < 0 ? -y : y;
  while (y) {
    const int t = x % y;
    x = y;
    y = t;
  }
  return x;
}
constexpr SasDirs make_sas_dirs() {
  SasDirs d{};
  int m = 0;
  for (int a = -2; a <= 2; ++a)
    for (int b = -2; b <= 2; ++b)
      for (int c = -2; c <= 2; ++c) {
        if ((a == 0 && b == 0 && c == 0) || gcd_abs(gcd_abs(a, b), c) != 1) continue;
        d.v[m][0] = (signed char)a;
        d.v[m][1] = (signed char)b;
        d.v[m][2] = (signed char)c;
        ++m;
      }
  return d;
}
static_assert(make_sas_dirs().v[97][0] == 2 && make_sas_dirs().v[97][1] == 2 && make_sas_dirs().v[97][2] == 1,
              "98 primitive directions");
__constant__ SasDirs c_sas_dirs = make_sas_dirs();

// Unit test direction m (0..97): the integer vector over its FP32 length
// (correctly rounded square root and division).
__device__ __forceinline__ float3 sas_direction(int m) {
  const int a = c_sas_dirs.v[m][0], b = c_sas_dirs.v[m][1], c = c_sas_dirs.v[m][2];
  const float len = __fsqrt_rn((float)(a * a + b * b + c * c));
  return make_float3(__fdiv_rn((float)a, len), __fdiv_rn((float)b, len), __fdiv_rn((float)c, len));
}

// Cells of 4 voxels: 9 per axis in the cube and one on either side for all that
// lies beyond it.
constexpr int kCells = kVoxN / 4 + 2;
constexpr int kCellCount = kCells * kCells * kCells;
constexpr float kCellInv = 36.0f / 70.0f / 4.0f;

// The sorted atoms' lists in the output array (4-byte aligned).
struct CellLists {
  int* start;         // [kCellCount + 1]
  float* max_radius;  // largest |r_i + 1.4|
  int* index;         // [n] the caller's index of each sorted atom
  float *x, *y, *z, *R;
};
constexpr int kListWords = kCellCount + 2;
constexpr int kMaxListed = (kVoxN * kVoxN * kVoxN * kVoxC - kListWords) / 5;
__host__ __device__ inline CellLists cell_lists(float* out, int n) {
  CellLists L;
  L.start = reinterpret_cast<int*>(out);
  L.max_radius = out + kCellCount + 1;
  float* p = out + kListWords;
  L.index = reinterpret_cast<int*>(p);
  L.x = p + n;
  L.y = p + 2 * n;
  L.z = p + 3 * n;
  L.R = p + 4 * n;
  return L;
}

// Cell of a coordinate along one axis (0: below the cube, kCells - 1: above);
// monotonic in x, so atoms closer than k cells are at most k cells apart.
__device__ __forceinline__ int cell_of(float x, float lo) {
  return (int)fminf(fmaxf(floorf((x - lo) * kCellInv) + 1.f, 0.f), (float)(kCells - 1));
}

__global__ void __launch_bounds__(1024) voxel_bin_kernel(int n, const float* __restrict__ xyz,
                                                         const float* __restrict__ radius, float lox, float loy,
                                                         float loz, CellLists L, unsigned long long* __restrict__ acc) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (blockIdx.x > 0) {
    const int total = kVoxN * kVoxN * kVoxN * kVoxC, stride = (gridDim.x - 1) * blockDim.x;
    const int q0 = (blockIdx.x - 1) * blockDim.x + tid;
    if ((reinterpret_cast<uintptr_t>(acc) & 15) == 0) {
      for (int q = q0; q < total / 2; q += stride) reinterpret_cast<ulonglong2*>(acc)[q] = make_ulonglong2(0ull, 0ull);
    } else {
      for (int q = q0; q < total; q += stride) acc[q] = 0ull;
    }
    return;
  }
  __shared__ int s_at[kCellCount];  // counts, then the next free place of each cell
  __shared__ int s_warp[32];
  __shared__ unsigned s_max;
  for (int c = tid; c < kCellCount; c += 1024) s_at[c] = 0;
  if (tid == 0) s_max = 0u;
  __syncthreads();
  // an atom that is not at a finite place is in no voxel and near no atom
  auto cell = [&](int i, float& x, float& y, float& z) {
    x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
    if (!isfinite(x) || !isfinite(y) || !isfinite(z)) return -1;
    return (cell_of(z, loz) * kCells + cell_of(y, loy)) * kCells + cell_of(x, lox);
  };
  float x, y, z, most = 0.f;
#pragma unroll 4
  for (int i = tid; i < n; i += 1024) {
    const int c = cell(i, x, y, z);
    if (c >= 0) atomicAdd(s_at + c, 1);
    most = fmaxf(most, fabsf(__fadd_rn(radius[i], kProbe)));  // NaN reaches nothing
  }
  atomicMax(&s_max, __float_as_uint(most));  // of non-negative floats
  __syncthreads();
  // exclusive prefix sums over the cells, two per thread
  const int c0 = 2 * tid, v0 = c0 < kCellCount ? s_at[c0] : 0, v1 = c0 + 1 < kCellCount ? s_at[c0 + 1] : 0;
  int inc = v0 + v1;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  int before = inc - v0 - v1 + __reduce_add_sync(0xffffffffu, lane < warp ? s_warp[lane] : 0);
  if (c0 < kCellCount) s_at[c0] = L.start[c0] = before;
  if (c0 + 1 < kCellCount) s_at[c0 + 1] = L.start[c0 + 1] = before + v0;
  if (c0 <= kCellCount - 1 && c0 + 2 > kCellCount - 1) L.start[kCellCount] = before + v0 + v1;
  if (tid == 0) *L.max_radius = __uint_as_float(s_max);
  __syncthreads();
#pragma unroll 4
  for (int i = tid; i < n; i += 1024) {
    const int c = cell(i, x, y, z);
    if (c < 0) continue;
    const int p = atomicAdd(s_at + c, 1);  // any order within a cell: what follows does not depend on it
    L.index[p] = i;
    L.x[p] = x, L.y[p] = y, L.z[p] = z;
    L.R[p] = __fadd_rn(radius[i], kProbe);
  }
}

// LISTED: atoms and neighbours from the cell lists; else every atom is scanned.
template <bool LISTED>
__global__ void __launch_bounds__(256) voxel_atoms_kernel(int n, const float* __restrict__ xyz,
                                                          const float* __restrict__ radius,
                                                          const float* __restrict__ feat, float lox, float loy,
                                                          float loz, CellLists L,
                                                          unsigned long long* __restrict__ acc) {
  const int lane = threadIdx.x & 31;
  const int warps = gridDim.x * (blockDim.x >> 5);
  // one direction per thread, shared by the CTA's warps: per lane and warp the
  // divergent reads of the constant table and the divisions were a third of the kernel
  __shared__ float3 s_dir[32 * kPointsPerLane];
  if (threadIdx.x < 32 * kPointsPerLane)
    s_dir[threadIdx.x] = threadIdx.x < 98 ? sas_direction(threadIdx.x) : make_float3(0.f, 0.f, 0.f);
  __syncthreads();
  float3 u[kPointsPerLane];
  bool used[kPointsPerLane];
#pragma unroll
  for (int s = 0; s < kPointsPerLane; ++s) {
    used[s] = lane + 32 * s < 98;
    u[s] = s_dir[lane + 32 * s];
  }
  const float inv = 36.0f / 70.0f;
  const int count = LISTED ? L.start[kCellCount] : n;
  // cells in reach on either side: no sphere reaches farther than the two largest;
  // a little more against the rounding of the cells
  const int reach_cells =
      LISTED ? (int)fminf(floorf((2.f * *L.max_radius + 0.02f) * kCellInv + 1e-3f) + 1.f, (float)kCells) : 0;
  for (int p = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < count; p += warps) {  // warp-uniform
    const int i = LISTED ? L.index[p] : p;
    const float xi = LISTED ? L.x[p] : xyz[3 * i], yi = LISTED ? L.y[p] : xyz[3 * i + 1],
                zi = LISTED ? L.z[p] : xyz[3 * i + 2];
    const float ux = __fmul_rn(__fsub_rn(xi, lox), inv), uy = __fmul_rn(__fsub_rn(yi, loy), inv),
                uz = __fmul_rn(__fsub_rn(zi, loz), inv);
    // floor(u) in [0, 36) exactly when u in [0, 36) (false for NaN): tested before any conversion
    if (!(ux >= 0.f && ux < (float)kVoxN && uy >= 0.f && uy < (float)kVoxN && uz >= 0.f && uz < (float)kVoxN))
      continue;
    const int kx = (int)ux, ky = (int)uy, kz = (int)uz;
    unsigned long long* v = acc + (((size_t)kz * kVoxN + ky) * kVoxN + kx) * kVoxC;
    if (lane < kVoxF) {
      const long long q = __float2ll_rn(__fmul_rn(feat[(size_t)kVoxF * i + lane], kFix));
      if (q) atomicAdd(v + lane, (unsigned long long)q);
    }
    // ---- surface test
    const float Ri = LISTED ? L.R[p] : __fadd_rn(radius[i], kProbe);
    float px[kPointsPerLane], py[kPointsPerLane], pz[kPointsPerLane];
    bool buried[kPointsPerLane];
#pragma unroll
    for (int s = 0; s < kPointsPerLane; ++s) {
      px[s] = __fadd_rn(xi, __fmul_rn(Ri, u[s].x));
      py[s] = __fadd_rn(yi, __fmul_rn(Ri, u[s].y));
      pz[s] = __fadd_rn(zi, __fmul_rn(Ri, u[s].z));
      buried[s] = !used[s];
    }
    // atoms [j0, j1) of the list (or of the receptor) against the points, until all are buried
    bool hidden = false;
    auto scan = [&](int j0, int j1) {
      for (; j0 < j1 && !hidden; j0 += 32) {
        const int j = j0 + lane;
        float xj = 0.f, yj = 0.f, zj = 0.f, Rj = 0.f;
        bool near = false;
        if (j < j1 && j != p) {
          xj = LISTED ? L.x[j] : xyz[3 * j];
          yj = LISTED ? L.y[j] : xyz[3 * j + 1];
          zj = LISTED ? L.z[j] : xyz[3 * j + 2];
          Rj = LISTED ? L.R[j] : __fadd_rn(radius[j], kProbe);
          // a sphere farther than Ri + Rj cannot cover a point of atom i's sphere;
          // 0.01 A of slack keeps the pre-test conservative under FP32 rounding
          const float dx = xj - xi, dy = yj - yi, dz = zj - zi, reach = Ri + Rj + 0.01f;
          near = dx * dx + dy * dy + dz * dz < reach * reach;
        }
        unsigned m = __ballot_sync(0xffffffffu, near);
        if (!m) continue;
        while (m) {  // warp-uniform
          const int src = __ffs(m) - 1;
          m &= m - 1;
          const float bx = __shfl_sync(0xffffffffu, xj, src), by = __shfl_sync(0xffffffffu, yj, src),
                      bz = __shfl_sync(0xffffffffu, zj, src), bR = __shfl_sync(0xffffffffu, Rj, src);
          const float R2 = __fmul_rn(bR, bR);
#pragma unroll
          for (int s = 0; s < kPointsPerLane; ++s) {
            const float dx = __fsub_rn(px[s], bx), dy = __fsub_rn(py[s], by), dz = __fsub_rn(pz[s], bz);
            const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
            buried[s] = buried[s] || d2 < R2;
          }
        }
        bool all = true;
#pragma unroll
        for (int s = 0; s < kPointsPerLane; ++s) all = all && buried[s];
        hidden = __all_sync(0xffffffffu, all);
      }
    };
    if (LISTED) {
      const int cx = cell_of(xi, lox), cy = cell_of(yi, loy), cz = cell_of(zi, loz);
      const int x0 = max(cx - reach_cells, 0), x1 = min(cx + reach_cells, kCells - 1), m = 2 * reach_cells + 1;
      // rows of cells along x are contiguous in the list; the atom's own row first
      for (int q = 0; q < m * m && !hidden; ++q) {
        const int r = (q + (m * m) / 2) % (m * m), rz = cz + r / m - reach_cells, ry = cy + r % m - reach_cells;
        if (rz < 0 || rz >= kCells || ry < 0 || ry >= kCells) continue;
        const int row = (rz * kCells + ry) * kCells;
        scan(L.start[row + x0], L.start[row + x1 + 1]);
      }
    } else {
      scan(0, n);
    }
    if (!hidden && lane == 0) atomicAdd(v + kVoxF, (unsigned long long)(1ll << 24));
  }
}

// Each sum times 2^-24, rounded to FP32 once.  Most voxels are empty and most sums
// whole numbers; the others go through FP64, of which an SM does two a cycle.
__global__ void __launch_bounds__(256) voxel_finish_kernel(const unsigned long long* __restrict__ acc,
                                                           float* __restrict__ out, int n) {
  const int stride = gridDim.x * blockDim.x;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride) {
    const long long v = (long long)acc[q];
    float f = 0.f;
    if (v != 0) {
      const long long whole = v >> 24;
      f = (v & 0xffffffll) == 0 && whole == (int)whole ? (float)(int)whole
                                                       : __double2float_rn(__ll2double_rn(v) * (1.0 / 16777216.0));
    }
    out[q] = f;
  }
}

bool overlap(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
  return x < y + nb && y < x + na;
}

}  // namespace
}  // namespace dsdp

using namespace dsdp;

extern "C" uint64_t dsdp_voxel_work_bytes(void) {
  return sizeof(unsigned long long) * (uint64_t)kVoxN * kVoxN * kVoxN * kVoxC;
}

extern "C" dsdp_status dsdp_voxelize_device(int32_t n_atoms, const float* d_xyz, const float* d_radius,
                                            const float* d_features, const double center[3], float* d_out,
                                            void* d_work, uint64_t work_bytes, void* stream) {
  if (n_atoms < 0) return set_error(DSDP_ERR_INVALID_ARG, "n_atoms %d < 0", n_atoms);
  if (!center || !d_out || !d_work) return set_error(DSDP_ERR_INVALID_ARG, "voxelize: center, out or work NULL");
  if (n_atoms > 0 && (!d_xyz || !d_radius || !d_features))
    return set_error(DSDP_ERR_INVALID_ARG, "voxelize: atom arrays NULL");
  if (work_bytes < dsdp_voxel_work_bytes())
    return set_error(DSDP_ERR_INVALID_ARG, "voxelize: work of %llu bytes < %llu", (unsigned long long)work_bytes,
                     (unsigned long long)dsdp_voxel_work_bytes());
  if (((uintptr_t)d_work & 7) != 0) return set_error(DSDP_ERR_INVALID_ARG, "voxelize: work not 8-byte aligned");
  for (int a = 0; a < 3; ++a)
    if (!isfinite(center[a])) return set_error(DSDP_ERR_INVALID_ARG, "voxelize: center not finite");
  const cudaStream_t st = (cudaStream_t)stream;
  unsigned long long* acc = (unsigned long long*)d_work;
  const int total = kVoxN * kVoxN * kVoxN * kVoxC;
  const float lox = (float)(center[0] - 35.0), loy = (float)(center[1] - 35.0), loz = (float)(center[2] - 35.0);
  const int sms = device_sms();
  const int want = (n_atoms + 7) / 8, cap = sms * 8;  // 8 warps (atoms) per CTA
  const int grid = want < cap ? want : cap;
  const CellLists lists = cell_lists(d_out, n_atoms);
  // the lists lie in the output: not where the output may take an input's place
  const size_t out_bytes = sizeof(float) * (size_t)total, atoms = (size_t)n_atoms;
  const bool listed = n_atoms > 0 && n_atoms <= kMaxListed && !overlap(d_out, out_bytes, d_xyz, 12 * atoms) &&
                      !overlap(d_out, out_bytes, d_radius, 4 * atoms) &&
                      !overlap(d_out, out_bytes, d_features, 4 * kVoxF * atoms);
  cudaError_t e = cudaSuccess;
  if (listed) {
    voxel_bin_kernel<<<1 + sms, 1024, 0, st>>>(n_atoms, d_xyz, d_radius, lox, loy, loz, lists, acc);
    voxel_atoms_kernel<true>
        <<<grid, 256, 0, st>>>(n_atoms, d_xyz, d_radius, d_features, lox, loy, loz, lists, acc);
    e = cudaGetLastError();
  } else {
    e = cudaMemsetAsync(acc, 0, dsdp_voxel_work_bytes(), st);
    if (e == cudaSuccess && n_atoms > 0) {
      voxel_atoms_kernel<false>
          <<<grid, 256, 0, st>>>(n_atoms, d_xyz, d_radius, d_features, lox, loy, loz, lists, acc);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess) {
    voxel_finish_kernel<<<sms * 8, 256, 0, st>>>(acc, d_out, total);
    e = cudaGetLastError();
  }
  return check_cuda(e, "voxelize launch");
}
