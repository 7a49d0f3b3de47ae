// pair_common.h -- what the short-range pair kernels of both precisions share:
// the pair functions' constants, the kernel arguments and the table of a
// target run's neighbour rows.
#pragma once

#include <climits>
#include <cmath>

#include "msm_internal.h"

namespace msm {

constexpr unsigned kFull = 0xffffffffu;

// Cutoff constants of the FP32 pair functions, and the cell grid.
struct PairArgs {
  int nc[3];
  int periodic;
  float a2f, inv_af, inv_a2f, two_inv_a3f;
};

// Constants of the Wolf pair function (damped, shifted force) with damping
// alpha and cutoff R = a: v(r) = erfc(alpha r)/r - vR + c1 (r - R),
// vR = erfc(alpha R)/R, c1 = erfc(alpha R)/R^2 + c2 exp(-alpha^2 R^2)/R,
// c2 = 2 alpha/sqrt(pi).
template <typename T>
struct WolfC {
  T alpha, alpha2, c2, vR, c1, R;
};

template <typename T>
WolfC<T> wolf_consts(double alpha, double R) {
  const double c2 = 2.0 * alpha / std::sqrt(M_PI);
  const double vR = std::erfc(alpha * R) / R;
  const double c1 = std::erfc(alpha * R) / (R * R) + c2 * std::exp(-alpha * alpha * R * R) / R;
  return WolfC<T>{(T)alpha, (T)(alpha * alpha), (T)c2, (T)vR, (T)c1, (T)R};
}

__device__ __forceinline__ float d_erfc(float x) { return erfcf(x); }
__device__ __forceinline__ double d_erfc(double x) { return erfc(x); }
__device__ __forceinline__ float d_exp(float x) { return expf(x); }
__device__ __forceinline__ double d_exp(double x) { return exp(x); }

// Pair functions: K = 0 is MSM's short-range kernel g*(r) = 1/r - gamma(r/a)/a
// (zero with its derivative at r = a); K = 1 is the plain Coulomb law 1/r of
// the cutoff method (the parareal section's coarse propagator G), which is
// not zero at a, so sources beyond the cutoff are masked; K = 2 is Wolf
// summation's damped, shifted-force pair potential (another coarse function
// of that section), masked beyond a as well.
constexpr int kPairMSM = 0, kPairCutoff = 1, kPairWolf = 2;

// gamma(r/a)/a and (2/a^3) dgamma/ds written straight as polynomials in r^2
// (host-scaled coefficients, duplicated into float2 pairs):
//   pot = 1/r - sum_k G[k] r2^k,   f' = 1/r^3 + sum_k D[k] r2^k.
// Beyond the cutoff r2 is clamped to a^2: pot and f' are zero there up to
// FP32 rounding (a few 1e-8 / a per source, measured to leave the energy and
// forces of the 1.07M-atom water box unchanged at the 1e-8 / 1e-7 level).
struct PairCoef {
  float2 G[4];
  float2 D[3];
};

constexpr int kMaxRows = 32;  // rows per cell: cells at least a/2 wide give at most 26

// Arguments of the packed pair kernel (one system).
struct PairKArgs {
  const R4<float>* atoms;
  const int* cell_start;
  const int4* rows;
  int nrows;
  PairArgs A;
  PairCoef C;
  WolfC<float> W;
  float cwx, cwy, cwz;
  int ncell;
  float* phis;
  R4<float>* fs;
  // target runs
  const int* scell;    // cell of every sorted atom
  const float* cellx;  // its x index
  int natoms;
  int runs;     // groups are runs of consecutive sorted atoms (else the chunks of a cell)
  int split;    // warps sharing a group's sources (1, or the block's kWarps)
  int maxspan;  // cells a run's piece may add to its first one
};

__device__ __forceinline__ float warp_min(float v) {
  float r;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float warp_max(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

// The sources of a piece (targets in cells cx .. cx + span of one row): rows
// of neighbour cells are contiguous in the sorted atoms (cells are numbered x
// fastest), one or two ranges each (two where a periodic row wraps).  rec: the
// range's first atom and end, the x base b and (dy + 3) | (dz + 3) << 4; an
// atom of the range lies cellx + b cells from cx along x.
struct SegList {
  int4 rec[2 * kMaxRows];
};

// Builds the list (lane r: row r of the plan's rows), each row widened by span
// cells in +x (the home row's right part moved past the piece's cells), then
// narrowed to the cells a source within a of the targets' bounding box
// (lx..hx, ly..hy, lz..hz, in the frame of cell cx) can lie in: a row at y gap
// gy and z gap gz from the box reaches sqrt(a^2 - gy^2 - gz^2) beyond it in x
// (with a margin for rounding; the culling tests each source exactly).
// Returns the number of ranges.
__device__ __forceinline__ int build_segments(SegList& L, const PairKArgs& K, int cx, int cy, int cz, int span,
                                              float lx, float ly, float lz, float hx, float hy, float hz, int lane) {
  const int* __restrict__ cell_start = K.cell_start;
  const PairArgs& A = K.A;
  const int ncx = A.nc[0], ncy = A.nc[1], ncz = A.nc[2];
  int4 r0 = make_int4(0, 0, 0, 0), r1 = r0;
  if (lane < K.nrows) {
    int4 row = K.rows[lane];  // (dy, dz, xlo, xhi)
    const int oyz = (row.x + 3) | ((row.y + 3) << 4);
    if (row.x == 0 && row.y == 0) {
      if (row.z > 0) { row.z += span; row.w += span; }  // the home row's right part
    } else {
      row.w += span;
    }
    const float gy = fmaxf(fmaxf(row.x * K.cwy - hy, ly - (row.x + 1) * K.cwy), 0.f);
    const float gz = fmaxf(fmaxf(row.y * K.cwz - hz, lz - (row.y + 1) * K.cwz), 0.f);
    const float r2 = A.a2f - gy * gy - gz * gz;
    bool inside = r2 > 0.f;
    if (inside) {
      const float reach = sqrtf(r2) * 1.0001f + 1e-3f;
      row.z = max(row.z, (int)floorf((lx - reach) / K.cwx));
      row.w = min(row.w, (int)floorf((hx + reach) / K.cwx));
    }
    int ny = cy + row.x, nz = cz + row.y;
    if (A.periodic) {
      ny += (ny < 0) ? ncy : ((ny >= ncy) ? -ncy : 0);
      nz += (nz < 0) ? ncz : ((nz >= ncz) ? -ncz : 0);
    } else if (ny < 0 || nz < 0 || ny >= ncy || nz >= ncz) {
      inside = false;
    }
    if (inside) {
      const int* cs = cell_start + (nz * ncy + ny) * ncx + cx;
      // the row's cells inside the grid, then those beyond one end (the row
      // holds at most ncx cells, so it wraps at one end at most)
      const int a0 = max(row.z, -cx), a1 = min(row.w, ncx - 1 - cx);
      if (a0 <= a1) r0 = make_int4(cs[a0], cs[a1 + 1], -cx, oyz);
      if (A.periodic && row.z < -cx) {
        const int b1 = min(row.w, -cx - 1);
        r1 = make_int4(cs[row.z + ncx], cs[b1 + ncx + 1], -cx - ncx, oyz);
      } else if (A.periodic && row.w >= ncx - cx) {
        const int b0 = max(row.z, ncx - cx);
        r1 = make_int4(cs[b0 - ncx], cs[row.w - ncx + 1], -cx + ncx, oyz);
      }
    }
  }
  const unsigned lt = (1u << lane) - 1u;
  const unsigned m0 = __ballot_sync(kFull, r0.x < r0.y), m1 = __ballot_sync(kFull, r1.x < r1.y);
  // a row's two ranges side by side: the rows keep the plan's order
  const int at = __popc(m0 & lt) + __popc(m1 & lt);
  if (r0.x < r0.y) L.rec[at] = r0;
  if (r1.x < r1.y) L.rec[at + (r0.x < r0.y ? 1 : 0)] = r1;
  __syncwarp();
  return __popc(m0) + __popc(m1);
}

// The arguments of plan P (kernels_pair.cu; natoms is the caller's).
PairKArgs pair_kargs(const Plan& P);
// The pair sums of an FP64 plan (kernels_pair64.cu); kind is one of kPair*.
cudaError_t launch_pair64(Plan& P, int kind, int64_t n, double alpha, cudaStream_t st);

}  // namespace msm
