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
  // target runs (short_range_run_body): cell of every input atom, the sorted
  // order's input indices and the atom count
  const int* key;
  const int* perm;
  int natoms;
};

constexpr int kRunBnd = 6;  // boundaries inside a row segment of up to 7 cells
struct SegTableR {
  int4 rec[2 * kMaxRows + 1];         // (first atom, flat start, x offset of the first cell, (dy + 3) | (dz + 3) << 4); sentinel at the end
  int4 bnd[2 * kMaxRows];             // first atom of the segment's 2nd..5th cell (INT_MAX where absent)
  int2 bnd2[2 * kMaxRows];            // ... of its 6th and 7th cell
  float2 shift[2 * kMaxRows];         // (y, z) shift of the row
};

// The segment table of the rows about cells (cx .. cx + span, cy, cz): as
// build_seg_table, each row widened by span cells in +x (the home row's
// right part moved past the piece's cells), then narrowed to the cells a
// source within a of the targets' bounding box (lx..hx, ly..hy, lz..hz, in
// the frame of cell cx) can lie in: a row at y gap gy and z gap gz from the
// box reaches sqrt(a^2 - gy^2 - gz^2) beyond it in x (with a margin for
// rounding; the culling tests each source exactly).
__device__ __forceinline__ int build_seg_table_run(SegTableR& T, const PairKArgs& K, int cx, int cy, int cz, int span,
                                                   float lx, float ly, float lz, float hx, float hy, float hz,
                                                   int lane) {
  const int* __restrict__ cell_start = K.cell_start;
  const PairArgs& A = K.A;
  const int ncx = A.nc[0], ncy = A.nc[1], ncz = A.nc[2];
  const int nrows = K.nrows;
  const float cwy = K.cwy, cwz = K.cwz;
  int len[2] = {0, 0}, j0s[2] = {0, 0}, ox0s[2] = {0, 0};
  int bb[2][kRunBnd];
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int t = 0; t < kRunBnd; ++t) bb[g][t] = INT_MAX;
  float2 sh = make_float2(0.f, 0.f);
  int oyz = 0;
  if (lane < nrows) {
    int4 row = K.rows[lane];  // (dy, dz, xlo, xhi)
    oyz = (row.x + 3) | ((row.y + 3) << 4);
    if (row.x == 0 && row.y == 0) {
      if (row.z > 0) { row.z += span; row.w += span; }  // the home row's right part
    } else {
      row.w += span;
    }
    const float gy = fmaxf(fmaxf(row.x * cwy - hy, ly - (row.x + 1) * cwy), 0.f);
    const float gz = fmaxf(fmaxf(row.y * cwz - hz, lz - (row.y + 1) * cwz), 0.f);
    const float r2 = A.a2f - gy * gy - gz * gz;
    bool inside = r2 > 0.f;
    if (inside) {
      const float reach = sqrtf(r2) * 1.0001f + 1e-3f;
      row.z = max(row.z, (int)floorf((lx - reach) / K.cwx));
      row.w = min(row.w, (int)floorf((hx + reach) / K.cwx));
      inside = row.z <= row.w;
    }
    int ny = cy + row.x, nz = cz + row.y;
    if (A.periodic) {
      ny += (ny < 0) ? ncy : ((ny >= ncy) ? -ncy : 0);
      nz += (nz < 0) ? ncz : ((nz >= ncz) ? -ncz : 0);
    } else if (ny < 0 || nz < 0 || ny >= ncy || nz >= ncz) {
      inside = false;
    }
    const int rbase = (nz * ncy + ny) * ncx;
    sh = make_float2(row.x * cwy, row.y * cwz);
#pragma unroll
    for (int seg = 0; seg < 2; ++seg) {
      int ox0 = 0, ox1 = -1;
      if (!inside) {
      } else if (A.periodic) {  // at most 7 <= ncx cells: the row wraps at one end at most
        const int xa = cx + row.z, xb = cx + row.w;
        if (xa < 0) {
          if (seg == 0) { ox0 = row.z; ox1 = -cx - 1; } else { ox0 = -cx; ox1 = row.w; }
        } else if (xb >= ncx) {
          if (seg == 0) { ox0 = row.z; ox1 = ncx - 1 - cx; } else { ox0 = ncx - cx; ox1 = row.w; }
        } else if (seg == 0) {
          ox0 = row.z; ox1 = row.w;
        }
      } else if (seg == 0) {
        ox0 = max(row.z, -cx);
        ox1 = min(row.w, ncx - 1 - cx);
      }
      if (ox0 <= ox1) {
        int x0 = cx + ox0, x1 = cx + ox1;
        if (A.periodic) {
          x0 += (x0 < 0) ? ncx : ((x0 >= ncx) ? -ncx : 0);
          x1 += (x1 < 0) ? ncx : ((x1 >= ncx) ? -ncx : 0);
        }
        const int j0 = cell_start[rbase + x0], j1 = cell_start[rbase + x1 + 1];
#pragma unroll
        for (int t = 0; t < kRunBnd; ++t) bb[seg][t] = (x0 + 1 + t <= x1) ? cell_start[rbase + x0 + 1 + t] : INT_MAX;
        len[seg] = j1 - j0;
        j0s[seg] = j0;
        ox0s[seg] = ox0;
      }
    }
  }
  const int mine = len[0] + len[1];
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  const int total = __shfl_sync(kFull, incl, 31);
  const int start = incl - mine;
  if (lane < nrows) {
#pragma unroll
    for (int seg = 0; seg < 2; ++seg) {
      T.rec[2 * lane + seg] = make_int4(j0s[seg], seg ? start + len[0] : start, ox0s[seg], oyz);
      T.bnd[2 * lane + seg] = make_int4(bb[seg][0], bb[seg][1], bb[seg][2], bb[seg][3]);
      T.bnd2[2 * lane + seg] = make_int2(bb[seg][4], bb[seg][5]);
      T.shift[2 * lane + seg] = sh;
    }
  }
  if (lane == 0) T.rec[2 * nrows] = make_int4(0, INT_MAX, 0, 0);
  __syncwarp();
  return total;
}


// The arguments of plan P (kernels_pair.cu; natoms is the caller's).
PairKArgs pair_kargs(const Plan& P);
// The pair sums of an FP64 plan (kernels_pair64.cu); kind is one of kPair*.
cudaError_t launch_pair64(Plan& P, int kind, int64_t n, double alpha, cudaStream_t st);

}  // namespace msm
