// kernels_pair.cu -- short-range part of MSM on mixed plans (FP64 plans:
// kernels_pair64.cu; Sec. "Multilevel Summation Method"):
// u_i^short = sum_{j != i, r_ij < a} q_j g*(r_ij) with
// g*(r) = 1/r - gamma(r/a)/a (Eq. msmgrid), and the force
// F_i = -q_i grad_i u_i^short.
//
// One warp owns one cell of the sort-binned atoms (cells at least a/2 wide):
// its lanes hold up to 32 target atoms and walk the neighbour cells within
// reach (offsets whose closest points are nearer than a).  Source atoms are
// shifted into the target cell's frame (every difference is between small
// cell-local coordinates), culled against the bounding box of the targets,
// and queued in the warp's shared memory; full queues are broadcast to the
// lanes in unrolled batches.  Each pair costs one rsqrt and ~20 FP32
// operations; rejected pairs are masked, not branched.  Mixed precision sums
// each batch in FP32 and folds the batch sums into the running totals with an
// error-free TwoSum (compensated accumulation).
#include <algorithm>
#include <new>

#include "pair_common.h"

namespace msm {

namespace {

PairArgs pair_args(const Plan& P) {
  PairArgs A;
  for (int d = 0; d < 3; ++d) A.nc[d] = P.nc[d];
  A.periodic = P.P.periodic;
  const double a = P.P.cutoff;
  A.a2f = (float)(a * a);
  A.inv_af = (float)(1.0 / a);
  A.inv_a2f = (float)(1.0 / (a * a));
  A.two_inv_a3f = (float)(2.0 / (a * a * a));
  return A;
}

template <typename T, int M>
struct Smooth;  // gamma(rho) and d gamma / d s as polynomials in s = rho^2 < 1

template <typename T>
struct Smooth<T, 1> {
  __device__ static T g(T s) { return T(1.5) - T(0.5) * s; }
  __device__ static T gs(T) { return T(-0.5); }
};
template <typename T>
struct Smooth<T, 2> {
  __device__ static T g(T s) { return T(1.875) + s * (T(-1.25) + T(0.375) * s); }
  __device__ static T gs(T s) { return T(-1.25) + T(0.75) * s; }
};
template <typename T>
struct Smooth<T, 3> {
  __device__ static T g(T s) {
    return T(2.1875) + s * (T(-2.1875) + s * (T(1.3125) - T(0.3125) * s));
  }
  __device__ static T gs(T s) { return T(-2.1875) + s * (T(2.625) - T(0.9375) * s); }
};

// error-free transformation s + x = t + err; the error goes to the compensation term
template <typename T>
__device__ __forceinline__ void two_sum_add(T& s, T& c, T x) {
  T t = s + x;
  T bp = t - s;
  c += (s - (t - bp)) + (x - bp);
  s = t;
}

constexpr int kWarps = 4;
constexpr int kBatch = 64;  // sources per queue drain (pairs per lane per drain)

__device__ __forceinline__ float fast_rsqrt(float x) {  // one MUFU.RSQ; inputs are >= a^2/... never denormal
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// One pair, scalar: target ai against source b (skipped at r = 0, the atom
// itself, and beyond the cutoff); adds q_j times the pair potential to pphi
// and f (r_i - r_j) to (px, py, pz) with f = q_j v'(r)/r.
template <typename T, int M, int K>
__device__ __forceinline__ void pair1(const R4<T>& ai, const R4<T>& b, T a2, T inv_a, T inv_a2, T two_inv_a3,
                                      const WolfC<T>& W, T& pphi, T& px, T& py, T& pz) {
  const T dx = ai.x - b.x, dy = ai.y - b.y, dz = ai.z - b.z;
  const T r2 = dx * dx + dy * dy + dz * dz;
  const bool ok = (r2 < a2) && (r2 > T(0));  // inside the cutoff, not the atom itself
  const T r2s = ok ? r2 : a2;
  const T qj = ok ? b.w : T(0);
  const T rinv = fast_rsqrt(r2s);
  T f;
  if (K == kPairMSM) {
    const T s = r2s * inv_a2;
    pphi += qj * (rinv - Smooth<T, M>::g(s) * inv_a);
    f = qj * (-(rinv * rinv * rinv) - two_inv_a3 * Smooth<T, M>::gs(s));
  } else if (K == kPairWolf) {  // f = q_j v'(r) / r
    const T r = r2s * rinv;
    const T e = d_erfc(W.alpha * r), g = W.c2 * d_exp(-W.alpha2 * r2s);
    pphi += qj * (e * rinv - W.vR + W.c1 * (r - W.R));
    f = qj * (W.c1 * rinv - (e * rinv + g) * rinv * rinv);
  } else {
    pphi += qj * rinv;
    f = -qj * (rinv * rinv * rinv);
  }
  px += f * dx;
  py += f * dy;
  pz += f * dz;
}

// ---- mixed precision: packed FP32x2 arithmetic (two sources per instruction) ----
// The queue is stored as four FP32 arrays (x, y, z, q), so sources j..j+3
// load as one float4 per array and feed FFMA2/FMUL2/FADD2 as two pairs.  With
// d = r_j - r_i, f' = q_j (1/r^3 + 2 gamma_s(s)/a^3) and
// F_i = -q_i sum_j f' d, which needs no negations in the loop.  The home cell
// (the only one that holds the target itself) goes through the scalar batch
// with the self test; every other cell skips that test.  Far-away padding
// sits at 1e6 so that the unmasked polynomial stays finite.
struct alignas(16) QueueF {
  float x[2 * kBatch], y[2 * kBatch], z[2 * kBatch], q[2 * kBatch];
};

template <int M>
__device__ __forceinline__ float2 poly_g(const PairCoef& C, float2 r2) {
  float2 t = C.G[M];
#pragma unroll
  for (int k = M - 1; k >= 0; --k) t = __ffma2_rn(t, r2, C.G[k]);
  return t;
}
template <int M>
__device__ __forceinline__ float2 poly_d(const PairCoef& C, float2 r2) {
  float2 t = C.D[M - 1];
#pragma unroll
  for (int k = M - 2; k >= 0; --k) t = __ffma2_rn(t, r2, C.D[k]);
  return t;
}

// One packed step: the lane's target (negated coordinates nax, nay, naz)
// against two sources (bx, by, bz, bq); adds q_j times the pair potential to
// sphi and f' d to (sx, sy, sz) with d = r_j - r_i.  Outside the home cell a
// source is never at r = 0; SELF (the home cell, which holds the target
// itself) drops a source at r = 0: its charge becomes 0 and r^2 becomes a^2.
template <int M, int K, bool SELF = false>
__device__ __forceinline__ void pair2(float2 bx, float2 by, float2 bz, float2 bq, float2 nax, float2 nay, float2 naz,
                                      float a2, const PairCoef& C, const WolfC<float>& W, float2& sphi, float2& sx,
                                      float2& sy, float2& sz) {
  const float2 dx = __fadd2_rn(bx, nax), dy = __fadd2_rn(by, nay), dz = __fadd2_rn(bz, naz);
  float2 r2 = __fmul2_rn(dx, dx);
  r2 = __ffma2_rn(dy, dy, r2);
  r2 = __ffma2_rn(dz, dz, r2);
  if (SELF) {
    bq = make_float2(r2.x > 0.f ? bq.x : 0.f, r2.y > 0.f ? bq.y : 0.f);
    r2 = make_float2(r2.x > 0.f ? r2.x : a2, r2.y > 0.f ? r2.y : a2);
  }
  float2 fp;
  if (K == kPairMSM) {
    // a source beyond the cutoff is evaluated at r = a, where g* and its
    // derivative vanish (C1 smoothing): no select on q_j is needed
    r2 = make_float2(fminf(r2.x, a2), fminf(r2.y, a2));
    const float2 qj = bq;
    const float2 rinv = make_float2(fast_rsqrt(r2.x), fast_rsqrt(r2.y));
    const float2 pot = __fadd2_rn(rinv, poly_g<M>(C, r2));  // G holds -gamma coefficients
    sphi = __ffma2_rn(qj, pot, sphi);
    fp = __fmul2_rn(__ffma2_rn(__fmul2_rn(rinv, rinv), rinv, poly_d<M>(C, r2)), qj);
  } else if (K == kPairWolf) {
    // damped shifted force within the cutoff; erfc(x) by Abramowitz and
    // Stegun 7.1.26, t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) exp(-x^2),
    // t = 1 / (1 + p x), |error| < 1.5e-7 for x >= 0, whose exp(-x^2) is the
    // force term's exp(-alpha^2 r^2) as well
    const bool okx = r2.x < a2, oky = r2.y < a2;
    const float2 r2s = make_float2(okx ? r2.x : a2, oky ? r2.y : a2);
    const float2 q = make_float2(okx ? bq.x : 0.f, oky ? bq.y : 0.f);
    const float2 ri = make_float2(fast_rsqrt(r2s.x), fast_rsqrt(r2s.y));
    const float2 r = __fmul2_rn(r2s, ri);
    const float2 al = make_float2(W.alpha, W.alpha);
    const float2 x = __fmul2_rn(al, r);
    const float2 den = __ffma2_rn(make_float2(0.3275911f, 0.3275911f), x, make_float2(1.f, 1.f));
    const float2 t = make_float2(__fdividef(1.f, den.x), __fdividef(1.f, den.y));
    float2 poly = make_float2(1.061405429f, 1.061405429f);
    poly = __ffma2_rn(poly, t, make_float2(-1.453152027f, -1.453152027f));
    poly = __ffma2_rn(poly, t, make_float2(1.421413741f, 1.421413741f));
    poly = __ffma2_rn(poly, t, make_float2(-0.284496736f, -0.284496736f));
    poly = __ffma2_rn(poly, t, make_float2(0.254829592f, 0.254829592f));
    const float2 ex = make_float2(__expf(-W.alpha2 * r2s.x), __expf(-W.alpha2 * r2s.y));
    const float2 e = __fmul2_rn(__fmul2_rn(poly, t), ex);  // erfc(alpha r)
    const float2 er = __fmul2_rn(e, ri);
    // q (erfc(alpha r) / r - v_R + c1 (r - R)) and -v'(r) / r = q ((e/r + c2 ex) / r^2 - c1 / r)
    const float2 c1v = make_float2(W.c1, W.c1);
    const float2 pot = __ffma2_rn(c1v, __fadd2_rn(r, make_float2(-W.R, -W.R)), __fadd2_rn(er, make_float2(-W.vR, -W.vR)));
    sphi = __ffma2_rn(q, pot, sphi);
    const float2 inner = __ffma2_rn(make_float2(W.c2, W.c2), ex, er);
    fp = __fmul2_rn(q, __ffma2_rn(__fmul2_rn(inner, ri), ri, __fmul2_rn(make_float2(-W.c1, -W.c1), ri)));
  } else {  // plain Coulomb within the cutoff
    const float2 qj = make_float2(r2.x < a2 ? bq.x : 0.f, r2.y < a2 ? bq.y : 0.f);
    const float2 rinv = make_float2(fast_rsqrt(r2.x), fast_rsqrt(r2.y));
    sphi = __ffma2_rn(qj, rinv, sphi);
    fp = __fmul2_rn(__fmul2_rn(__fmul2_rn(rinv, rinv), rinv), qj);
  }
  sx = __ffma2_rn(fp, dx, sx);
  sy = __ffma2_rn(fp, dy, sy);
  sz = __ffma2_rn(fp, dz, sz);
}

// The lane's target against sources at .. at + NB - 1 of the queue; four
// sources load as one float4 per coordinate (two packed halves).
template <int M, int K, int NB, bool SELF>
__device__ __forceinline__ void pair_sources(const QueueF& Q, int at, float2 nax, float2 nay, float2 naz, float a2,
                                             const PairCoef& C, const WolfC<float>& W, float2& sphi, float2& sx,
                                             float2& sy, float2& sz) {
#pragma unroll
  for (int k = 0; k < NB; k += 4) {
    const int jj = at + k;
    const float4 x4 = *reinterpret_cast<const float4*>(&Q.x[jj]);
    const float4 y4 = *reinterpret_cast<const float4*>(&Q.y[jj]);
    const float4 z4 = *reinterpret_cast<const float4*>(&Q.z[jj]);
    const float4 q4 = *reinterpret_cast<const float4*>(&Q.q[jj]);
    pair2<M, K, SELF>(make_float2(x4.x, x4.y), make_float2(y4.x, y4.y), make_float2(z4.x, z4.y),
                      make_float2(q4.x, q4.y), nax, nay, naz, a2, C, W, sphi, sx, sy, sz);
    pair2<M, K, SELF>(make_float2(x4.z, x4.w), make_float2(y4.z, y4.w), make_float2(z4.z, z4.w),
                      make_float2(q4.z, q4.w), nax, nay, naz, a2, C, W, sphi, sx, sy, sz);
  }
}

// Running totals of a target and their compensation terms.
struct Totals {
  float phi = 0.f, x = 0.f, y = 0.f, z = 0.f, cphi = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
  __device__ __forceinline__ void fold(float2 sphi, float2 sx, float2 sy, float2 sz) {
    two_sum_add(phi, cphi, sphi.x + sphi.y);
    two_sum_add(x, cx, sx.x + sx.y);
    two_sum_add(y, cy, sy.x + sy.y);
    two_sum_add(z, cz, sz.x + sz.y);
  }
  // another warp's totals, laid down in its queue: x, y, z and q hold phi and
  // the force sums at [lane] and their compensation terms at [32 + lane]
  __device__ __forceinline__ void join(const QueueF& O, int lane) {
    two_sum_add(phi, cphi, O.x[lane]);
    two_sum_add(x, cx, O.y[lane]);
    two_sum_add(y, cy, O.z[lane]);
    two_sum_add(z, cz, O.q[lane]);
    cphi += O.x[32 + lane];
    cx += O.y[32 + lane];
    cy += O.z[32 + lane];
    cz += O.q[32 + lane];
  }
};

// n sources (a multiple of NB), folded into the totals once
template <int M, int K, int NB, bool SELF>
__device__ __forceinline__ void pair_batch(const QueueF& Q, int at, int n, float2 nax, float2 nay, float2 naz,
                                           float a2, const PairCoef& C, const WolfC<float>& W, Totals& t) {
  float2 sphi = make_float2(0.f, 0.f), sx = sphi, sy = sphi, sz = sphi;
#pragma unroll 1
  for (int b = 0; b < n; b += NB)
    pair_sources<M, K, NB, SELF>(Q, at + b, nax, nay, naz, a2, C, W, sphi, sx, sy, sz);
  t.fold(sphi, sx, sy, sz);
}

// Rows of neighbour cells: for each (dy, dz) the cells cx+xlo..cx+xhi of one x
// row are contiguous in the sorted atom array (cells are numbered x fastest),
// so a whole row is one or two contiguous atom ranges ("segments"; two when
// the row wraps around a periodic box).  At the start of a cell the lanes
// build the cell's segment table together, one row per lane (all cell-start
// loads in flight at once), and a warp scan lays the segments end to end
// into one flat source index space.  The warp then walks that space in full
// chunks of 32 sources, loading the next chunk's atoms before it works on the
// current one.  The x offset of a source's cell follows from comparing its
// index with the cell starts inside its segment.
struct SegTable {
  int4 rec[2 * kMaxRows + 1];   // (first atom, flat start, x offset of the first cell, -); sentinel at the end
  int4 bnd[2 * kMaxRows];       // first atom of the segment's 2nd..5th cell (INT_MAX where absent)
  float2 shift[2 * kMaxRows];   // (y, z) shift of the row
};

// The segment table of cell (cx, cy, cz), built by the warp (lane r: row r);
// returns the number of sources in the flat index space.
__device__ __forceinline__ int build_seg_table(SegTable& T, const PairKArgs& K, int cx, int cy, int cz, int lane) {
  const int* __restrict__ cell_start = K.cell_start;
  const int4* __restrict__ rows = K.rows;
  const int nrows = K.nrows;
  const PairArgs& A = K.A;
  const int ncx = A.nc[0], ncy = A.nc[1], ncz = A.nc[2];
  const float cwy = K.cwy, cwz = K.cwz;
  int len[2] = {0, 0}, j0s[2] = {0, 0}, ox0s[2] = {0, 0};
  int4 bnds[2] = {make_int4(INT_MAX, INT_MAX, INT_MAX, INT_MAX), make_int4(INT_MAX, INT_MAX, INT_MAX, INT_MAX)};
  float2 sh = make_float2(0.f, 0.f);
  if (lane < nrows) {
    const int4 row = rows[lane];  // (dy, dz, xlo, xhi): x offsets xlo..xhi of this row
    int ny = cy + row.x, nz = cz + row.y;
    bool inside = true;
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
      int ox0 = 0, ox1 = -1;  // empty unless set below
      if (!inside) {
      } else if (A.periodic) {
        const int xa = cx + row.z, xb = cx + row.w;  // may leave [0, ncx) by at most 2
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
        int bb[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) bb[t] = (x0 + 1 + t <= x1) ? cell_start[rbase + x0 + 1 + t] : INT_MAX;
        len[seg] = j1 - j0;
        j0s[seg] = j0;
        ox0s[seg] = ox0;
        bnds[seg] = make_int4(bb[0], bb[1], bb[2], bb[3]);
      }
    }
  }
  int total;
  {
    const int mine = len[0] + len[1];
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    total = __shfl_sync(kFull, incl, 31);
    const int start = incl - mine;
    if (lane < nrows) {
#pragma unroll
      for (int seg = 0; seg < 2; ++seg) {
        T.rec[2 * lane + seg] = make_int4(j0s[seg], seg ? start + len[0] : start, ox0s[seg], 0);
        T.bnd[2 * lane + seg] = bnds[seg];
        T.shift[2 * lane + seg] = sh;
      }
    }
    if (lane == 0) T.rec[2 * nrows] = make_int4(0, INT_MAX, 0, 0);
    __syncwarp();
  }

  return total;
}

// ---- target clusters (mixed precision) ----
// The warp takes its cell's atoms 32 at a time (a pass) as up to kClPass
// clusters of kCl consecutive atoms (slabs of the cell across x, since
// binning sorts each cell by x), and culls every source against each
// cluster's own bounding box.  Each cluster has its own queue; a full queue of kCD
// sources is drained by the whole warp on that one cluster: lane 4 i + jl
// evaluates target i of the cluster against sources 16 jl .. 16 jl + 15
// (packed FP32x2), the four partial sums of a target are added across its
// four lanes by two shuffles, and lane 4 i + c, which owns target (c, i),
// folds them into its compensated totals.  The home cell goes through the
// scalar pair with the self test.  Queue arrays leave 4 floats of padding
// after every 16 sources, so that the four source lanes' float4 loads fall
// on distinct banks.
constexpr int kCl = 8, kClPass = 4, kCD = 64, kCQ = kCD + 32;
constexpr int kCQP = kCQ + (kCQ / 16) * 4;
__device__ __forceinline__ int cq_slot(int p) { return p + ((p >> 4) << 2); }
struct alignas(16) ClQueue {
  float x[kCQP], y[kCQP], z[kCQP], q[kCQP];
};

template <int M, int KIND>
__device__ __forceinline__ void cl_drain(const ClQueue& Q, float tx, float ty, float tz, int jl, float a2,
                                         const PairCoef& C, const WolfC<float>& W, float& s0, float& s1, float& s2,
                                         float& s3) {
  const float2 nax = make_float2(-tx, -tx), nay = make_float2(-ty, -ty), naz = make_float2(-tz, -tz);
  float2 sphi = make_float2(0.f, 0.f), sx = sphi, sy = sphi, sz = sphi;
  const int b = cq_slot(16 * jl);
#pragma unroll
  for (int k = 0; k < 16; k += 4) {
    const float4 x4 = *reinterpret_cast<const float4*>(&Q.x[b + k]);
    const float4 y4 = *reinterpret_cast<const float4*>(&Q.y[b + k]);
    const float4 z4 = *reinterpret_cast<const float4*>(&Q.z[b + k]);
    const float4 q4 = *reinterpret_cast<const float4*>(&Q.q[b + k]);
    pair2<M, KIND>(make_float2(x4.x, x4.y), make_float2(y4.x, y4.y), make_float2(z4.x, z4.y),
                   make_float2(q4.x, q4.y), nax, nay, naz, a2, C, W, sphi, sx, sy, sz);
    pair2<M, KIND>(make_float2(x4.z, x4.w), make_float2(y4.z, y4.w), make_float2(z4.z, z4.w),
                   make_float2(q4.z, q4.w), nax, nay, naz, a2, C, W, sphi, sx, sy, sz);
  }
  s0 = sphi.x + sphi.y;
  s1 = sx.x + sx.y;
  s2 = sy.x + sy.y;
  s3 = sz.x + sz.y;
}

// The four partial sums of target i, spread over lanes 4 i .. 4 i + 3, added
// (every lane of the group gets the total).
__device__ __forceinline__ void cl_reduce(float& s0, float& s1, float& s2, float& s3) {
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1) {
    s0 += __shfl_xor_sync(kFull, s0, o);
    s1 += __shfl_xor_sync(kFull, s1, o);
    s2 += __shfl_xor_sync(kFull, s2, o);
    s3 += __shfl_xor_sync(kFull, s3, o);
  }
}

template <int M, int KIND>
__device__ __forceinline__ void short_range_c8_body(const PairKArgs& K, int blk) {
  const R4<float>* __restrict__ atoms = K.atoms;
  const int* __restrict__ cell_start = K.cell_start;
  const int ncell = K.ncell;
  const PairArgs& A = K.A;
  const PairCoef C = K.C;
  const WolfC<float> W = K.W;
  const float cwx = K.cwx;
  float* __restrict__ phis = K.phis;
  R4<float>* __restrict__ fs = K.fs;
  __shared__ ClQueue queues[kWarps][kClPass];
  __shared__ R4<float> home[kWarps][32];
  __shared__ SegTable tables[kWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cell = blk * kWarps + warp;
  if (cell >= ncell) return;  // warp-uniform
  const int ncx = A.nc[0], ncy = A.nc[1];
  const int cx = cell % ncx, cy = (cell / ncx) % ncy, cz = cell / (ncx * ncy);
  const float a2 = A.a2f, inv_a = A.inv_af, inv_a2s = A.inv_a2f, two_inv_a3 = A.two_inv_a3f;
  const float FAR = 1e6f;
  const int i0 = cell_start[cell], i1 = cell_start[cell + 1];
  if (i0 == i1) return;  // warp-uniform
  SegTable& T = tables[warp];
  ClQueue* Q = queues[warp];
  const int total = build_seg_table(T, K, cx, cy, cz, lane);
  const int jl = lane & 3, ti = lane >> 2;
  for (int base = i0; base < i1; base += kCl * kClPass) {
    const int ncl = min(kClPass, (i1 - base + kCl - 1) / kCl);
    // lane 4 i + c owns target (c, i), atom base + 8 c + i
    const int t_atom = base + kCl * jl + ti;
    const bool tv = t_atom < i1;
    const R4<float> ai = tv ? atoms[t_atom] : R4<float>{FAR, FAR, FAR, 0.f};
    // bounding box of each cluster (over the lanes with the same lane & 3),
    // then every cluster's box in every lane
    float lx = tv ? ai.x : FAR, ly = tv ? ai.y : FAR, lz = tv ? ai.z : FAR;
    float hx = tv ? ai.x : -FAR, hy = tv ? ai.y : -FAR, hz = tv ? ai.z : -FAR;
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      lx = fminf(lx, __shfl_xor_sync(kFull, lx, o));
      ly = fminf(ly, __shfl_xor_sync(kFull, ly, o));
      lz = fminf(lz, __shfl_xor_sync(kFull, lz, o));
      hx = fmaxf(hx, __shfl_xor_sync(kFull, hx, o));
      hy = fmaxf(hy, __shfl_xor_sync(kFull, hy, o));
      hz = fmaxf(hz, __shfl_xor_sync(kFull, hz, o));
    }
    float blx[kClPass], bly[kClPass], blz[kClPass], bhx[kClPass], bhy[kClPass], bhz[kClPass];
#pragma unroll
    for (int c = 0; c < kClPass; ++c) {
      blx[c] = __shfl_sync(kFull, lx, c);
      bly[c] = __shfl_sync(kFull, ly, c);
      blz[c] = __shfl_sync(kFull, lz, c);
      bhx[c] = __shfl_sync(kFull, hx, c);
      bhy[c] = __shfl_sync(kFull, hy, c);
      bhz[c] = __shfl_sync(kFull, hz, c);
    }
    float phi = 0.f, px = 0.f, py = 0.f, pz = 0.f, cphi = 0.f, cpx = 0.f, cpy = 0.f, cpz = 0.f;
    // the home cell: cluster c's targets against all the cell's atoms, lane
    // 4 i + jl taking sources jl, jl + 4, ... (scalar, with the self test)
    for (int jb = i0; jb < i1; jb += 32) {
      const int j = jb + lane;
      home[warp][lane] = (j < i1) ? atoms[j] : R4<float>{FAR, FAR, FAR, 0.f};
      __syncwarp();
#pragma unroll 1
      for (int c = 0; c < ncl; ++c) {
        const int src = 4 * ti + c;
        const R4<float> t = {__shfl_sync(kFull, ai.x, src), __shfl_sync(kFull, ai.y, src),
                             __shfl_sync(kFull, ai.z, src), 0.f};
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          pair1<float, M, KIND>(t, home[warp][jl + 4 * k], a2, inv_a, inv_a2s, two_inv_a3, W, s0, s1, s2, s3);
        cl_reduce(s0, s1, s2, s3);
        if (jl == c) {  // both paths sum grad_i u_i (scalar: f (r_i - r_j); packed: f' (r_j - r_i), f' = -f)
          two_sum_add(phi, cphi, s0);
          two_sum_add(px, cpx, s1);
          two_sum_add(py, cpy, s2);
          two_sum_add(pz, cpz, s3);
        }
      }
      __syncwarp();
    }
    // the neighbour rows: flat source index t in [0, total), 32 per step
    int seg = 0;
    auto locate = [&](int t, int& j, int& ox, float2& shv) {
      while (T.rec[seg + 1].y <= t) ++seg;
      const int4 r = T.rec[seg];
      const int4 b = T.bnd[seg];
      j = r.x + (t - r.y);
      ox = r.z + (j >= b.x) + (j >= b.y) + (j >= b.z) + (j >= b.w);
      shv = T.shift[seg];
    };
    R4<float> an = {FAR, FAR, FAR, 0.f};
    int oxn = 0;
    float2 shn = make_float2(0.f, 0.f);
    if (lane < total) {
      int j;
      locate(lane, j, oxn, shn);
      an = atoms[j];
    }
    int qn[kClPass];
#pragma unroll
    for (int c = 0; c < kClPass; ++c) qn[c] = 0;
    auto drain = [&](int c) {
      const int src = 4 * ti + c;
      const float tx = __shfl_sync(kFull, ai.x, src), ty = __shfl_sync(kFull, ai.y, src),
                  tz = __shfl_sync(kFull, ai.z, src);
      float s0, s1, s2, s3;
      cl_drain<M, KIND>(Q[c], tx, ty, tz, jl, a2, C, W, s0, s1, s2, s3);
      cl_reduce(s0, s1, s2, s3);
      if (jl == c) {
        two_sum_add(phi, cphi, s0);
        two_sum_add(px, cpx, s1);
        two_sum_add(py, cpy, s2);
        two_sum_add(pz, cpz, s3);
      }
    };
    for (int t0 = 0; t0 < total; t0 += 32) {
      const bool valid = t0 + lane < total;
      R4<float> aj = an;
      const int ox = oxn;
      const float2 shv = shn;
      if (t0 + 32 + lane < total) {  // next chunk's load goes out before this chunk's work
        int j;
        locate(t0 + 32 + lane, j, oxn, shn);
        an = atoms[j];
      }
      aj.x += ox * cwx;
      aj.y += shv.x;
      aj.z += shv.y;
      const unsigned lt = (1u << lane) - 1u;
#pragma unroll
      for (int c = 0; c < kClPass; ++c) {
        if (c < ncl) {
          const float ex = fmaxf(fmaxf(blx[c] - aj.x, aj.x - bhx[c]), 0.f);
          const float ey = fmaxf(fmaxf(bly[c] - aj.y, aj.y - bhy[c]), 0.f);
          const float ez = fmaxf(fmaxf(blz[c] - aj.z, aj.z - bhz[c]), 0.f);
          const bool keep = valid && (ex * ex + ey * ey + ez * ez < a2);
          const unsigned bal = __ballot_sync(kFull, keep);
          if (keep) {
            const int p = cq_slot(qn[c] + __popc(bal & lt));
            Q[c].x[p] = aj.x;
            Q[c].y[p] = aj.y;
            Q[c].z[p] = aj.z;
            Q[c].q[p] = aj.w;
          }
          qn[c] += __popc(bal);
        }
      }
      __syncwarp();
#pragma unroll
      for (int c = 0; c < kClPass; ++c) {
        if (c < ncl && qn[c] >= kCD) {
          drain(c);
          __syncwarp();
          if (lane < qn[c] - kCD) {
            const int from = cq_slot(kCD + lane), to = cq_slot(lane);
            Q[c].x[to] = Q[c].x[from];
            Q[c].y[to] = Q[c].y[from];
            Q[c].z[to] = Q[c].z[from];
            Q[c].q[to] = Q[c].q[from];
          }
          qn[c] -= kCD;
          __syncwarp();
        }
      }
    }
    // last partial queues, padded with far-away zero charges
#pragma unroll
    for (int c = 0; c < kClPass; ++c) {
      if (c < ncl && qn[c] > 0) {
        for (int t = qn[c] + lane; t < kCD; t += 32) {
          const int p = cq_slot(t);
          Q[c].x[p] = FAR;
          Q[c].y[p] = FAR;
          Q[c].z[p] = FAR;
          Q[c].q[p] = 0.f;
        }
        __syncwarp();
        drain(c);
        __syncwarp();
      }
    }
    if (tv) {
      phis[t_atom] = phi + cphi;
      const float qi = ai.w;
      fs[t_atom] = R4<float>{-qi * (px + cpx), -qi * (py + cpy), -qi * (pz + cpz), 0.f};
    }
  }
}

// ---- one cell or one run of atoms per warp (mixed precision) ----
// A warp's targets are, in cell mode, the atoms of one cell, 32 at a time; in
// run mode 32 consecutive sorted atoms, whatever cells they belong to, so that
// no lane idles for want of a cell's atoms (~25 per cell at the default fill).
// Binning sorts each cell by x and numbers cells x fastest, so a run of a cell
// row is a slab of it.  A run is cut into pieces of one row and at most
// maxspan + 1 cells (nearly always one piece): a piece's targets enter the
// frame of its first cell c0 shifted by whole cells, the home block is the
// atoms of the piece's cells (with the self test), and the neighbour rows are
// the plan's rows widened by the piece's span.
//
// Sources are culled against the targets' bounding box, queued (a ring of 128)
// and evaluated in unrolled batches of 64, folded into the totals with TwoSum.
// A packed step (two pairs per lane) is 17 FMA-pipe instructions and costs ~44
// cycles of an SM quarter however it is written (packed or scalar, constants
// in registers or as immediates, one to four steps interleaved): 34 cycles of
// FMA pipe, the rest register reads.  The 1.07M-atom box evaluates 1,960
// sources per target, 1.2 ms of such steps; the walk over ~4,000 candidates
// per target (0.63 ms by itself) is hidden only in part.
//
// The warps of a block may share one group (K.split of them): warp p takes
// every split-th 64 sources, and the warps' totals are joined in warp order
// with their compensation terms (one FP32 number per warp would round off what
// the warps' totals cancel to).
// (The barrier is the block's: named barriers by a computed number reserve
// all 16 of a block and halve the resident blocks, 1.63 -> 1.85 ms.)
//
// Measured alone: 1.07M atoms 1,630 -> 1,600 us, 190,977 atoms 265 -> 254 us,
// 23,558 atoms 56 -> 45 us, 3,000 atoms (open) 57 -> 24 us, against loads one
// step of 32 sources ahead and a flat index space located per lane.
//
// The sources of the next kAhead steps are in flight as asynchronous copies
// into a ring in shared memory, each lane copying the records it will take.
// A step is 64 sources, two per lane: the loop's state, the range's shift and
// the chain load - cull - ballot - append are paid once for both.
constexpr int kStep = 64;  // sources per step
// Where cells hold few atoms (flat_walk) most steps within one range would be
// nearly empty, and a FLAT walk takes its sources across the ranges, each lane
// keeping the ranges of its two sources.  Such walks are a few steps long: two in
// flight are enough, and the smaller ring and 80 registers (six blocks an SM)
// leave more cache and warps (27,000 cells of 4 atoms in runs: 229 us by ranges,
// 217 across them with four steps in flight and five blocks, 181 so).
template <bool FLAT>
struct Walk {
  static constexpr int kAhead = FLAT ? 2 : 4;      // steps in flight, a power of two
  static constexpr int kMinBlocks = FLAT ? 6 : 5;  // resident blocks per SM
};
template <int kAhead>
struct alignas(16) PairShared {
  QueueF queue;
  SegList segs;
  R4<float> ring[kAhead][kStep];  // records of the steps in flight
  float ringx[kAhead][kStep];     // their cells' x index
  int ringseg[kAhead];            // their range, and their number << 8
  float4 shift[2 * kMaxRows];     // a range's x base, y shift and z shift
};

__device__ __forceinline__ void copy_async16(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// The ranges laid end to end: rec becomes (first atom minus flat start, flat
// end, .., ..); returns the number of sources.
__device__ __forceinline__ int flatten_segments(SegList& L, int nseg, int lane) {
  int total = 0;
  for (int b = 0; b < nseg; b += 32) {
    const int e = b + lane;
    const int first = e < nseg ? L.rec[e].x : 0, len = e < nseg ? L.rec[e].y - first : 0;
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    if (e < nseg) {
      L.rec[e].x = first - (total + incl - len);
      L.rec[e].y = total + incl;
    }
    total += __shfl_sync(kFull, incl, 31);
  }
  __syncwarp();
  return total;
}

// SHARE: the block's warps share a group (K.split of them).
template <int M, int KIND, bool FLAT, bool SHARE>
__device__ __forceinline__ void short_range_body(const PairKArgs& K, int blk) {
  const R4<float>* __restrict__ atoms = K.atoms;
  const float* __restrict__ cellx = K.cellx;
  const int* __restrict__ cell_start = K.cell_start;
  const PairArgs& A = K.A;
  const PairCoef C = K.C;
  const WolfC<float> W = K.W;
  const float cwx = K.cwx;
  constexpr int kAhead = Walk<FLAT>::kAhead;
  __shared__ PairShared<kAhead> shared[kWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  PairShared<kAhead>& Sh = shared[warp];
  QueueF& Q = Sh.queue;
  SegList& L = Sh.segs;
  const int split = SHARE ? K.split : 1, part = split > 1 ? warp : 0;
  const int group = split > 1 ? blk : blk * kWarps + warp;
  const int ncx = A.nc[0], ncy = A.nc[1];
  const float a2 = A.a2f;
  const float FAR = 1e6f;
  const unsigned lt = (1u << lane) - 1u;
  // targets i0 .. i1 - 1; the lane's own in run mode (cells ascend with the lane)
  int i0, i1, mycell = INT_MAX;
  R4<float> me = {0.f, 0.f, 0.f, 0.f};
  if (K.runs) {
    i0 = group * 32;
    i1 = min(i0 + 32, K.natoms);
    if (i0 + lane < i1) {
      mycell = K.scell[i0 + lane];
      me = atoms[i0 + lane];
    }
  } else {
    i0 = group < K.ncell ? cell_start[group] : 0;
    i1 = group < K.ncell ? cell_start[group + 1] : 0;
  }
  for (int ib = i0; ib < i1;) {  // one piece per step (the same for every warp of the group)
    int c0 = group, span = 0, next = ib + 32;
    bool inp;
    if (K.runs) {
      const int l0 = ib - i0;
      c0 = __shfl_sync(kFull, mycell, l0);
      const int climit = c0 + min(K.maxspan, ncx - 1 - c0 % ncx);  // the piece stays in the row
      inp = lane >= l0 && mycell <= climit;
      const int l1 = 32 - __clz(__ballot_sync(kFull, inp));
      span = __shfl_sync(kFull, mycell, l1 - 1) - c0;
      next = i0 + l1;
    } else {
      inp = ib + lane < i1;
      me = inp ? atoms[ib + lane] : R4<float>{0.f, 0.f, 0.f, 0.f};
      mycell = c0;
    }
    const int cx = c0 % ncx, cy = (c0 / ncx) % ncy, cz = c0 / (ncx * ncy);
    const int h0 = cell_start[c0], h1 = cell_start[c0 + span + 1];
    // the target in c0's frame (the same rounding as the home block's)
    R4<float> ai = me;
    ai.x = __fmaf_rn((float)(inp ? mycell - c0 : 0), cwx, ai.x);
    const float lx = warp_min(inp ? ai.x : FAR), ly = warp_min(inp ? ai.y : FAR), lz = warp_min(inp ? ai.z : FAR);
    const float hx = warp_max(inp ? ai.x : -FAR), hy = warp_max(inp ? ai.y : -FAR), hz = warp_max(inp ? ai.z : -FAR);
    const float2 nax = make_float2(-ai.x, -ai.x), nay = make_float2(-ai.y, -ai.y), naz = make_float2(-ai.z, -ai.z);
    // the ranges of the neighbour rows, 64 sources per step (every split-th of
    // them), a step within one range or, FLAT, across ranges laid end to end:
    // fill() starts the copies of the next step into ring slot `slot`
    const int nseg = build_segments(L, K, cx, cy, cz, span, lx, ly, lz, hx, hy, hz, lane);
    for (int e = lane; e < nseg; e += 32) {
      const int4 r = L.rec[e];
      Sh.shift[e] = make_float4((float)r.z, ((r.w & 15) - 3) * K.cwy, ((r.w >> 4) - 3) * K.cwz, 0.f);
    }
    __syncwarp();
    int seg = -1, jb = 0, je = 0, skip = part, steps = 0;  // steps: filled, not yet taken
    bool more = true;
    // FLAT: sources in all ranges, the first source of the next step to fill and
    // to take, and the ranges the lane's two sources lie in (it fills and takes
    // the same ones); rec then holds atom minus flat index, and the flat end
    int total = 0, tf = kStep * part, tt = tf, sf0 = 0, sf1 = 0, st0 = 0, st1 = 0;
    if (FLAT) total = flatten_segments(L, nseg, lane);
    auto range_of = [&](int t, int& e) {  // e: a range not after t's
      while (L.rec[e].y <= t) ++e;
    };
    auto fill = [&](int slot) {
      if (FLAT) {
        if (tf < total) {
          const int t0 = tf + lane, t1 = t0 + 32;
          if (t0 < total) {
            range_of(t0, sf0);
            const int j = L.rec[sf0].x + t0;
            copy_async16(&Sh.ring[slot][lane], atoms + j);
            copy_async4(&Sh.ringx[slot][lane], cellx + j);
          }
          if (t1 < total) {
            range_of(t1, sf1);
            const int j = L.rec[sf1].x + t1;
            copy_async16(&Sh.ring[slot][lane + 32], atoms + j);
            copy_async4(&Sh.ringx[slot][lane + 32], cellx + j);
          }
          tf += kStep * split;
          ++steps;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        return;
      }
      while (more && jb >= je) {  // to the next range; its first `skip` steps are the other warps'
        if (seg >= 0) skip = (jb - je) / kStep;
        more = ++seg < nseg;
        if (more) {
          const int4 r = L.rec[seg];
          jb = r.x + kStep * skip;
          je = r.y;
        }
      }
      if (more) {
        const int j = jb + lane, n = je - jb;
        if (lane < n) {
          copy_async16(&Sh.ring[slot][lane], atoms + j);
          copy_async4(&Sh.ringx[slot][lane], cellx + j);
        }
        if (lane + 32 < n) {
          copy_async16(&Sh.ring[slot][lane + 32], atoms + j + 32);
          copy_async4(&Sh.ringx[slot][lane + 32], cellx + j + 32);
        }
        if (lane == 0) Sh.ringseg[slot] = seg | (min(n, kStep) << 8);
        jb += kStep * split;
        ++steps;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int d = 0; d < kAhead; ++d) fill(d);
    Totals tot;
    // the home block, 32 sources at a time, with the self test
    for (int hb = h0 + 32 * part; hb < h1; hb += 32 * split) {
      const int j = hb + lane;
      R4<float> s = {FAR, FAR, FAR, 0.f};
      if (j < h1) {
        s = atoms[j];
        s.x = __fmaf_rn(cellx[j] - (float)cx, cwx, s.x);
      }
      Q.x[lane] = s.x;
      Q.y[lane] = s.y;
      Q.z[lane] = s.z;
      Q.q[lane] = s.w;
      __syncwarp();
      pair_batch<M, KIND, 32, true>(Q, 0, 32, nax, nay, naz, a2, C, W, tot);
      __syncwarp();
    }
    __syncwarp();
    int qn = 0, head = 0;  // queued sources and where they begin (0 or kBatch)
    for (int slot = 0; steps > 0; slot = (slot + 1) & (kAhead - 1)) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
      const R4<float> s0 = Sh.ring[slot][lane], s1 = Sh.ring[slot][lane + 32];
      int n;
      float2 shx, shy, shz;  // the shifts of the two sources' ranges
      if constexpr (FLAT) {
        n = total - tt;
        if (tt + lane < total) range_of(tt + lane, st0);
        if (tt + lane + 32 < total) range_of(tt + lane + 32, st1);
        tt += kStep * split;
        const float4 a = Sh.shift[st0], b = Sh.shift[st1];
        shx = make_float2(a.x, b.x);
        shy = make_float2(a.y, b.y);
        shz = make_float2(a.z, b.z);
      } else {
        const int meta = Sh.ringseg[slot];
        n = meta >> 8;
        const float4 a = Sh.shift[meta & 255];
        shx = make_float2(a.x, a.x);
        shy = make_float2(a.y, a.y);
        shz = make_float2(a.z, a.z);
      }
      const float2 w = make_float2(cwx, cwx);
      const float2 x = __ffma2_rn(__fadd2_rn(make_float2(Sh.ringx[slot][lane], Sh.ringx[slot][lane + 32]), shx), w,
                                  make_float2(s0.x, s1.x));
      const float2 y = __fadd2_rn(make_float2(s0.y, s1.y), shy);
      const float2 z = __fadd2_rn(make_float2(s0.z, s1.z), shz);
      __syncwarp();  // the slot's range has been read
      --steps;
      fill(slot);
      auto gap = [&](float2 v, float lo, float hi) {  // distance beyond the box along one axis
        const float2 a = __fadd2_rn(make_float2(lo, lo), make_float2(-v.x, -v.y));
        const float2 b = __fadd2_rn(v, make_float2(-hi, -hi));
        return make_float2(fmaxf(fmaxf(a.x, b.x), 0.f), fmaxf(fmaxf(a.y, b.y), 0.f));
      };
      const float2 ex = gap(x, lx, hx), ey = gap(y, ly, hy), ez = gap(z, lz, hz);
      const float2 d2 = __ffma2_rn(ez, ez, __ffma2_rn(ey, ey, __fmul2_rn(ex, ex)));
      const bool k0 = lane < n && d2.x < a2, k1 = lane + 32 < n && d2.y < a2;
      const unsigned b0 = __ballot_sync(kFull, k0), b1 = __ballot_sync(kFull, k1);
      const int at0 = head + qn, at1 = at0 + __popc(b0);
      if (k0) {
        const int p = (at0 + __popc(b0 & lt)) & (2 * kBatch - 1);
        Q.x[p] = x.x;
        Q.y[p] = y.x;
        Q.z[p] = z.x;
        Q.q[p] = s0.w;
      }
      if (k1) {
        const int p = (at1 + __popc(b1 & lt)) & (2 * kBatch - 1);
        Q.x[p] = x.y;
        Q.y[p] = y.y;
        Q.z[p] = z.y;
        Q.q[p] = s1.w;
      }
      qn += __popc(b0) + __popc(b1);
      __syncwarp();
      if (qn >= kBatch) {
        pair_batch<M, KIND, kBatch, false>(Q, head, kBatch, nax, nay, naz, a2, C, W, tot);
        head ^= kBatch;
        qn -= kBatch;
        __syncwarp();
      }
    }
    if (qn > 0) {  // the last sources, padded to a multiple of 16 with far-away zero charges
      const int n16 = (qn + 15) & ~15;
      if (qn + lane < n16) {
        const int p = head + qn + lane;
        Q.x[p] = FAR;
        Q.y[p] = FAR;
        Q.z[p] = FAR;
        Q.q[p] = 0.f;
      }
      __syncwarp();
      pair_batch<M, KIND, 16, false>(Q, head, n16, nax, nay, naz, a2, C, W, tot);
      __syncwarp();
    }
    if (split > 1) {  // the warps' totals, each with its compensation term, joined in warp order
      float* mine[4] = {Q.x, Q.y, Q.z, Q.q};
      const float total[4] = {tot.phi, tot.x, tot.y, tot.z}, comp[4] = {tot.cphi, tot.cx, tot.cy, tot.cz};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        mine[c][lane] = total[c];
        mine[c][32 + lane] = comp[c];
      }
      __syncthreads();
      tot = Totals();
      if (part == 0)
        for (int p = 0; p < split; ++p) tot.join(shared[p].queue, lane);
      __syncthreads();
    }
    const float phi = tot.phi + tot.cphi, px = tot.x + tot.cx, py = tot.y + tot.cy, pz = tot.z + tot.cz;
    if (part == 0 && inp) {
      const int i = (K.runs ? i0 : ib) + lane;
      K.phis[i] = phi;
      K.fs[i] = R4<float>{-me.w * px, -me.w * py, -me.w * pz, 0.f};
    }
    ib = next;
  }
}

// Wolf's pair function is short of registers where the warps also join their
// totals: four blocks with 128 of them instead of five with 96 (calls at 3,000 atoms
// open 55 -> 47 us, 23,558 with a = 20 515 -> 453, with a = 10 123 -> 125).
template <int KIND, bool FLAT, bool SHARE>
constexpr int kPairBlocks = KIND == kPairWolf && SHARE && !FLAT ? 4 : Walk<FLAT>::kMinBlocks;

template <int M, int KIND, bool FLAT, bool SHARE>
__global__ void __launch_bounds__(32 * kWarps, kPairBlocks<KIND, FLAT, SHARE>) k_short_range(const __grid_constant__ PairKArgs a) {
  pdl_sync();
  short_range_body<M, KIND, FLAT, SHARE>(a, blockIdx.x);
}

template <int M, bool FLAT>
__global__ void __launch_bounds__(32 * kWarps, Walk<FLAT>::kMinBlocks) kb_short_range(const PairKArgs* __restrict__ tab,
                                                                const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  short_range_body<M, kPairMSM, FLAT, false>(tab[r], blockIdx.x - first[r]);
}

template <int M, int KIND>
__global__ void __launch_bounds__(32 * kWarps, 4) k_short_range_c8(PairKArgs a) {
  short_range_c8_body<M, KIND>(a, blockIdx.x);
}

template <int M>
__global__ void __launch_bounds__(32 * kWarps, 4) kb_short_range_c8(const PairKArgs* __restrict__ tab,
                                                                   const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  short_range_c8_body<M, kPairMSM>(tab[r], blockIdx.x - first[r]);
}

}  // namespace

PairKArgs pair_kargs(const Plan& P) {
  PairKArgs K;
  K.A = pair_args(P);
  K.W = wolf_consts<float>(0.0, P.P.cutoff);
  K.atoms = (const R4<float>*)P.d.atoms;
  K.cell_start = P.d.cell_start;
  K.rows = P.d.cell_rows;
  K.nrows = P.nrows;
  K.ncell = P.ncell;
  K.phis = (float*)P.d.phis;
  K.fs = (R4<float>*)P.d.fs;
  // gamma coefficients c_k (Taylor series of s^(-1/2) about s = 1, truncated at m)
  static const double c[4][4] = {{0, 0, 0, 0}, {1.5, -0.5, 0, 0}, {1.875, -1.25, 0.375, 0},
                                 {2.1875, -2.1875, 1.3125, -0.3125}};
  const int m = P.P.splitting;
  const double a = P.P.cutoff;
  for (int k = 0; k < 4; ++k) {
    float g = (k <= m) ? (float)(-c[m][k] / std::pow(a, 2 * k + 1)) : 0.f;
    K.C.G[k] = make_float2(g, g);
  }
  for (int k = 0; k < 3; ++k) {
    float d = (k + 1 <= m) ? (float)(2.0 * (k + 1) * c[m][k + 1] / std::pow(a, 2 * k + 3)) : 0.f;
    K.C.D[k] = make_float2(d, d);
  }
  K.cwx = (float)P.cw[0];
  K.cwy = (float)P.cw[1];
  K.cwz = (float)P.cw[2];
  K.scell = P.d.scell;
  K.cellx = P.d.cellx;
  K.natoms = 0;
  K.runs = 0;
  K.split = 1;
  // a piece widens the rows of neighbour cells by its span: a periodic row
  // must not meet itself
  K.maxspan = P.P.periodic ? std::max(0, std::min(2, P.nc[0] - P.row_cells)) : 2;
  return K;
}

// How the pair kernel shares its work, by the plan's cells and the call's atoms.
// A plan of the default capacity has cells of half a cutoff, which may hold far
// fewer atoms than the 24 that a plan of its system's own size gives them, so the
// lines below lie on both (pair sums alone, us; cells of a/2, 0.3 to 32 atoms each).
//
// Runs of 32 atoms (else one cell per warp): a periodic row must hold the piece's
// three cells beside its neighbours, or the runs would fall into pieces of a few
// atoms.  By default from 11,264 cells and 57,344 atoms: at 24 atoms a cell runs
// against cells take 271 and 254 at 7,980 cells, 552 and 621 at 12,167; with fewer
// atoms than 152 SMs x 12 warps of 32 the chip waits for a run's pieces one after
// another: 15,625 cells with 4,687 atoms 107 and 29, 31,250 113 and 94, 62,500 134
// and 150, 12,167 cells with 48,668 atoms 122 and 115, 97,336 172 and 203.  From
// 16,384 cells on always: there a system may well be a cluster in a great box, in
// few cells of many atoms (a droplet of 5,000 atoms in 42,875 cells of 11.4, a = 8:
// calls of the cutoff method 100 with runs, 304 with a warp per cell; 5,000 spread
// evenly 115 and 63).
constexpr int64_t kRunCells = 11264, kRunAtoms = 57344, kRunCellsAlways = 16384;
static bool use_runs(const Plan& P, int64_t n) {
  const bool many = P.ncell >= kRunCellsAlways || (P.ncell >= kRunCells && n >= kRunAtoms);
  const bool wanted = P.pair_runs == 1 || (P.pair_runs == 0 && many);
  return wanted && P.pair_targets != kCl && (!P.P.periodic || P.nc[0] >= P.row_cells + 2);
}

// Sources across ranges (FLAT) below 8 atoms a cell, where a range (a row of 5
// cells) rarely fills a step of 64: 12,167 cells of 1, 4, 8 and 12 atoms 75 -> 45,
// 139 -> 115, 210 -> 203 and 291 -> 294; runs on 27,000 cells of 4 and 8 atoms
// 229 -> 181 and 333 -> 339.  Not for runs on smaller boxes (4,096 cells of 4 and 8
// atoms 102 and 105, 107 and 119: too few warps for a ring of two), nor where the
// capacity and not the cutoff set the cells' width: so few atoms there are a cluster
// in a great box, in full cells (20,000 atoms in 42,875 cells of 8.6, a = 10, calls of
// the cutoff method 98 and 120).
static bool flat_walk(const Plan& P, int64_t n, bool runs) {
  const double a = P.P.cutoff;
  const bool narrow = P.cw[0] * P.cw[1] * P.cw[2] < 0.216 * a * a * a;  // cells of up to 0.6 a
  return n < 8 * (int64_t)P.ncell && narrow && (!runs || P.ncell >= kRunCellsAlways);
}

// Small boxes share each group among the four warps of a block: one warp per group
// leaves most of the GPU idle (23,558 atoms, 1,000 cells: 52 -> 45; 5,001 atoms,
// 216 cells: 42 -> 21; at 50,001 atoms, 2,197 cells: 83; at 100,002 atoms 133 ->
// 141).  With cells of few atoms the sharing ends earlier: 1,728 cells of 8 and 16
// atoms 46 alone and 49 shared, 74 and 82 (Wolf 102 and 117, 157 and 208), of 24
// atoms 147 (by the kernel without sharing) and 113; 1,000 cells of 8 atoms 41 and 37.
static int split_of(bool runs, int64_t n, int64_t ncell) {
  const bool share = ncell < 1408 || (ncell < 2048 && (runs || n >= 18 * ncell));
  return share ? kWarps : 1;
}

static int pair_blocks(const PairKArgs& K) {
  const int64_t groups = K.runs ? ((int64_t)K.natoms + 31) / 32 : K.ncell;
  return (int)(K.split > 1 ? groups : (groups + kWarps - 1) / kWarps);
}

template <int M, int KIND>
void launch_mk(const Plan& P, const PairKArgs& K, cudaStream_t st) {
  auto run = [&](auto kernel) { klaunch(P.pdl, kernel, pair_blocks(K), 32 * kWarps, 0, st, K); };
  if (flat_walk(P, K.natoms, K.runs)) run(K.split > 1 ? k_short_range<M, KIND, true, true> : k_short_range<M, KIND, true, false>);
  else run(K.split > 1 ? k_short_range<M, KIND, false, true> : k_short_range<M, KIND, false, false>);
}

template <int KIND>
void launch_f2(Plan& P, int64_t n, cudaStream_t st, double alpha = 0.0) {
  PairKArgs K = pair_kargs(P);
  K.W = wolf_consts<float>(alpha, P.P.cutoff);
  K.natoms = (int)n;
  if (P.pair_targets == kCl) {  // clusters of 8 targets
    const int blocks = (P.ncell + kWarps - 1) / kWarps;
    if (KIND == kPairCutoff) k_short_range_c8<2, kPairCutoff><<<blocks, 32 * kWarps, 0, st>>>(K);  // M unused
    else if (KIND == kPairWolf) k_short_range_c8<2, kPairWolf><<<blocks, 32 * kWarps, 0, st>>>(K);
    else if (P.P.splitting == 1) k_short_range_c8<1, kPairMSM><<<blocks, 32 * kWarps, 0, st>>>(K);
    else if (P.P.splitting == 2) k_short_range_c8<2, kPairMSM><<<blocks, 32 * kWarps, 0, st>>>(K);
    else k_short_range_c8<3, kPairMSM><<<blocks, 32 * kWarps, 0, st>>>(K);
    return;
  }
  K.runs = use_runs(P, n);
  K.split = split_of(K.runs, n, P.ncell);
  if (KIND == kPairCutoff) launch_mk<2, kPairCutoff>(P, K, st);  // M unused
  else if (KIND == kPairWolf) launch_mk<2, kPairWolf>(P, K, st);
  else if (P.P.splitting == 1) launch_mk<1, kPairMSM>(P, K, st);
  else if (P.P.splitting == 2) launch_mk<2, kPairMSM>(P, K, st);
  else launch_mk<3, kPairMSM>(P, K, st);
}

cudaError_t launch_short_range(Plan& P, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  P.launches += 1;
  if (P.fp64) return launch_pair64(P, kPairMSM, n, 0.0, st);
  launch_f2<kPairMSM>(P, n, st);
  return cudaGetLastError();
}

cudaError_t launch_cutoff_pairs(Plan& P, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  P.launches += 1;
  if (P.fp64) return launch_pair64(P, kPairCutoff, n, 0.0, st);
  launch_f2<kPairCutoff>(P, n, st);
  return cudaGetLastError();
}

cudaError_t launch_wolf_pairs(Plan& P, int64_t n, double alpha, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  P.launches += 1;
  if (P.fp64) return launch_pair64(P, kPairWolf, n, alpha, st);
  launch_f2<kPairWolf>(P, n, st, alpha);
  return cudaGetLastError();
}

struct PairBatch {
  BatchTable<PairKArgs> cells;  // kWarps groups per block
  int splitting = 2;
  int targets = 8;  // the first replica's pair_targets
  bool flat = false;
};

cudaError_t pair_batch_build(const std::vector<BatchRep>& reps, PairBatch** out) {
  *out = nullptr;
  PairBatch* b = new (std::nothrow) PairBatch();
  if (!b) return cudaErrorMemoryAllocation;
  std::vector<PairKArgs> ka;
  std::vector<int> kb;
  int64_t sparse = 0, dense = 0;
  if (!reps.empty()) b->targets = reps[0].plan->pair_targets;
  for (const BatchRep& r : reps) {
    PairKArgs K = pair_kargs(*r.plan);
    K.natoms = (int)r.n;
    K.runs = b->targets != kCl && use_runs(*r.plan, r.n);
    ka.push_back(K);
    kb.push_back(r.n > 0 ? pair_blocks(K) : 0);
    b->splitting = r.plan->P.splitting;
    // one kernel for all replicas: the walk that suits most of their atoms
    (flat_walk(*r.plan, r.n, K.runs) ? sparse : dense) += r.n;
  }
  b->flat = sparse > dense;
  cudaError_t e = make_table(b->cells, ka, kb);
  if (e != cudaSuccess) {
    pair_batch_free(b);
    return e;
  }
  *out = b;
  return cudaSuccess;
}

cudaError_t pair_batch_launch(PairBatch* b, cudaStream_t st) {
  const int nb = b->cells.total;
  if (nb == 0) return cudaSuccess;
  const auto& t = b->cells;
  if (b->targets == kCl) {
    if (b->splitting == 1) kb_short_range_c8<1><<<nb, 32 * kWarps, 0, st>>>(t.args, t.first, t.nrep);
    else if (b->splitting == 2) kb_short_range_c8<2><<<nb, 32 * kWarps, 0, st>>>(t.args, t.first, t.nrep);
    else kb_short_range_c8<3><<<nb, 32 * kWarps, 0, st>>>(t.args, t.first, t.nrep);
    return cudaGetLastError();
  }
  auto run = [&](auto kernel) { kernel<<<nb, 32 * kWarps, 0, st>>>(t.args, t.first, t.nrep); };
  if (b->splitting == 1) run(b->flat ? kb_short_range<1, true> : kb_short_range<1, false>);
  else if (b->splitting == 2) run(b->flat ? kb_short_range<2, true> : kb_short_range<2, false>);
  else run(b->flat ? kb_short_range<3, true> : kb_short_range<3, false>);
  return cudaGetLastError();
}

void pair_batch_free(PairBatch* b) {
  if (!b) return;
  b->cells.release();
  delete b;
}

}  // namespace msm
