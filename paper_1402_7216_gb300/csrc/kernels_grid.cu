// kernels_grid.cu -- the long-range steps of MSM (Sec. "Multilevel Summation
// Method"), in the order the thesis lists them:
//   anterpolation   q^0_mu = sum_j phi^0_mu(r_j) q_j
//   restriction     q^{k+1}_mu = sum_nu phi^{k+1}_mu(r^k_nu) q^k_nu
//   lattice cutoff  u^{k,cutoff}_mu = sum_nu g^k(r^k_mu, r^k_nu) q^k_nu
//   top level       u^{l-1}_mu = sum_nu g^{l-1}(r_mu, r_nu) q^{l-1}_nu (all pairs)
//   prolongation    u^k_mu = u^{k,cutoff}_mu + sum_nu phi^{k+1}_nu(r^k_mu) u^{k+1}_nu
//   interpolation   u_i^long = sum_mu phi^0_mu(r_i) u^0_mu (and its gradient)
// with phi^k_mu = Phi(x)Phi(y)Phi(z) on spacing 2^k h, Phi the C1 cubic
// (numerical Hermite) or C1 quintic interpolant.  Grids are dense arrays,
// x fastest.  The adjoint (backward) pass reuses the same kernels: the
// transpose of interpolation is anterpolation, the transpose of prolongation
// is restriction, and the lattice and top kernels are symmetric.
#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>

#include "msm_internal.h"

namespace msm {

namespace {

// ---- nodal basis Phi ----
// Piece j of Phi covers |d| in [j, j+1]; it is written as a polynomial in the
// local coordinate u = |d| - j in [0, 1], where every coefficient is small,
// so FP32 evaluation keeps full relative accuracy (expanding in |d| instead
// would cancel terms up to ~60 against weights of ~0.01).
//   cubic   P0 = 1 - 5/2 u^2 + 3/2 u^3          P1 = -u (1 - u)^2 / 2
//   quintic Q0 = (1 - u^2)(2 - u)(6 + 3u - 5u^2)/12
//           Q1 = u (u - 1)(u - 2)(5u^2 + u - 8)/24
//           Q2 = -(u + 1) u (u - 1)^2 (u - 2)/24
template <typename T, int ORDER>
struct Basis;

template <typename T>
struct Basis<T, 3> {
  static constexpr int S = 2;
  __device__ static T p(int j, T u) {
    return j == 0 ? T(1) + u * u * (T(-2.5) + T(1.5) * u) : u * (T(-0.5) + u * (T(1) - T(0.5) * u));
  }
  __device__ static T dp(int j, T u) {
    return j == 0 ? u * (T(-5) + T(4.5) * u) : T(-0.5) + u * (T(2) - T(1.5) * u);
  }
};

template <typename T>
struct Basis<T, 5> {
  static constexpr int S = 3;
  __device__ static T p(int j, T u) {
    if (j == 0)
      return T(1) + u * u * (T(-25.0 / 12) + u * (T(5.0 / 12) + u * (T(13.0 / 12) - T(5.0 / 12) * u)));
    if (j == 1)
      return u * (T(-16.0 / 24) + u * (T(26.0 / 24) + u * (T(-1.0 / 24) + u * (T(-14.0 / 24) + T(5.0 / 24) * u))));
    return u * (T(2.0 / 24) + u * (T(-3.0 / 24) + u * (T(-1.0 / 24) + u * (T(3.0 / 24) - T(1.0 / 24) * u))));
  }
  __device__ static T dp(int j, T u) {
    if (j == 0)
      return u * (T(-50.0 / 12) + u * (T(15.0 / 12) + u * (T(52.0 / 12) - T(25.0 / 12) * u)));
    if (j == 1)
      return T(-16.0 / 24) + u * (T(52.0 / 24) + u * (T(-3.0 / 24) + u * (T(-56.0 / 24) + T(25.0 / 24) * u)));
    return T(2.0 / 24) + u * (T(-6.0 / 24) + u * (T(-3.0 / 24) + u * (T(12.0 / 24) - T(5.0 / 24) * u)));
  }
};

// Weights of the 2S support points base + s (s = 0..2S-1) for an atom at
// fractional offset f in [0,1) past grid point base + S - 1.  The signed
// distance to point s is d = f + S - 1 - s: piece S-1-s at u = f for s < S,
// piece s-S at u = 1 - f beyond.
template <typename T, int ORDER>
__device__ __forceinline__ void weights(T f, T* w) {
  constexpr int S = Basis<T, ORDER>::S;
  const T g = T(1) - f;
#pragma unroll
  for (int s = 0; s < 2 * S; ++s)
    w[s] = (s < S) ? Basis<T, ORDER>::p(S - 1 - s, f) : Basis<T, ORDER>::p(s - S, g);
}

// dPhi/dd at the same points (d > 0 for s < S, d < 0 beyond).
template <typename T, int ORDER>
__device__ __forceinline__ void dweights(T f, T* w) {
  constexpr int S = Basis<T, ORDER>::S;
  const T g = T(1) - f;
#pragma unroll
  for (int s = 0; s < 2 * S; ++s)
    w[s] = (s < S) ? Basis<T, ORDER>::dp(S - 1 - s, f) : -Basis<T, ORDER>::dp(s - S, g);
}

struct GridDims {
  int n[3];
  int lo[3];
  int periodic;
};

__device__ __forceinline__ int slot(int idx, int n, int lo, int periodic) {
  if (periodic) {
    int r = idx % n;
    return r < 0 ? r + n : r;
  }
  return idx - lo;  // callers only pass indices inside the open grid
}

// ---- anterpolation: per-block shared-memory patches (mixed plans) ----
// A block owns B x B x B short-range cells; the level-0 points their atoms
// can reach form a patch of at most PD^3 points held in shared memory.  Each
// atom adds its (2S)^3 weighted charges into the patch (shared-memory
// reductions); the block then adds the patch into the global grid, so
// global reductions only meet where neighbouring patches overlap.
struct AnterpArgs {
  int nc[3];        // short-range cells per dimension
  int B;            // cells per block side
  int pd;           // patch points per dimension
  double cw_h[3];   // cell width in units of h
};

// A block's atoms: the cells of one x row of the block are contiguous in the
// sorted order, so they are B * B ranges, found in parallel (thread r: range
// r) and laid end to end.
constexpr int kAnterpMaxAtoms = 4096;  // atoms per block listed in shared memory
constexpr int kBlockRows = 16;         // B <= 4
constexpr int kPatchThreads = 1024;    // largest block of the anterpolation kernel

struct BlockAtoms {
  int start[kBlockRows];    // first atom of a range
  int pre[kBlockRows + 1];  // atoms in the ranges before it
};

// Fills R (all threads of the block call this) and returns the atom count.
__device__ __forceinline__ int block_atoms(const AnterpArgs& A, const int* __restrict__ cell_start, int bx, int by,
                                           int bz, BlockAtoms& R) {
  if (threadIdx.x < 32) {
    const int r = threadIdx.x, x0 = bx * A.B, y = by * A.B + r % A.B, z = bz * A.B + r / A.B;
    int s = 0, len = 0;
    if (r < A.B * A.B && y < A.nc[1] && z < A.nc[2]) {
      const int* row = cell_start + (z * A.nc[1] + y) * A.nc[0];
      s = row[x0];
      len = row[min(x0 + A.B, A.nc[0])] - s;
    }
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (r >= o) incl += v;
    }
    if (r < kBlockRows) R.start[r] = s;
    if (r <= kBlockRows) R.pre[r] = incl - len;
  }
  __syncthreads();
  return R.pre[kBlockRows];
}

// The block's kk-th atom (0 <= kk < total).
__device__ __forceinline__ int block_atom(const BlockAtoms& R, int kk) {
  int r = 0;
#pragma unroll
  for (int h = kBlockRows / 2; h > 0; h >>= 1) r += kk >= R.pre[r + h] ? h : 0;
  return R.start[r] + kk - R.pre[r];
}
// The same with neighbours in kk 1/32 of the block apart (kk < 32 ceil(total / 32);
// -1 past the end): the lanes of a warp then take atoms of different cells.
__device__ __forceinline__ int spread_atom(const BlockAtoms& R, int kk, int total) {
  const int k = (kk & 31) * ((total + 31) >> 5) + (kk >> 5);
  return k < total ? block_atom(R, k) : -1;
}

// FP64 plans: one thread per atom adds its (2S)^3 weighted charges straight to
// the grid (FP64 reductions in L2).  Thread t takes atom (t mod 32) stride +
// t / 32, so the lanes of a warp lie far apart and their reductions fall on
// different points.  Bound by the FP64 rate and the reductions; patches in
// shared memory (whose FP64 additions are compare-and-swap loops) took 138 us
// in the 8 blocks of a 3,000-atom system and 123 us at 23,558 atoms.
constexpr int kWide = 64;  // threads per block of the FP64 atom kernels: small systems still reach every SM

template <int ORDER>
__global__ void __launch_bounds__(kWide) k_anterp64(const R4<double>* __restrict__ gfrac,
                                                   const int4* __restrict__ gbase, int n, int stride, GridDims G,
                                                   double* __restrict__ grid, const double* __restrict__ dscale,
                                                   double factor) {
  pdl_sync();
  constexpr int W = 2 * Basis<double, ORDER>::S;
  const int t = blockIdx.x * kWide + threadIdx.x, i = (t & 31) * stride + (t >> 5);
  if ((t >> 5) >= stride || i >= n) return;
  const R4<double> f = gfrac[i];
  const int4 b = gbase[i];
  double wx[W], wy[W], wz[W];
  weights<double, ORDER>(f.x, wx);
  weights<double, ORDER>(f.y, wy);
  weights<double, ORDER>(f.z, wz);
  const double q = f.w * (factor * (dscale ? *dscale : 1.0));
  int ix[W];
#pragma unroll
  for (int a = 0; a < W; ++a) ix[a] = slot(b.x + a, G.n[0], G.lo[0], G.periodic);
#pragma unroll
  for (int c = 0; c < W; ++c) {
    const int sz = slot(b.z + c, G.n[2], G.lo[2], G.periodic);
    const double qz = q * wz[c];
#pragma unroll
    for (int bb = 0; bb < W; ++bb) {
      const int sy = slot(b.y + bb, G.n[1], G.lo[1], G.periodic);
      const double qyz = qz * wy[bb];
      double* row = grid + ((size_t)sz * G.n[1] + sy) * G.n[0];
#pragma unroll
      for (int a = 0; a < W; ++a) atomicAdd(row + ix[a], qyz * wx[a]);
    }
  }
}

// ---- mixed precision: exact fixed-point patch sums ----
// Shared-memory FP32 atomic adds return through a compare-and-swap round
// trip, while 32-bit integer reductions are fire-and-forget.  So the mixed
// plan accumulates each patch point as two integer sums: a contribution
// c = q_j w (|w| <= 1) becomes t = c 2^12, a coarse part round(t) and a
// residual round((t - round(t)) 2^19), each added with an integer reduction.
// The patch sums are then exact, independent of order, at a resolution of
// 2^-31.  Integer sums wrap modulo 2^32, so only the final sums must fit:
// the coarse sum stays below 2^31 while |q_j| * (atoms of the block) <= 2^18
// for every atom in the patch, and the residuals (|.| <= 2^18, one per atom)
// of at most kAnterpMaxAtoms = 2^12 atoms stay below 2^30.  An atom with a
// larger charge (or |q_j| >= 2^10) goes straight to the FP64 grid.  The device-side scale (the
// adjoint's upstream gradient) multiplies the patch sums when they are
// flushed, so the fixed-point resolution is relative to the charges alone.
constexpr float kFxMagic = 12582912.0f;  // 1.5 * 2^23: adding it rounds |x| < 2^22 to an integer
constexpr float kFxCoarse = 4096.0f;     // 2^12
constexpr float kFxFine = 524288.0f;     // 2^19

__device__ __forceinline__ void fx_split(float t, int& hi, int& lo) {
  const float m = __fadd_rn(t, kFxMagic);
  hi = __float_as_int(m) - __float_as_int(kFxMagic);
  const float r = __fsub_rn(t, __fsub_rn(m, kFxMagic));  // t - round(t), exact
  lo = __float_as_int(__fmaf_rn(r, kFxFine, kFxMagic)) - __float_as_int(kFxMagic);
}

// Bank-ordered atom list.  Every tap of an atom sits at a fixed offset from
// the patch index of its first support point, so two lanes whose atoms' first
// points share a shared-memory bank (index mod 32) collide on every one of
// their (2S)^3 reductions.  The block therefore buckets its atoms by that
// bank and lays the list out in rounds of 32 slots, slot L of round r holding
// the r-th atom of bucket L: the 32 lanes of a warp instruction then touch 32
// different banks.  There are as many rounds R as the fullest bucket has atoms
// (~25 % more than total/32; with R = total/32 the overflow of the fuller
// buckets shared a bank with another lane in nearly every round, 2.2 passes of
// shared memory per instruction); where the list is too short for that, the
// overflow spills into the empty slots of the other buckets.  Integer sums do not depend on the order, so neither the
// bucket ranks nor the spill order affect the result.  Returns the slot count
// 32 R (unfilled slots hold -1); scratch (at least 32 R ints) is the not yet
// zeroed patch, else the list is in the plain order.
__device__ __forceinline__ int bank_order(const BlockAtoms& A, int total, int* list,
                                          const int4* __restrict__ gbase, int lo0, int lo1, int lo2, int PD,
                                          int* scratch, int nscratch) {
  __shared__ int bcnt[32], bempty[33], ovf, rounds;
  const int nspread = ((total + 31) >> 5) << 5;
  const int tid = threadIdx.x;
  if (total == 0) return 0;  // block-uniform
  if (nscratch < nspread) {  // a patch smaller than its atoms: the plain order
    for (int kk = tid; kk < total; kk += blockDim.x) list[kk] = block_atom(A, kk);
    __syncthreads();
    return total;
  }
  if (tid < 32) bcnt[tid] = 0;
  if (tid == 0) ovf = 0;
  __syncthreads();
  for (int kk = tid; kk < nspread; kk += blockDim.x) {
    const int i = spread_atom(A, kk, total);
    if (i < 0) continue;
    const int4 b = gbase[i];
    const int key = (((b.z - lo2) * PD + (b.y - lo1)) * PD + (b.x - lo0)) & 31;
    scratch[kk] = key | (atomicAdd(&bcnt[key], 1) << 5);
  }
  __syncthreads();
  if (tid < 32) {
    // rounds: the fullest bucket's atoms, as far as the list holds them
    const int Rm = max(nspread >> 5, min(__reduce_max_sync(0xffffffffu, bcnt[tid]), kAnterpMaxAtoms / 32 + 1));
    // empty slots of bucket L: rounds bcnt[L] .. R-1; exclusive prefix over L
    const int e = max(0, Rm - bcnt[tid]);
    int incl = e;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (tid >= o) incl += y;
    }
    bempty[tid] = incl - e;
    if (tid == 31) bempty[32] = incl;
    if (tid == 0) rounds = Rm;
  }
  __syncthreads();
  const int R = rounds, nslot = R << 5;
  for (int e = tid; e < nslot; e += blockDim.x)
    if ((e >> 5) >= bcnt[e & 31]) list[e] = -1;
  __syncthreads();
  for (int kk = tid; kk < nspread; kk += blockDim.x) {
    const int i = spread_atom(A, kk, total);
    if (i < 0) continue;
    const int key = scratch[kk] & 31, rank = scratch[kk] >> 5;
    int slot;
    if (rank < R) {
      slot = (rank << 5) | key;
    } else {
      const int o = atomicAdd(&ovf, 1);  // o < total empty slots, since 32 R >= total
      int L = 0;
      while (bempty[L + 1] <= o) ++L;
      slot = ((bcnt[L] + (o - bempty[L])) << 5) | L;
    }
    list[slot] = i;
  }
  __syncthreads();
  return nslot;
}

// Where the patch's points lie on the level-0 grid: offsets of its rows and
// planes, wrapped (or -1 outside an open grid) once per block.
struct PatchMap {
  int64_t plane[32];
  int row[32];
};

__device__ __forceinline__ int wrap_or_out(int i, int n, int lo, int periodic) {
  if (!periodic) return i - lo < 0 || i - lo >= n ? -1 : i - lo;
  while (i < 0) i += n;
  while (i >= n) i -= n;
  return i;
}

// Threads 0..63 (PD <= 32); the block synchronises before patch_rows.
__device__ __forceinline__ void patch_map(int PD, int lo1, int lo2, const GridDims& G, PatchMap& M) {
  const int t = threadIdx.x & 31;
  if (t >= PD) return;
  if (threadIdx.x < 32) {
    const int y = wrap_or_out(lo1 + t, G.n[1], G.lo[1], G.periodic);
    M.row[t] = y < 0 ? -1 : y * G.n[0];
  } else if (threadIdx.x < 64) {
    const int z = wrap_or_out(lo2 + t, G.n[2], G.lo[2], G.periodic);
    M.plane[t] = z < 0 ? -1 : (int64_t)z * G.n[1] * G.n[0];
  }
}

// Walks the PD x PD rows of a patch, a warp per row, its lanes along x: f(patch
// index, grid index or -1).
template <typename F>
__device__ __forceinline__ void patch_rows(int PD, int lo0, const GridDims& G, const PatchMap& M, F&& f) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (lane >= PD) return;
  const int x = wrap_or_out(lo0 + lane, G.n[0], G.lo[0], G.periodic);
  int y = threadIdx.x >> 5, z = 0;
  for (int e = y * PD + lane; e < PD * PD * PD; e += nw * PD, y += nw) {
    while (y >= PD) {
      y -= PD;
      ++z;
    }
    const int r = M.row[y];
    const int64_t p = M.plane[z];
    f(e, (x | r) < 0 || p < 0 ? (int64_t)-1 : p + (r + x));
  }
}

// One atom's (2S)^3 weighted charges straight into the fixed-point grid
// (global 64-bit integer reductions, 2^-31 units, computed in FP64); kept out
// of line so that the patch loop holds its weights in registers.
template <int ORDER>
__device__ __noinline__ void anterp_atom_global(const R4<float> f, const int4 b, const GridDims G,
                                                unsigned long long* __restrict__ gfx) {
  constexpr int W = 2 * Basis<float, ORDER>::S;
  float wx[W], wy[W], wz[W];
  weights<float, ORDER>(f.x, wx);
  weights<float, ORDER>(f.y, wy);
  weights<float, ORDER>(f.z, wz);
  const double qd = 2147483648.0 * (double)f.w;  // 2^31 q
#pragma unroll
  for (int c = 0; c < W; ++c) {
    const int sz = slot(b.z + c, G.n[2], G.lo[2], G.periodic);
#pragma unroll
    for (int bb = 0; bb < W; ++bb) {
      const int sy = slot(b.y + bb, G.n[1], G.lo[1], G.periodic);
      unsigned long long* row = gfx + ((size_t)sz * G.n[1] + sy) * G.n[0];
#pragma unroll
      for (int a = 0; a < W; ++a)
        atomicAdd(row + slot(b.x + a, G.n[0], G.lo[0], G.periodic),
                  (unsigned long long)__double2ll_rn(qd * (double)(wz[c] * wy[bb] * wx[a])));
    }
  }
}

template <int ORDER>
__device__ __forceinline__ void anterp_fx_body(const R4<float>* __restrict__ gfrac, const int4* __restrict__ gbase,
                                               const int* __restrict__ cell_start, const AnterpArgs& A,
                                               const GridDims& G, unsigned long long* __restrict__ gfx, int bx, int by,
                                               int bz) {
  constexpr int S = Basis<float, ORDER>::S, W = 2 * S;
  extern __shared__ unsigned char smem_raw[];
  const int PD = A.pd, np = PD * PD * PD, tid = threadIdx.x;
  int* phi_ = reinterpret_cast<int*>(smem_raw);  // coarse sums
  int* plo = phi_ + np;                          // residual sums
  __shared__ int list[kAnterpMaxAtoms + 32];  // + one round of slots
  __shared__ BlockAtoms R;
  __shared__ PatchMap M;
  const int lo0 = (int)floor(bx * A.B * A.cw_h[0]) - S - 1;
  const int lo1 = (int)floor(by * A.B * A.cw_h[1]) - S - 1;
  const int lo2 = (int)floor(bz * A.B * A.cw_h[2]) - S - 1;
  patch_map(PD, lo1, lo2, G, M);
  const int total = block_atoms(A, cell_start, bx, by, bz, R);
  if (total == 0) return;
  // |q_j| <= 2^18 / (atoms in the patch) bounds the coarse sums; |q_j| < 2^10
  // keeps |t| < 2^22, where the magic-number rounding of fx_split is exact
  const float qmax = fminf(262144.0f / (float)total, 1023.0f);
  const int count = total <= kAnterpMaxAtoms ? bank_order(R, total, list, gbase, lo0, lo1, lo2, PD, phi_, 2 * np) : 0;
  for (int e = tid; e < np; e += blockDim.x) reinterpret_cast<int2*>(phi_)[e] = make_int2(0, 0);
  __syncthreads();
  for (int kk = tid; kk < count; kk += blockDim.x) {
    const int i = list[kk];
    if (i < 0) continue;  // unfilled slot of the bank-ordered list
    const R4<float> f = gfrac[i];
    const int4 b = gbase[i];
    float wx[W], wy[W], wz[W];
    weights<float, ORDER>(f.x, wx);
    weights<float, ORDER>(f.y, wy);
    weights<float, ORDER>(f.z, wz);
    const int px = b.x - lo0, py = b.y - lo1, pz = b.z - lo2;
    if (fabsf(f.w) < qmax && px >= 0 && py >= 0 && pz >= 0 && px + W <= PD && py + W <= PD && pz + W <= PD) {
      const float qs = f.w * kFxCoarse;
#pragma unroll
      for (int c = 0; c < W; ++c) {
        const float qz = qs * wz[c];
#pragma unroll
        for (int bb = 0; bb < W; ++bb) {
          const float qyz = qz * wy[bb];
          const int off = ((pz + c) * PD + py + bb) * PD + px;
#pragma unroll
          for (int a = 0; a < W; ++a) {
            int h, l;
            fx_split(qyz * wx[a], h, l);
            atomicAdd(phi_ + off + a, h);
            atomicAdd(plo + off + a, l);
          }
        }
      }
    } else {  // large charge, or outside the patch: straight to the global grid
      anterp_atom_global<ORDER>(f, b, G, gfx);
    }
  }
  if (total > kAnterpMaxAtoms) {  // more atoms than the list holds: one thread per atom, straight to the grid
    for (int kk = tid; kk < total; kk += blockDim.x) {
      const int i = block_atom(R, kk);
      anterp_atom_global<ORDER>(gfrac[i], gbase[i], G, gfx);
    }
  }
  __syncthreads();
  // flush: the point's value in 2^-31 units, h 2^19 + l, added to the global
  // fixed-point grid with an integer reduction (no FP64 arithmetic)
  patch_rows(PD, lo0, G, M, [&](int e, int64_t g) {
    const int h = phi_[e], l = plo[e];
    if ((h | l) != 0 && g >= 0) atomicAdd(gfx + g, (unsigned long long)((long long)h * 524288LL + (long long)l));
  });
}

template <int ORDER>
__global__ void __launch_bounds__(kPatchThreads) k_anterp_fx(const R4<float>* __restrict__ gfrac, const int4* __restrict__ gbase,
                                                   const int* __restrict__ cell_start, AnterpArgs A, GridDims G,
                                                   unsigned long long* __restrict__ gfx) {
  pdl_sync();
  anterp_fx_body<ORDER>(gfrac, gbase, cell_start, A, G, gfx, blockIdx.x, blockIdx.y, blockIdx.z);
}

// Fixed-point level-0 charges (2^-31 units) to the FP64 grid, times the
// device-side scale: one conversion per grid point.
__device__ __forceinline__ void fx_to_f64_body(const unsigned long long* __restrict__ gfx, double* __restrict__ q0,
                                               int64_t count, const double* __restrict__ dscale, double factor,
                                               int64_t i) {
  if (i >= count) return;
  const double sc = factor * (dscale ? *dscale : 1.0) * (1.0 / 2147483648.0);
  q0[i] = (double)(long long)gfx[i] * sc;
}

__global__ void k_fx_to_f64(const unsigned long long* __restrict__ gfx, double* __restrict__ q0, int64_t count,
                            const double* __restrict__ dscale, double factor) {
  pdl_sync();
  fx_to_f64_body(gfx, q0, count, dscale, factor, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// ---- restriction and prolongation: separable 1-D passes ----
// phi^{k+1}_mu(r^k_nu) = prod_d Phi((nu_d - 2 mu_d)/2), so restriction is
// three 1-D filters (x, then y, then z) and prolongation, its transpose, the
// same filters in reverse order.  1-D weights Phi(d/2): cubic d = 0, +-1,
// +-3 -> 1, 9/16, -1/16; quintic d = 0, +-1, +-3, +-5 -> 1, 75/128, -25/256,
// 3/256 (Phi vanishes at the other integers).
template <int ORDER>
__device__ __forceinline__ double rweight(int ad) {
  if (ad == 0) return 1.0;
  if (ORDER == 3) return ad == 1 ? 9.0 / 16 : -1.0 / 16;
  return ad == 1 ? 75.0 / 128 : (ad == 3 ? -25.0 / 256 : 3.0 / 256);
}

struct AxisArgs {
  int nin[3], nout[3];  // array dims (x, y, z) of input and output
  int axis;             // 0, 1, 2
  int lo_in, lo_out;    // first absolute index along the axis
  int periodic;
};

// The output point t of an axis pass as (x, y, z): 32-bit divisions while
// the grid has fewer than 2^32 points (64-bit integer division is a long
// software sequence on the GPU), 64-bit beyond.
__device__ __forceinline__ void axis_point(int64_t t, const int nout[3], int64_t np, int c[3]) {
  if (np <= 0xffffffffLL) {
    const unsigned tu = (unsigned)t, n0 = (unsigned)nout[0], n1 = (unsigned)nout[1];
    const unsigned q = tu / n0;
    c[0] = (int)(tu - q * n0);
    c[1] = (int)(q % n1);
    c[2] = (int)(q / n1);
  } else {
    c[0] = (int)(t % nout[0]);
    c[1] = (int)((t / nout[0]) % nout[1]);
    c[2] = (int)(t / ((int64_t)nout[0] * nout[1]));
  }
}

// index s into [0, n) on a periodic axis: s is at most a few taps outside,
// so a wrap by additions replaces the integer modulo
__device__ __forceinline__ int wrap_periodic(int s, int n) {
  while (s < 0) s += n;
  while (s >= n) s -= n;
  return s;
}

// restriction along one axis: out[.., c, ..] = sum_d w(d) in[.., 2(lo_out + c) + d - lo_in, ..]
template <typename T, int ORDER>
__device__ __forceinline__ void restrict_axis_body(const T* __restrict__ in, T* __restrict__ out, const AxisArgs& A,
                                                   int64_t t) {
  constexpr int R = ORDER;  // taps reach |d| <= 2S - 1 = ORDER
  int64_t np = (int64_t)A.nout[0] * A.nout[1] * A.nout[2];
  if (t >= np) return;
  int c[3];
  axis_point(t, A.nout, np, c);
  int64_t stride = A.axis == 0 ? 1 : (A.axis == 1 ? (int64_t)A.nin[0] : (int64_t)A.nin[0] * A.nin[1]);
  int cc = c[A.axis];
  c[A.axis] = 0;
  const T* base = in + ((int64_t)c[2] * A.nin[1] + c[1]) * A.nin[0] + c[0];
  int n = A.nin[A.axis];
  int nu0 = 2 * (A.lo_out + cc);
  T sum = 0;
#pragma unroll
  for (int d = -R; d <= R; ++d) {
    if (d != 0 && (d & 1) == 0) continue;
    int s = nu0 + d - A.lo_in;
    if (A.periodic) {
      s = wrap_periodic(s, n);
    } else if (s < 0 || s >= n) {
      continue;
    }
    sum += T(rweight<ORDER>(d < 0 ? -d : d)) * base[s * stride];
  }
  out[t] = sum;
}

template <typename T, int ORDER>
__global__ void k_restrict_axis(const T* __restrict__ in, T* __restrict__ out, AxisArgs A) {
  pdl_sync();
  restrict_axis_body<T, ORDER>(in, out, A, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// prolongation along one axis: out[.., f, ..] (+)= sum_mu w(nu - 2 mu) in[.., mu - lo_in, ..]
template <typename T, int ORDER>
__device__ __forceinline__ void prolong_axis_body(const T* __restrict__ in, T* __restrict__ out, const AxisArgs& A,
                                                  int accumulate, int64_t t) {
  constexpr int R = ORDER;
  int64_t np = (int64_t)A.nout[0] * A.nout[1] * A.nout[2];
  if (t >= np) return;
  int c[3];
  axis_point(t, A.nout, np, c);
  int64_t stride = A.axis == 0 ? 1 : (A.axis == 1 ? (int64_t)A.nin[0] : (int64_t)A.nin[0] * A.nin[1]);
  int f = c[A.axis];
  c[A.axis] = 0;
  const T* base = in + ((int64_t)c[2] * A.nin[1] + c[1]) * A.nin[0] + c[0];
  int n = A.nin[A.axis];
  int nu = A.lo_out + f;
  T sum = 0;
#pragma unroll
  for (int d = -R; d <= R; ++d) {  // nu - 2 mu = d, d = 0 or odd
    if (d != 0 && (d & 1) == 0) continue;
    if (((nu - d) & 1) != 0) continue;
    int s = (nu - d) / 2 - A.lo_in;
    if (A.periodic) {
      s = wrap_periodic(s, n);
    } else if (s < 0 || s >= n) {
      continue;
    }
    sum += T(rweight<ORDER>(d < 0 ? -d : d)) * base[s * stride];
  }
  out[t] = accumulate ? out[t] + sum : sum;
}

// ---- restriction and prolongation in one launch per level ----
// A block computes a tile of the output from the input region it reaches,
// staged in shared memory, as the three axis passes above in turn: the same
// taps in the same order and association (restriction x, y, z; prolongation z,
// y, x), so the result is bit-identical to the three passes, in one launch
// and with no temporaries in global memory.
struct Grid3Args {
  int nin[3], nout[3];  // array dims (x, y, z) of input and output
  int lo_in[3], lo_out[3];
  int periodic;
};

// Array index of absolute index i on an axis, wrapped, or -1 outside an open grid.
__device__ __forceinline__ int axis_index(int i, int n, int lo, int periodic) {
  if (!periodic) return i - lo >= 0 && i - lo < n ? i - lo : -1;
  while (i < 0) i += n;
  while (i >= n) i -= n;
  return i;
}

// One value from global to shared memory without waiting (0 where g < 0);
// tile_wait() completes the thread's copies.
template <typename T>
__device__ __forceinline__ void tile_copy(T* dst, const T* __restrict__ src, int64_t g) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const T* p = g >= 0 ? src + g : src;
  const int bytes = g >= 0 ? (int)sizeof(T) : 0;
  if (sizeof(T) == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(p), "r"(bytes) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tile_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Restriction: kTileC^3 coarse points per block of 256 threads; small levels
// are bound by latency, so the tile's loads are all in flight at once (against
// a loop of loads and 128 threads, all levels: 80^3 fine points 80 -> 57 us,
// 32^3 27 -> 19 us, 16^3 23 -> 17 us).  The FP64
// arithmetic (2 lanes per SM and clock) of the halo makes the tile cost about
// twice the axis passes' operations, so large levels keep those (see
// restrict_by_tiles).
constexpr int kTileC = 4;
template <int ORDER>
struct RestrictTile {
  static constexpr int R = ORDER, F = 2 * kTileC + 2 * R - 1;  // fine points per side
  int idx[3][F];
  double a[F * F * F], b[F * F * kTileC];
};

template <int ORDER>
__device__ __forceinline__ void restrict_tile_body(const double* __restrict__ in, double* __restrict__ out,
                                                   const Grid3Args& A, int tile) {
  using RT = RestrictTile<ORDER>;
  constexpr int R = RT::R, F = RT::F, C = kTileC;
  __shared__ RT S;
  const int tx = (A.nout[0] + C - 1) / C, ty = (A.nout[1] + C - 1) / C;
  const int c0[3] = {tile % tx * C, tile / tx % ty * C, tile / (tx * ty) * C};
  const int tid = threadIdx.x;
  for (int e = tid; e < 3 * F; e += blockDim.x) {
    const int d = e / F, f = e - d * F;
    S.idx[d][f] = axis_index(2 * (A.lo_out[d] + c0[d]) - R + f, A.nin[d], A.lo_in[d], A.periodic);
  }
  __syncthreads();
  for (int e = tid; e < F * F * F; e += blockDim.x) {
    const int x = S.idx[0][e % F], y = S.idx[1][e / F % F], z = S.idx[2][e / (F * F)];
    tile_copy(S.a + e, in, (x | y | z) < 0 ? (int64_t)-1 : ((int64_t)z * A.nin[1] + y) * A.nin[0] + x);
  }
  tile_wait();
  __syncthreads();
  auto taps = [&](const double* v, int stride) {  // v: the point at offset 0
    double sum = 0.0;
#pragma unroll
    for (int d = -R; d <= R; ++d)
      if (d == 0 || (d & 1)) sum += rweight<ORDER>(d < 0 ? -d : d) * v[d * stride];
    return sum;
  };
  for (int e = tid; e < F * F * C; e += blockDim.x) S.b[e] = taps(S.a + e / C * F + 2 * (e % C) + R, 1);
  __syncthreads();
  for (int e = tid; e < F * C * C; e += blockDim.x) {
    const int c = e % C, y = e / C % C, z = e / (C * C);
    S.a[e] = taps(S.b + (z * F + 2 * y + R) * C + c, C);
  }
  __syncthreads();
  for (int e = tid; e < C * C * C; e += blockDim.x) {
    const int c = e % C, y = e / C % C, z = e / (C * C);
    const int x = c0[0] + c, yy = c0[1] + y, zz = c0[2] + z;
    if (x < A.nout[0] && yy < A.nout[1] && zz < A.nout[2])
      out[((size_t)zz * A.nout[1] + yy) * A.nout[0] + x] = taps(S.a + ((2 * z + R) * C + y) * C + c, C * C);
  }
}

template <int ORDER>
__global__ void __launch_bounds__(256) k_restrict_tile(const double* __restrict__ in, double* __restrict__ out,
                                                       Grid3Args A) {
  pdl_sync();
  restrict_tile_body<ORDER>(in, out, A, blockIdx.x);
}

// Prolongation: 32 x TYZ x TYZ fine points per block of 256 threads, added
// onto the output.  Bound by memory on large levels (the output read and
// written once, the coarse grid read once): 240^3 points in 3 axis passes took
// 352 us.
constexpr int kTileX = 32;
template <typename T, int ORDER, int TYZ>
struct ProlongTile {
  static constexpr int R = ORDER, CX = kTileX / 2 + R + 1, CY = TYZ / 2 + R + 1;  // coarse points reached
  int idx[3][CX];
  T a[CY * CY * CX], b[TYZ * CY * CX];
};

template <typename T, int ORDER, int TYZ>
__device__ __forceinline__ void prolong_tile_body(const T* __restrict__ in, T* __restrict__ out, const Grid3Args& A,
                                                  int tile) {
  using PT = ProlongTile<T, ORDER, TYZ>;
  constexpr int R = PT::R, CX = PT::CX, CY = PT::CY;
  __shared__ PT S;
  const int tx = (A.nout[0] + kTileX - 1) / kTileX, ty = (A.nout[1] + TYZ - 1) / TYZ;
  const int f0[3] = {tile % tx * kTileX, tile / tx % ty * TYZ, tile / (tx * ty) * TYZ};
  const int tid = threadIdx.x;
  int nu0[3], co[3];  // absolute fine index of the tile's corner, lowest coarse index it reaches
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    nu0[d] = A.lo_out[d] + f0[d];
    co[d] = (nu0[d] + 1 - R) >> 1;
  }
  for (int e = tid; e < 3 * CX; e += blockDim.x) {
    const int d = e / CX, c = e - d * CX;
    S.idx[d][c] = axis_index(co[d] + c, A.nin[d], A.lo_in[d], A.periodic);
  }
  __syncthreads();
  for (int e = tid; e < CY * CY * CX; e += blockDim.x) {
    const int x = S.idx[0][e % CX], y = S.idx[1][e / CX % CY], z = S.idx[2][e / (CX * CY)];
    tile_copy(S.a + e, in, (x | y | z) < 0 ? (int64_t)-1 : ((int64_t)z * A.nin[1] + y) * A.nin[0] + x);
  }
  tile_wait();
  __syncthreads();
  // fine index nu (even: the coarse point nu / 2; odd: those at odd distances up to R); v: coarse point co
  auto taps = [&](const T* v, int stride, int nu, int c) {
    if ((nu & 1) == 0) return v[((nu >> 1) - c) * stride];
    T sum = 0;
#pragma unroll
    for (int d = -R; d <= R; d += 2) sum += T(rweight<ORDER>(d < 0 ? -d : d)) * v[(((nu - d) >> 1) - c) * stride];
    return sum;
  };
  for (int e = tid; e < TYZ * CY * CX; e += blockDim.x) {
    const int z = e / (CY * CX), yx = e - z * CY * CX;
    S.b[e] = taps(S.a + yx, CY * CX, nu0[2] + z, co[2]);
  }
  __syncthreads();
  for (int e = tid; e < TYZ * TYZ * CX; e += blockDim.x) {
    const int x = e % CX, y = e / CX % TYZ, z = e / (CX * TYZ);
    S.a[e] = taps(S.b + z * CY * CX + x, CX, nu0[1] + y, co[1]);
  }
  __syncthreads();
  for (int e = tid; e < TYZ * TYZ * kTileX; e += blockDim.x) {
    const int x = e % kTileX, y = e / kTileX % TYZ, z = e / (kTileX * TYZ);
    if (f0[0] + x < A.nout[0] && f0[1] + y < A.nout[1] && f0[2] + z < A.nout[2]) {
      T* o = out + ((size_t)(f0[2] + z) * A.nout[1] + f0[1] + y) * A.nout[0] + f0[0] + x;
      *o = *o + taps(S.a + (z * TYZ + y) * CX, 1, nu0[0] + x, co[0]);  // onto u^{k, cutoff}
    }
  }
}

template <typename T, int ORDER, int TYZ>
__global__ void __launch_bounds__(256) k_prolong_tile(const T* __restrict__ in, T* __restrict__ out, Grid3Args A) {
  pdl_sync();
  prolong_tile_body<T, ORDER, TYZ>(in, out, A, blockIdx.x);
}

// ---- lattice cutoff by the stencil, FP64 ----
// One thread per output point, the stencil as rows of taps along x (dy, dz, half
// length X, coefficients of dx = -X .. X).  Bound by the FP64 rate (2 lanes per
// SM and clock), so what counts is one FP64 FMA per tap and no other: the rows
// hold no padding, the coefficients are warp-uniform loads, the charges come
// through the cache, and all index arithmetic runs beside the FMAs.  Small
// grids share the rows among gridDim.y blocks, whose parts k_lattice_reduce
// adds in order (no atomics: reproducible).  Register tiles of 8 outputs with
// segments of 8 taps spent ~3x the FMAs on padding and idle lanes on a 16^3
// grid: 251 -> 65 us for both levels of a 3,000-atom open system alone, and
// 888 -> 146 us beside the pair sums.
constexpr int kLat64 = 128;  // threads per block

template <bool PERIODIC>
__global__ void __launch_bounds__(kLat64) k_lattice64(const double* __restrict__ q, double* __restrict__ u,
                                                     double* __restrict__ up, GridDims G,
                                                     const int4* __restrict__ rows, const double* __restrict__ coef,
                                                     int nrows, int per, double scale) {
  pdl_sync();
  const int n0 = G.n[0], n1 = G.n[1], n2 = G.n[2];
  const int64_t np = (int64_t)n0 * n1 * n2, p = (int64_t)blockIdx.x * kLat64 + threadIdx.x;
  if (p >= np) return;
  const int x = (int)(p % n0), y = (int)((p / n0) % n1), z = (int)(p / ((int64_t)n0 * n1));
  const int r1 = min(nrows, ((int)blockIdx.y + 1) * per);
  double acc = 0.0;
  for (int r = blockIdx.y * per; r < r1; ++r) {
    const int4 R = rows[r];  // (dy, dz, X, first coefficient)
    int yy = y + R.x, zz = z + R.y;
    if (PERIODIC) {
      while (yy < 0) yy += n1;
      while (yy >= n1) yy -= n1;
      while (zz < 0) zz += n2;
      while (zz >= n2) zz -= n2;
    } else if (yy < 0 || zz < 0 || yy >= n1 || zz >= n2) {
      continue;
    }
    const double* row = q + ((int64_t)zz * n1 + yy) * n0;
    const double* g = coef + R.w;
    double sum = 0.0;
    if (PERIODIC) {
      int i = x - R.z;
      while (i < 0) i += n0;
#pragma unroll 4
      for (int k = 0; k <= 2 * R.z; ++k) {
        sum = fma(g[k], row[i], sum);
        i = i + 1 == n0 ? 0 : i + 1;
      }
    } else {
#pragma unroll 4
      for (int k = 0; k <= 2 * R.z; ++k) {
        const int i = x - R.z + k;
        const double v = i >= 0 && i < n0 ? row[i] : 0.0;
        sum = fma(g[k], v, sum);
      }
    }
    acc += sum;
  }
  acc *= scale;
  if (gridDim.y > 1) up[(int64_t)blockIdx.y * np + p] = acc;
  else u[p] = acc;
}

// ---- lattice cutoff by the stencil, FP32: z-streaming shared-memory planes, register tiles ----
// A block of 4 warps owns a brick of outputs 32 (x) x 16 (y) x 4 (z); warp w
// owns plane z0 + w.  The input planes are staged one at a time in shared
// memory (a 2-D window with halo Ex, Ey; odd row pitch so the lanes of a warp
// sit on distinct banks); for staged plane zi, warp w applies the stencil rows
// of dz = zi - (z0 + w) as segments of 8 taps along x on register tiles of
// 8 consecutive x outputs per lane, two rows packed into float2 (one FFMA2
// per two outputs).  Coarse levels with few bricks split the input planes over
// several blocks (nsplit): block part writes its partial sums to
// up[part][point] and k_lattice_reduce adds the parts in order.
constexpr int LBX = 32;         // see lattice_fits
constexpr int kLatticeLP = 8;   // x outputs per lane of the FP32 lattice kernel (8 or 16)
constexpr int kLatticeZ = 4;    // warps (output planes) per block of the FP32 lattice kernel
constexpr size_t kLatticeSmemMax = 200 * 1024;  // dynamic shared memory the FP32 lattice kernels may use

struct LatticeArgs {
  int Ex, Ey, Ez;
  int nsplit;  // blocks sharing one brick's input planes
  int nbz;     // bricks along z
  int txn, tyn;  // lanes along x (LP outputs each) and along y (two rows each) of a warp's tile
};

// Window offsets of a block, computed once (the periodic wrap costs integer
// divisions): col[xx] = grid x index of window column xx (-1 outside an open
// grid), row[yy] = (grid y index) * n_x (-1 outside).
__device__ __forceinline__ void window_offsets(const GridDims& G, int x0, int y0, int Ex, int Ey, int SXw, int SY,
                                               int* col, int* row) {
  for (int t = threadIdx.x; t < SXw + SY; t += blockDim.x) {
    const bool isx = t < SXw;
    const int n = isx ? G.n[0] : G.n[1];
    int g = isx ? x0 - Ex + t : y0 - Ey + (t - SXw);
    if (G.periodic) {
      g %= n;
      if (g < 0) g += n;
    } else if (g < 0 || g >= n) {
      g = -1;
    }
    if (isx) col[t] = g;
    else row[t - SXw] = g < 0 ? -1 : g * G.n[0];
  }
}

// Asynchronous staging of one plane (cp.async: global -> shared without
// registers); points outside an open grid are zero-filled (source size 0).
// Each thread walks the window with a fixed stride of blockDim.x elements,
// stepping its (row, column) incrementally.  Window rows are stored even rows
// first, then odd rows (row yy at yy / 2 + (yy odd) * SY / 2): lanes reading
// rows 2 ty + c then read rows ty apart, one odd row stride SX apart, which
// keeps the lanes of a warp on distinct banks.
__device__ __forceinline__ void stage_plane_async(float* plane, const float* __restrict__ q, const GridDims& G,
                                                  int zi, const int* col, const int* row, int SXw, int SX, int SY) {
  int gz;
  bool zok;
  if (G.periodic) {
    gz = zi % G.n[2];
    if (gz < 0) gz += G.n[2];
    zok = true;
  } else {
    gz = zi;
    zok = (zi >= 0 && zi < G.n[2]);
  }
  const float* qz = q + (size_t)(zok ? gz : 0) * G.n[1] * G.n[0];
  const int step = blockDim.x, dyy = step / SXw, dxx = step - dyy * SXw;
  int xx = threadIdx.x % SXw, yy = threadIdx.x / SXw;
  for (; yy < SY; ) {
    const int gx = col[xx], go = row[yy];
    const bool ok = zok && gx >= 0 && go >= 0;
    const float* src = ok ? qz + go + gx : q;
    unsigned dst = (unsigned)__cvta_generic_to_shared(plane + ((yy >> 1) + (yy & 1) * (SY >> 1)) * SX + xx);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(ok ? 4 : 0));
    xx += dxx;
    yy += dyy;
    if (xx >= SXw) {
      xx -= SXw;
      ++yy;
    }
  }
}

// FP32: each lane owns LP consecutive x outputs of two adjacent rows (y,
// y + 1), packed into float2 (one FFMA2 per two outputs); a warp covers TXN LP
// (x) x 2 TYN (y) of one plane.  An input row y + e feeds both outputs, row y
// through the taps of stencil row e and row y + 1 through those of row e - 1,
// so the table holds those coefficient pairs and one shared load serves both
// rows (against two rows TYN apart with one coefficient each: 5% faster on
// the 1.07M-atom system, 9% on the 64-replica batch).  The next input plane
// is staged by cp.async while the current one is applied (double buffer).  A
// segment of 8 taps is applied as a sliding window: input column k feeds the
// outputs j = k - t of every tap t, so one shared load serves up to 8 FFMA2
// (LP + 7 loads per 8 LP FFMA2); the row pairing costs 2 Ey + 2 input rows per
// output pair instead of 2 Ey + 1.  The block's warps share each input plane
// and apply to it different stencil planes dz, of unequal size, so a warp
// may wait at the plane's barrier; stepping the warps through dz together
// (each on its own input plane, a ring of kLatticeZ + 1 buffers) removes the
// wait but measured 15-20% slower, the larger ring costing resident blocks.  Taps accumulate straight into the outputs (summing each
// plane first measured no different on the 1.07M-atom system: mixed-vs-FP64
// energy 4.4e-8, force 4.9e-7).
// TXC, TYC: the warp tile fixed at compile time (the common 32 x 16 tile),
// or 0 to take it from L (other shapes, batches of uneven grids).
template <int LP, int TXC, int TYC>
__device__ __forceinline__ void lattice_f2_body(const float* __restrict__ q, float* __restrict__ u,
                                                float* __restrict__ up, const GridDims G,
                                                const Segment2* __restrict__ seg, const int* __restrict__ seg_start,
                                                const LatticeArgs L, float scale, int bx, int by, int bzs) {
  const int TXN = TXC ? TXC : L.txn, TYN = TYC ? TYC : L.tyn, TW = LP * TXN, LBY = 2 * TYN;  // tile: TW (x) by LBY (y)
  extern __shared__ unsigned char smem_raw[];
  const int Ex = L.Ex, Ey = L.Ey, Ez = L.Ez;
  const int SXw = TW + 2 * Ex + kSeg, SX = SXw | 1, SY = LBY + 2 * Ey;
  float* buf0 = reinterpret_cast<float*>(smem_raw);
  float* buf1 = buf0 + SX * SY;
  int* col = reinterpret_cast<int*>(buf1 + SX * SY);  // window offsets (SXw + SY ints)
  int* row = col + SXw;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tx = lane % TXN, ty = lane / TXN;
  const bool active = (TXC * TYC == 32) || ty < TYN;  // lanes past TXN * TYN only help with staging
  const int bz = bzs % L.nbz, part = bzs / L.nbz;
  const int x0 = bx * TW, y0 = by * LBY, z0 = bz * kLatticeZ, zo = z0 + warp;
  const int nplanes = kLatticeZ + 2 * Ez, per = (nplanes + L.nsplit - 1) / L.nsplit;
  const int zbeg = z0 - Ez + part * per, zend = min(z0 - Ez + nplanes, zbeg + per);
  float2 acc[LP];  // (row 2 ty, row 2 ty + 1) of the LP x outputs
#pragma unroll
  for (int j = 0; j < LP; ++j) acc[j] = make_float2(0.f, 0.f);
  window_offsets(G, x0, y0, Ex, Ey, SXw, SY, col, row);
  __syncthreads();
  if (zbeg < zend) stage_plane_async(buf0, q, G, zbeg, col, row, SXw, SX, SY);
  asm volatile("cp.async.commit_group;\n" ::);
  for (int zi = zbeg; zi < zend; ++zi) {
    float* cur = ((zi - zbeg) & 1) ? buf1 : buf0;
    float* nxt = ((zi - zbeg) & 1) ? buf0 : buf1;
    if (zi + 1 < zend) stage_plane_async(nxt, q, G, zi + 1, col, row, SXw, SX, SY);
    asm volatile("cp.async.commit_group;\n" ::);
    asm volatile("cp.async.wait_group 1;\n" ::);  // plane zi has landed (this thread's copies)
    __syncthreads();                               // ... and everyone else's
    const int dz = zi - zo;
    if (active && dz >= -Ez && dz <= Ez && zo < G.n[2]) {
      const int s1 = seg_start[dz + Ez + 1];
#pragma unroll 2  // the next segment's coefficients load under this one's FMAs
      for (int s = seg_start[dz + Ez]; s < s1; ++s) {
        const Segment2 sg = seg[s];
        const int c = Ey + sg.dy;  // window row 2 ty + c, stored at ty + c / 2 (+ SY / 2 when c is odd)
        const float* r0 = cur + (ty + (c >> 1) + (c & 1) * (SY >> 1)) * SX + tx * LP + Ex + sg.dx0;
#pragma unroll
        for (int k = 0; k < LP + kSeg - 1; ++k) {
          const float v = r0[k];
          const float2 w = make_float2(v, v);
#pragma unroll
          for (int t = 0; t < kSeg; ++t)
            if (k - t >= 0 && k - t < LP) acc[k - t] = __ffma2_rn(sg.g[t], w, acc[k - t]);
        }
      }
    }
    __syncthreads();  // the buffer just read is restaged two planes from now
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
  if (zo >= G.n[2] || !active) return;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int y = y0 + 2 * ty + r;
    if (y >= G.n[1]) continue;
#pragma unroll
    for (int j = 0; j < LP; ++j) {
      int x = x0 + tx * LP + j;
      if (x >= G.n[0]) continue;
      float v = scale * (r == 0 ? acc[j].x : acc[j].y);
      const size_t o = ((size_t)zo * G.n[1] + y) * G.n[0] + x;
      if (L.nsplit > 1) up[(size_t)part * G.n[0] * G.n[1] * G.n[2] + o] = v;  // summed in order by k_lattice_reduce
      else u[o] = v;
    }
  }
}

template <int LP, int TXC, int TYC>
__global__ void __launch_bounds__(32 * kLatticeZ, 6) k_lattice_f2(const float* __restrict__ q, float* __restrict__ u,
                                                               float* __restrict__ up, GridDims G,
                                                               const Segment2* __restrict__ seg,
                                                               const int* __restrict__ seg_start, LatticeArgs L,
                                                               float scale) {
  pdl_sync();
  lattice_f2_body<LP, TXC, TYC>(q, u, up, G, seg, seg_start, L, scale, blockIdx.x, blockIdx.y, blockIdx.z);
}

// u[i] = sum over the parts p = 0..nsplit-1 of up[p][i], in that order.
template <typename T>
__device__ __forceinline__ void lattice_reduce_body(const T* __restrict__ up, T* __restrict__ u, int64_t np,
                                                    int nsplit, int64_t i) {
  if (i >= np) return;
  T v = up[i];
  for (int p = 1; p < nsplit; ++p) v += up[(size_t)p * np + i];
  u[i] = v;
}

template <typename T>
__global__ void __launch_bounds__(256) k_lattice_reduce(const T* __restrict__ up, T* __restrict__ u, int64_t np,
                                                        int nsplit) {
  pdl_sync();
  lattice_reduce_body<T>(up, u, np, nsplit, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// ---- top level: all pairs of the coarsest grid, FP64 ----
// One warp per output point: the lanes split the sum over the points of the
// coarsest grid and combine their FP64 partial sums with shuffles.
template <typename T>
__device__ __forceinline__ void top_body(const double* __restrict__ qt, T* __restrict__ ut, double* __restrict__ ut64,
                                         const GridDims& G, const double* __restrict__ K, int tx, int ty,
                                         int64_t m) {
  const int lane = threadIdx.x & 31;
  const int n0 = G.n[0], n1 = G.n[1], n2 = G.n[2];
  const int np = n0 * n1 * n2;
  if (m >= np) return;  // warp-uniform
  const int mx = (int)(m % n0), my = (int)((m / n0) % n1), mz = (int)(m / ((int64_t)n0 * n1));
  double sum = 0.0;
  for (int v = lane; v < np; v += 32) {
    const int vx = v % n0, vy = (v / n0) % n1, vz = v / (n0 * n1);
    int dx = mx - vx, dy = my - vy, dz = mz - vz;
    if (G.periodic) {
      dx += dx < 0 ? n0 : 0;
      dy += dy < 0 ? n1 : 0;
      dz += dz < 0 ? n2 : 0;
    } else {
      dx += n0 - 1;
      dy += n1 - 1;
      dz += n2 - 1;
    }
    sum += K[((size_t)dz * ty + dy) * tx + dx] * qt[v];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) {
    ut[m] = (T)sum;
    ut64[m] = sum;
  }
}

constexpr int kTopWarps = 4;  // output points per block of the top-level kernel

template <typename T>
__global__ void __launch_bounds__(32 * kTopWarps) k_top(const double* __restrict__ qt, T* __restrict__ ut,
                                                        double* __restrict__ ut64, GridDims G,
                                                        const double* __restrict__ K, int tx, int ty, int tz) {
  pdl_sync();
  top_body<T>(qt, ut, ut64, G, K, tx, ty, (int64_t)blockIdx.x * kTopWarps + (threadIdx.x >> 5));
  (void)tz;
}

// ---- interpolation at the atoms and assembly (forward) ----
template <typename T, int ORDER>
__device__ __forceinline__ void interp_atom(const R4<T>& f, const int4& b, const T* __restrict__ u0,
                                            const GridDims& G, const T inv_h[3], T& p, T g[3]) {
  constexpr int W = 2 * Basis<T, ORDER>::S;
  T wx[W], wy[W], wz[W], dx[W], dy[W], dz[W];
  weights<T, ORDER>(f.x, wx);
  weights<T, ORDER>(f.y, wy);
  weights<T, ORDER>(f.z, wz);
  dweights<T, ORDER>(f.x, dx);
  dweights<T, ORDER>(f.y, dy);
  dweights<T, ORDER>(f.z, dz);
  int ix[W], iy[W], iz[W];
#pragma unroll
  for (int s = 0; s < W; ++s) {
    ix[s] = slot(b.x + s, G.n[0], G.lo[0], G.periodic);
    iy[s] = slot(b.y + s, G.n[1], G.lo[1], G.periodic);
    iz[s] = slot(b.z + s, G.n[2], G.lo[2], G.periodic);
  }
  T P = 0, Gx = 0, Gy = 0, Gz = 0;
#pragma unroll
  for (int c = 0; c < W; ++c) {
    T pz = 0, gxz = 0, gyz = 0;
#pragma unroll
    for (int bb = 0; bb < W; ++bb) {
      const T* row = u0 + ((size_t)iz[c] * G.n[1] + iy[bb]) * G.n[0];
      T sa = 0, sd = 0;
#pragma unroll
      for (int a = 0; a < W; ++a) {
        T v = __ldg(row + ix[a]);
        sa += wx[a] * v;
        sd += dx[a] * v;
      }
      pz += wy[bb] * sa;
      gxz += wy[bb] * sd;
      gyz += dy[bb] * sa;
    }
    P += wz[c] * pz;
    Gx += wz[c] * gxz;
    Gy += wz[c] * gyz;
    Gz += dz[c] * pz;
  }
  p = P;
  g[0] = Gx * inv_h[0];
  g[1] = Gy * inv_h[1];
  g[2] = Gz * inv_h[2];
}

template <int BLOCK>
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double red[BLOCK / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (w == 0) {
    s = (lane < BLOCK / 32) ? red[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  return s;  // valid in thread 0
}

struct AssembleArgs {
  double self_c;  // gamma(0)/a
  double kc;      // Coulomb prefactor
  double inv_h[3];
  float self_cf, kcf;  // the same in FP32 (mixed plans assemble in FP32)
};

// Per-atom assembly of phi_i, F_i (forward) and of dL/dq_i, dL/dr_i
// (adjoint).  The mixed plan works in FP32 and converts once per output (FP64
// operations, conversions included, issue at 1/64 of the FP32 rate here); the
// FP64 plan works in FP64.
template <typename T>
struct Assemble;
template <>
struct Assemble<float> {
  template <typename OUT>
  __device__ static double forward(const AssembleArgs& A, float q, float phis, float p, const R4<float>& s,
                                   const float g[3], int o, OUT* phi_out, OUT* force_out) {
    const float phi = A.kcf * ((phis + p) - q * A.self_cf);
    if (phi_out) phi_out[o] = (OUT)phi;
    if (force_out) {
      force_out[3 * (size_t)o + 0] = (OUT)(A.kcf * (s.x - q * g[0]));
      force_out[3 * (size_t)o + 1] = (OUT)(A.kcf * (s.y - q * g[1]));
      force_out[3 * (size_t)o + 2] = (OUT)(A.kcf * (s.z - q * g[2]));
    }
    return (double)(q * phi);
  }
  template <typename OUT>
  __device__ static void backward(const AssembleArgs& A, float gg, float q, float phis, const R4<float>& s,
                                  const R4<float>& gl, float v, const float gv[3], int o, OUT* grad_pos,
                                  OUT* grad_q) {
    const float hg = 0.5f * gg;
    if (grad_q) grad_q[o] = (OUT)(A.kcf * (gg * (phis - q * A.self_cf) + hg * gl.w + v));
    if (grad_pos) {
      grad_pos[3 * (size_t)o + 0] = (OUT)(A.kcf * (-gg * s.x + hg * q * gl.x + q * gv[0]));
      grad_pos[3 * (size_t)o + 1] = (OUT)(A.kcf * (-gg * s.y + hg * q * gl.y + q * gv[1]));
      grad_pos[3 * (size_t)o + 2] = (OUT)(A.kcf * (-gg * s.z + hg * q * gl.z + q * gv[2]));
    }
  }
};
template <>
struct Assemble<double> {
  template <typename OUT>
  __device__ static double forward(const AssembleArgs& A, double q, double phis, double p, const R4<double>& s,
                                   const double g[3], int o, OUT* phi_out, OUT* force_out) {
    const double phi = A.kc * (phis + p - q * A.self_c);
    if (phi_out) phi_out[o] = (OUT)phi;
    if (force_out) {
      force_out[3 * (size_t)o + 0] = (OUT)(A.kc * (s.x - q * g[0]));
      force_out[3 * (size_t)o + 1] = (OUT)(A.kc * (s.y - q * g[1]));
      force_out[3 * (size_t)o + 2] = (OUT)(A.kc * (s.z - q * g[2]));
    }
    return q * phi;
  }
  template <typename OUT>
  __device__ static void backward(const AssembleArgs& A, double gg, double q, double phis, const R4<double>& s,
                                  const R4<double>& gl, double v, const double gv[3], int o, OUT* grad_pos,
                                  OUT* grad_q) {
    if (grad_q) grad_q[o] = (OUT)(A.kc * (gg * (phis - q * A.self_c) + 0.5 * gg * gl.w + v));
    if (grad_pos) {
      grad_pos[3 * (size_t)o + 0] = (OUT)(A.kc * (-gg * s.x + 0.5 * gg * q * gl.x + q * gv[0]));
      grad_pos[3 * (size_t)o + 1] = (OUT)(A.kc * (-gg * s.y + 0.5 * gg * q * gl.y + q * gv[1]));
      grad_pos[3 * (size_t)o + 2] = (OUT)(A.kc * (-gg * s.z + 0.5 * gg * q * gl.z + q * gv[2]));
    }
  }
};

// Interpolation through the same per-block patches: a block stages the u^0
// points its atoms can reach (PD^3, wrapped) in shared memory, then each
// thread gathers its atoms' (2S)^3 taps from there.
template <typename T, int ORDER>
__device__ __forceinline__ void interp_patch_atom(const R4<T>& f, const int4& b, const T* __restrict__ patch, int PD,
                                                  int lo0, int lo1, int lo2, const T* __restrict__ u0,
                                                  const GridDims& G, const T ih[3], T& p, T g[3]) {
  constexpr int W = 2 * Basis<T, ORDER>::S;
  const int px = b.x - lo0, py = b.y - lo1, pz = b.z - lo2;
  if (px >= 0 && py >= 0 && pz >= 0 && px + W <= PD && py + W <= PD && pz + W <= PD) {
    T wx[W], wy[W], wz[W], dx[W], dy[W], dz[W];
    weights<T, ORDER>(f.x, wx);
    weights<T, ORDER>(f.y, wy);
    weights<T, ORDER>(f.z, wz);
    dweights<T, ORDER>(f.x, dx);
    dweights<T, ORDER>(f.y, dy);
    dweights<T, ORDER>(f.z, dz);
    T P = 0, Gx = 0, Gy = 0, Gz = 0;
#pragma unroll
    for (int c = 0; c < W; ++c) {
      T pzv = 0, gxz = 0, gyz = 0;
#pragma unroll
      for (int bb = 0; bb < W; ++bb) {
        const T* row = patch + ((pz + c) * PD + py + bb) * PD + px;
        T sa = 0, sd = 0;
#pragma unroll
        for (int a = 0; a < W; ++a) {
          T v = row[a];
          sa += wx[a] * v;
          sd += dx[a] * v;
        }
        pzv += wy[bb] * sa;
        gxz += wy[bb] * sd;
        gyz += dy[bb] * sa;
      }
      P += wz[c] * pzv;
      Gx += wz[c] * gxz;
      Gy += wz[c] * gyz;
      Gz += dz[c] * pzv;
    }
    p = P;
    g[0] = Gx * ih[0];
    g[1] = Gy * ih[1];
    g[2] = Gz * ih[2];
  } else {
    interp_atom<T, ORDER>(f, b, u0, G, ih, p, g);
  }
}

// Lists the block's atoms (bank-ordered with the patch as scratch: the gathers
// of one warp instruction then read 32 different banks) and stages the patch
// of u^0.  Returns the slot count of the list (unfilled slots hold -1), or -1
// when the block holds more atoms than the list takes.
__device__ __forceinline__ int stage_interp_block(const AnterpArgs& A, const int* __restrict__ cell_start,
                                                  const int4* __restrict__ gbase, const float* __restrict__ u0,
                                                  const GridDims& G, float* patch, int lo0, int lo1, int lo2,
                                                  BlockAtoms& R, int* list, int bx, int by, int bz) {
  const int PD = A.pd;
  __shared__ PatchMap M;
  patch_map(PD, lo1, lo2, G, M);
  int total = block_atoms(A, cell_start, bx, by, bz, R);
  if (total == 0) return 0;
  total = total <= kAnterpMaxAtoms
              ? bank_order(R, total, list, gbase, lo0, lo1, lo2, PD, reinterpret_cast<int*>(patch), PD * PD * PD)
              : -1;
  // asynchronous copies: every row's loads are in flight together
  patch_rows(PD, lo0, G, M, [&](int e, int64_t g) {
    if (g >= 0)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(patch + e)),
                   "l"(u0 + g)
                   : "memory");
    else
      patch[e] = 0.f;
  });
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  return total;
}

// Arguments of the interpolation kernels (one system): the forward kernel
// writes phi_out, force_out, fs.w, glong and the per-block energy partials;
// the adjoint kernel reads fs and glong and writes grad_pos, grad_q.
template <typename T, typename OUT>
struct InterpKArgs {
  const R4<T>* gfrac;
  const int4* gbase;
  const int* perm;
  const int* cell_start;
  AnterpArgs AA;
  const T* u0;  // u^0 (forward) or the adjoint grid (backward)
  GridDims G;
  AssembleArgs A;
  const T* phis;
  R4<T>* fs;
  R4<T>* glong;
  OUT* phi_out;
  OUT* force_out;
  double* partial;
  const double* gE;
  OUT* grad_pos;
  OUT* grad_q;
  int nbx, nby;  // blocks along x and y
};

// GATHER: interpolate only (u_long and its gradient into glong; no pair
// results needed, so this runs while the pair sums are still being computed),
// else also assemble phi, F and the energy partials.
template <int ORDER, typename OUT, bool GATHER = false>
__device__ __forceinline__ void interp_fwd_body(
    const R4<float>* __restrict__ gfrac, const int4* __restrict__ gbase, const int* __restrict__ perm,
    const int* __restrict__ cell_start, const AnterpArgs& AA, const float* __restrict__ u0, const GridDims& G,
    const AssembleArgs& A, const float* __restrict__ phis, R4<float>* __restrict__ fs, R4<float>* __restrict__ glong,
    OUT* __restrict__ phi_out, OUT* __restrict__ force_out, double* __restrict__ partial, int bx, int by, int bz,
    int lin) {
  constexpr int S = Basis<float, ORDER>::S;
  extern __shared__ unsigned char smem_raw[];
  float* patch = reinterpret_cast<float*>(smem_raw);
  __shared__ int list[kAnterpMaxAtoms + 32];  // + one round of slots
  __shared__ BlockAtoms R;
  const int lo0 = (int)floor(bx * AA.B * AA.cw_h[0]) - S - 1;
  const int lo1 = (int)floor(by * AA.B * AA.cw_h[1]) - S - 1;
  const int lo2 = (int)floor(bz * AA.B * AA.cw_h[2]) - S - 1;
  const int total =
      stage_interp_block(AA, cell_start, gbase, u0, G, patch, lo0, lo1, lo2, R, list, bx, by, bz);
  const float ih[3] = {(float)A.inv_h[0], (float)A.inv_h[1], (float)A.inv_h[2]};
  double e = 0.0;
  // atoms from the list, or (over-full block) in the plain order
  const int nlist = total >= 0 ? total : R.pre[kBlockRows];
  for (int kk = threadIdx.x; kk < nlist; kk += blockDim.x) {
    const int i = total >= 0 ? list[kk] : block_atom(R, kk);
    if (i < 0) continue;  // unfilled slot of the bank-ordered list
    const R4<float> f = gfrac[i];
    float p, g[3];
    interp_patch_atom<float, ORDER>(f, gbase[i], patch, AA.pd, lo0, lo1, lo2, u0, G, ih, p, g);
    if (!GATHER) e += Assemble<float>::forward(A, f.w, phis[i], p, fs[i], g, perm[i], phi_out, force_out);
    glong[i] = R4<float>{g[0], g[1], g[2], p};
  }
  if (!GATHER) {
    double bsum = block_sum<256>(e);
    if (threadIdx.x == 0) partial[lin] = bsum;
  }
}

template <int ORDER, typename OUT>
__device__ __forceinline__ void interp_fwd_call(const InterpKArgs<float, OUT>& K, int bx, int by, int bz, int lin) {
  interp_fwd_body<ORDER, OUT>(K.gfrac, K.gbase, K.perm, K.cell_start, K.AA, K.u0, K.G, K.A, K.phis, K.fs, K.glong,
                              K.phi_out, K.force_out, K.partial, bx, by, bz, lin);
}

template <int ORDER>
__global__ void __launch_bounds__(256, 3) k_interp_gather(const R4<float>* __restrict__ gfrac,
                                                          const int4* __restrict__ gbase,
                                                          const int* __restrict__ cell_start, AnterpArgs AA,
                                                          const float* __restrict__ u0, GridDims G, AssembleArgs A,
                                                          R4<float>* __restrict__ glong) {
  pdl_sync();
  interp_fwd_body<ORDER, double, true>(gfrac, gbase, nullptr, cell_start, AA, u0, G, A, nullptr, nullptr, glong,
                                       nullptr, nullptr, nullptr, blockIdx.x, blockIdx.y, blockIdx.z, 0);
}

// FP64 plans: one thread per atom, taps read through the cache (the FP64
// instructions, two lanes per SM and clock, are the bound: ~300 per atom for
// the cubic, ~850 for the quintic basis).  Staged patches ran in 8 to 27
// blocks on small systems (141 us at 3,000 and 23,558 atoms).
template <int ORDER>
__global__ void __launch_bounds__(kWide) k_interp_gather64(const R4<double>* __restrict__ gfrac,
                                                          const int4* __restrict__ gbase, int n,
                                                          const double* __restrict__ u0, GridDims G, AssembleArgs A,
                                                          R4<double>* __restrict__ glong) {
  pdl_sync();
  const int i = blockIdx.x * kWide + threadIdx.x;
  if (i >= n) return;
  double p, g[3];
  interp_atom<double, ORDER>(gfrac[i], gbase[i], u0, G, A.inv_h, p, g);
  glong[i] = R4<double>{g[0], g[1], g[2], p};
}

// The energy from the blocks' partials, by the block that finishes last (ticket:
// one counter, back to 0 afterwards), in a fixed order: thread t takes partials
// t, t + 256, ...
__device__ __forceinline__ void energy_by_last_block(double bsum, double* __restrict__ partial, int* ticket,
                                                     double* __restrict__ energy) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = bsum;
    __threadfence();
    last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double v = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += 256) v += __ldcg(partial + i);
  const double s = block_sum<256>(v);
  if (threadIdx.x == 0) {
    *energy = 0.5 * s;
    *ticket = 0;
  }
}

// An atom's short-range sums: on the FP64 plan its own and the two of the pairs
// that other atoms evaluated.
__device__ __forceinline__ R4<float> short_sums(const R4<float>* fs, const R4<double>*, int64_t i) { return fs[i]; }
__device__ __forceinline__ R4<double> short_sums(const R4<double>* fs, const R4<double>* react, int64_t i) {
  const R4<double> a = fs[i], n = react[2 * i], f = react[2 * i + 1];
  return R4<double>{a.x + (n.x + f.x), a.y + (n.y + f.y), a.z + (n.z + f.z), a.w + (n.w + f.w)};
}

// The short-range potential: an array of its own on the mixed plan, beside the
// force on the FP64 plan.
__device__ __forceinline__ float short_phi(const float* phis, int64_t i, const R4<float>&) { return phis[i]; }
__device__ __forceinline__ double short_phi(const double*, int64_t, const R4<double>& s) { return s.w; }

// Assembly after the pair sums and the gather: phi_i, F_i in the caller's
// order and the per-block energy partials (grid-stride over sorted atoms).
template <typename T, typename OUT>
__global__ void __launch_bounds__(256) k_interp_assemble(int64_t n, const int* __restrict__ perm,
                                                         const R4<T>* __restrict__ gfrac, const T* __restrict__ phis,
                                                         const R4<T>* __restrict__ fs,
                                                         const R4<double>* __restrict__ react,
                                                         const R4<T>* __restrict__ glong, AssembleArgs A,
                                                         OUT* __restrict__ phi_out, OUT* __restrict__ force_out,
                                                         double* __restrict__ partial, int* ticket,
                                                         double* __restrict__ energy) {
  pdl_sync();
  double e = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const R4<T> gl = glong[i];
    const T g[3] = {gl.x, gl.y, gl.z};
    const R4<T> s = short_sums(fs, react, i);
    e += Assemble<T>::forward(A, gfrac[i].w, short_phi(phis, i, s), gl.w, s, g, perm[i], phi_out, force_out);
  }
  const double bsum = block_sum<256>(e);
  __syncthreads();  // block_sum's buffer is used again by the last block
  energy_by_last_block(bsum, partial, ticket, energy);
}

__device__ __forceinline__ void energy_final_body(const double* __restrict__ partial, int nb,
                                                  double* __restrict__ energy) {
  double v = 0.0;
  for (int i = threadIdx.x; i < nb; i += 1024) v += partial[i];
  double s = block_sum<1024>(v);
  if (threadIdx.x == 0) *energy = 0.5 * s;
}

__global__ void __launch_bounds__(1024) k_energy_final(const double* __restrict__ partial, int nb,
                                                       double* __restrict__ energy) {
  pdl_sync();
  energy_final_body(partial, nb, energy);
}

// adjoint assembly: av0 = M (anterpolated 1/2 gE q) on the grid
template <int ORDER, typename OUT>
__device__ __forceinline__ void interp_bwd_body(
    const R4<float>* __restrict__ gfrac, const int4* __restrict__ gbase, const int* __restrict__ perm,
    const int* __restrict__ cell_start, const AnterpArgs& AA, const float* __restrict__ av0, const GridDims& G,
    const AssembleArgs& A, const float* __restrict__ phis, const R4<float>* __restrict__ fs,
    const R4<float>* __restrict__ glong, const double* __restrict__ gE, OUT* __restrict__ grad_pos,
    OUT* __restrict__ grad_q, int bx, int by, int bz) {
  constexpr int S = Basis<float, ORDER>::S;
  extern __shared__ unsigned char smem_raw[];
  float* patch = reinterpret_cast<float*>(smem_raw);
  __shared__ int list[kAnterpMaxAtoms + 32];  // + one round of slots
  __shared__ BlockAtoms R;
  const int lo0 = (int)floor(bx * AA.B * AA.cw_h[0]) - S - 1;
  const int lo1 = (int)floor(by * AA.B * AA.cw_h[1]) - S - 1;
  const int lo2 = (int)floor(bz * AA.B * AA.cw_h[2]) - S - 1;
  const int total =
      stage_interp_block(AA, cell_start, gbase, av0, G, patch, lo0, lo1, lo2, R, list, bx, by, bz);
  const float ih[3] = {(float)A.inv_h[0], (float)A.inv_h[1], (float)A.inv_h[2]};
  const float gg = (float)*gE;
  const int nlist = total >= 0 ? total : R.pre[kBlockRows];
  for (int kk = threadIdx.x; kk < nlist; kk += blockDim.x) {
    const int i = total >= 0 ? list[kk] : block_atom(R, kk);
    if (i < 0) continue;  // unfilled slot of the bank-ordered list
    const R4<float> f = gfrac[i];
    float v, gv[3];
    interp_patch_atom<float, ORDER>(f, gbase[i], patch, AA.pd, lo0, lo1, lo2, av0, G, ih, v, gv);
    Assemble<float>::backward(A, gg, f.w, phis[i], fs[i], glong[i], v, gv, perm[i], grad_pos, grad_q);
  }
}

template <int ORDER, typename OUT>
__device__ __forceinline__ void interp_bwd_call(const InterpKArgs<float, OUT>& K, int bx, int by, int bz) {
  interp_bwd_body<ORDER, OUT>(K.gfrac, K.gbase, K.perm, K.cell_start, K.AA, K.u0, K.G, K.A, K.phis, K.fs, K.glong,
                              K.gE, K.grad_pos, K.grad_q, bx, by, bz);
}

template <int ORDER, typename OUT>
__global__ void __launch_bounds__(256, 3) k_interp_bwd(
    const R4<float>* __restrict__ gfrac, const int4* __restrict__ gbase, const int* __restrict__ perm,
    const int* __restrict__ cell_start, AnterpArgs AA, const float* __restrict__ av0, GridDims G, AssembleArgs A,
    const float* __restrict__ phis, const R4<float>* __restrict__ fs, const R4<float>* __restrict__ glong,
    const double* __restrict__ gE, OUT* __restrict__ grad_pos, OUT* __restrict__ grad_q) {
  pdl_sync();
  interp_bwd_body<ORDER, OUT>(gfrac, gbase, perm, cell_start, AA, av0, G, A, phis, fs, glong, gE, grad_pos, grad_q,
                              blockIdx.x, blockIdx.y, blockIdx.z);
}

// FP64 plans: one thread per atom, as k_interp_gather64
template <int ORDER, typename OUT>
__global__ void __launch_bounds__(kWide) k_interp_bwd64(
    const R4<double>* __restrict__ gfrac, const int4* __restrict__ gbase, const int* __restrict__ perm, int n,
    const double* __restrict__ av0, GridDims G, AssembleArgs A,
    const R4<double>* __restrict__ fs, const R4<double>* __restrict__ react, const R4<double>* __restrict__ glong,
    const double* __restrict__ gE, OUT* __restrict__ grad_pos, OUT* __restrict__ grad_q) {
  pdl_sync();
  const int i = blockIdx.x * kWide + threadIdx.x;
  if (i >= n) return;
  const R4<double> f = gfrac[i];
  double v, gv[3];
  interp_atom<double, ORDER>(f, gbase[i], av0, G, A.inv_h, v, gv);
  const R4<double> s = short_sums(fs, react, i);
  Assemble<double>::backward(A, *gE, f.w, s.w, s, glong[i], v, gv, perm[i], grad_pos, grad_q);
}

template <typename T>
__global__ void k_to_double(const T* __restrict__ src, double* __restrict__ dst, int64_t count) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) dst[i] = (double)src[i];
}

GridDims dims_of(const Plan& P, int k) {
  GridDims G;
  for (int d = 0; d < 3; ++d) {
    G.n[d] = P.n[k][d];
    G.lo[d] = P.lo[k][d];
  }
  G.periodic = P.P.periodic;
  return G;
}

AssembleArgs assemble_args(const Plan& P) {
  AssembleArgs A;
  A.self_c = P.gamma0 / P.P.cutoff;
  A.kc = P.P.coulomb_k;
  for (int d = 0; d < 3; ++d) A.inv_h[d] = 1.0 / P.h[d];
  A.self_cf = (float)A.self_c;
  A.kcf = (float)A.kc;
  return A;
}

unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

// batch: the patch of the batched launches (replicas fill the GPU together,
// so they keep the larger patch that a small system alone gives up)
AnterpArgs patch_args(const Plan& P, bool batch = false) {
  AnterpArgs A;
  for (int d = 0; d < 3; ++d) {
    A.nc[d] = P.nc[d];
    A.cw_h[d] = P.cw[d] / P.h[d];
  }
  A.B = batch ? P.ablk_batch : P.ablk;
  A.pd = batch ? P.apd_batch : P.apd;
  return A;
}

// Threads per anterpolation block: the patch leaves room for two blocks per SM
// (512 threads: 1.07M atoms 166 -> 148 us against 256) or, beyond 100 KB, for
// one (1,024 threads: 4.1M atoms 1,175 -> 907 us).
static int anterp_threads(size_t patch_bytes) { return patch_bytes > 100 * 1024 ? 1024 : 512; }

// Mixed precision: patch sums into the fixed-point grid (in the restriction
// temporary tmp[0], free until the first restriction pass, zeroed by the binning), then one
// conversion to the FP64 level-0 grid that applies the scale.
template <int ORDER>
void anterp_fx(Plan& P, int64_t n, void* grid0, const double* dscale, double factor, cudaStream_t st) {
  const int64_t np = grid_points(P, 0);
  auto* gfx = (unsigned long long*)P.d.tmp[0];
  P.launches += 1;
  if (n > 0) {
    AnterpArgs A = patch_args(P);
    dim3 grid(blocks_for(P.nc[0], A.B), blocks_for(P.nc[1], A.B), blocks_for(P.nc[2], A.B));
    size_t sm = 2 * sizeof(int) * (size_t)A.pd * A.pd * A.pd;  // coarse and residual sums
    klaunch(false, k_anterp_fx<ORDER>, grid, anterp_threads(sm), sm, st, (const R4<float>*)P.d.gfrac, P.d.gbase, P.d.cell_start, A,
                                              dims_of(P, 0), gfx);
    P.launches += 1;
  }
  klaunch(P.pdl, k_fx_to_f64, blocks_for(np, 256), 256, 0, st, gfx, (double*)grid0, np, dscale, factor);
}

cudaError_t launch_anterpolate(Plan& P, int64_t n, void* grid0, const double* dscale, double factor,
                               cudaStream_t st) {
  if (!P.fp64) {
    if (P.P.order == 3) anterp_fx<3>(P, n, grid0, dscale, factor, st);
    else anterp_fx<5>(P, n, grid0, dscale, factor, st);
    return cudaGetLastError();
  }
  if (n <= 0) return cudaGetLastError();
  P.launches += 1;
  const int stride = (int)((n + 31) / 32);
  const unsigned nb = blocks_for((int64_t)32 * stride, kWide);
  const R4<double>* f = (const R4<double>*)P.d.gfrac;
  if (P.P.order == 3)
    klaunch(false, k_anterp64<3>, nb, kWide, 0, st, f, P.d.gbase, (int)n, stride, dims_of(P, 0), (double*)grid0, dscale, factor);
  else
    klaunch(false, k_anterp64<5>, nb, kWide, 0, st, f, P.d.gbase, (int)n, stride, dims_of(P, 0), (double*)grid0, dscale, factor);
  return cudaGetLastError();
}

// dst = factor * dscale[0] * src over the level-0 grid (FP64)
__global__ void k_scale_grid(const double* __restrict__ src, double* __restrict__ dst, int64_t count,
                             const double* __restrict__ dscale, double factor) {
  pdl_sync();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  dst[i] = src[i] * (factor * *dscale);
}

cudaError_t launch_scale_grid(Plan& P, const void* src, void* dst, const double* dscale, double factor,
                              cudaStream_t st) {
  P.launches += 1;
  const int64_t np = grid_points(P, 0);
  klaunch(false, k_scale_grid, blocks_for(np, 256), 256, 0, st, (const double*)src, (double*)dst, np, dscale, factor);
  return cudaGetLastError();
}

// Whether a level's restriction runs by tiles (one launch) or as three axis
// passes: up to 24^3 coarse points, where the launches are the cost (16^3
// coarse points, cubic: 14 -> 5 us; 48^3, quintic: 25 us by passes, FP64-bound
// at about twice that by tiles).
static bool restrict_by_tiles(int64_t coarse_points) { return coarse_points <= 24 * 24 * 24; }
// Prolongation tiles: 8 planes a side once the blocks fill the GPU many times over.
static int prolong_tyz(int64_t fine_points) { return fine_points > ((int64_t)1 << 18) ? 8 : 4; }
static int64_t restrict_tiles(const int* n) {
  return (int64_t)((n[0] + kTileC - 1) / kTileC) * ((n[1] + kTileC - 1) / kTileC) * ((n[2] + kTileC - 1) / kTileC);
}
static int64_t prolong_tiles(const int* n, int tyz) {
  return (int64_t)((n[0] + kTileX - 1) / kTileX) * ((n[1] + tyz - 1) / tyz) * ((n[2] + tyz - 1) / tyz);
}

static Grid3Args grid3_args(const Plan& P, int kin, int kout) {
  Grid3Args A;
  for (int d = 0; d < 3; ++d) {
    A.nin[d] = P.n[kin][d];
    A.nout[d] = P.n[kout][d];
    A.lo_in[d] = P.lo[kin][d];
    A.lo_out[d] = P.lo[kout][d];
  }
  A.periodic = P.P.periodic;
  return A;
}

cudaError_t launch_restrict(Plan& P, int k, const void* fine, void* coarse, cudaStream_t st) {
  const int* nf = P.n[k];
  const int* nc = P.n[k + 1];
  const int64_t ncp = (int64_t)nc[0] * nc[1] * nc[2];
  if (restrict_by_tiles(ncp)) {
    P.launches += 1;
    const Grid3Args A = grid3_args(P, k, k + 1);
    const unsigned nb = (unsigned)restrict_tiles(nc);
    if (P.P.order == 3) klaunch(P.pdl, k_restrict_tile<3>, nb, 256, 0, st, (const double*)fine, (double*)coarse, A);
    else klaunch(P.pdl, k_restrict_tile<5>, nb, 256, 0, st, (const double*)fine, (double*)coarse, A);
    return cudaGetLastError();
  }
  P.launches += 3;
  double* t1 = (double*)P.d.tmp[0];
  double* t2 = (double*)P.d.tmp[1];
  const double* src[3] = {(const double*)fine, t1, t2};
  double* dst[3] = {t1, t2, (double*)coarse};
  int cur[3] = {nf[0], nf[1], nf[2]};
  for (int ax = 0; ax < 3; ++ax) {
    AxisArgs A;
    for (int d = 0; d < 3; ++d) A.nin[d] = cur[d];
    cur[ax] = nc[ax];
    for (int d = 0; d < 3; ++d) A.nout[d] = cur[d];
    A.axis = ax;
    A.lo_in = P.lo[k][ax];
    A.lo_out = P.lo[k + 1][ax];
    A.periodic = P.P.periodic;
    unsigned nb = blocks_for((int64_t)cur[0] * cur[1] * cur[2], 256);
    if (P.P.order == 3) klaunch(P.pdl, k_restrict_axis<double, 3>, nb, 256, 0, st, src[ax], dst[ax], A);
    else klaunch(P.pdl, k_restrict_axis<double, 5>, nb, 256, 0, st, src[ax], dst[ax], A);
  }
  return cudaGetLastError();
}

template <typename T, int TYZ>
static void prolong_t(Plan& P, int k, const T* coarse, T* fine, cudaStream_t st) {
  const Grid3Args A = grid3_args(P, k + 1, k);
  const unsigned nb = (unsigned)prolong_tiles(P.n[k], TYZ);
  if (P.P.order == 3) klaunch(P.pdl, k_prolong_tile<T, 3, TYZ>, nb, 256, 0, st, coarse, fine, A);
  else klaunch(P.pdl, k_prolong_tile<T, 5, TYZ>, nb, 256, 0, st, coarse, fine, A);
}

cudaError_t launch_prolong(Plan& P, int k, const void* coarse, void* fine, cudaStream_t st) {
  P.launches += 1;
  const bool big = prolong_tyz(grid_points(P, k)) == 8;
  if (P.fp64) {
    if (big) prolong_t<double, 8>(P, k, (const double*)coarse, (double*)fine, st);
    else prolong_t<double, 4>(P, k, (const double*)coarse, (double*)fine, st);
  } else {
    if (big) prolong_t<float, 8>(P, k, (const float*)coarse, (float*)fine, st);
    else prolong_t<float, 4>(P, k, (const float*)coarse, (float*)fine, st);
  }
  return cudaGetLastError();
}

__device__ __forceinline__ void f64_to_f32_body(const double* __restrict__ src, float* __restrict__ dst,
                                                int64_t count, int64_t i) {
  if (i < count) dst[i] = (float)src[i];
}

__global__ void k_f64_to_f32(const double* __restrict__ src, float* __restrict__ dst, int64_t count) {
  pdl_sync();
  f64_to_f32_body(src, dst, count, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// Warp tile of the FP32 lattice kernel for an n0 x n1 plane: txn lanes of
// kLatticeLP x outputs by tyn lanes of two rows (txn * tyn <= 32).  Every
// tile costs one warp's pass over the stencil whatever its idle lanes, plus
// the staging of its input window; the cost counts both (a warp's stencil
// pass at a plane is ~14,000 instructions, staging ~1/3 instruction per
// window element), so ragged small grids get tiles that fit them.
static size_t lattice_smem(int txn, int tyn, const int E[3]);

static void lattice_tile(int n0, int n1, const int E[3], int& txn, int& tyn) {
  double best = -1.0;
  txn = 4;
  tyn = 8;
  for (int a = 1; a <= 32; ++a)
    for (int b = 1; a * b <= 32; ++b) {
      if (lattice_smem(a, b, E) > kLatticeSmemMax) continue;
      const double tiles = (double)((n0 + kLatticeLP * a - 1) / (kLatticeLP * a)) * ((n1 + 2 * b - 1) / (2 * b));
      const double window = (double)(kLatticeLP * a + 2 * E[0] + kSeg) * (2 * b + 2 * E[1]);
      const double cost = tiles * (14000.0 + window / 3.0);
      if (best < 0 || cost < best) {
        best = cost;
        txn = a;
        tyn = b;
      }
    }
}

static size_t lattice_smem(int txn, int tyn, const int E[3]) {
  const int SXw = kLatticeLP * txn + 2 * E[0] + kSeg, SX = SXw | 1, SY = 2 * tyn + 2 * E[1];
  return sizeof(float) * 2 * SX * SY + sizeof(int) * (SXw + SY);
}

// Lattice cutoff of level k by the stencil from the FP64 charges qk.
static void lattice_fp64(Plan& P, int k, const double* qk, double* uk, cudaStream_t st) {
  const GridDims G = dims_of(P, k);
  const int64_t np = grid_points(P, k);
  const int ns = lattice_nsplit(P, k), per = (P.nlrows + ns - 1) / ns;
  double* up = (double*)P.d.lparts;
  dim3 grid(blocks_for(np, kLat64), ns);
  const double scale = std::ldexp(1.0, -k);
  const double* coef = (const double*)P.d.seg;
  if (G.periodic) klaunch(P.pdl, k_lattice64<true>, grid, kLat64, 0, st, qk, uk, up, G, P.d.lrows, coef, P.nlrows, per, scale);
  else klaunch(P.pdl, k_lattice64<false>, grid, kLat64, 0, st, qk, uk, up, G, P.d.lrows, coef, P.nlrows, per, scale);
  if (ns > 1) {
    klaunch(P.pdl, k_lattice_reduce<double>, blocks_for(np, 256), 256, 0, st, up, uk, np, ns);
    P.launches += 1;
  }
}

// The same on the mixed plan, which first converts the level's charges to
// FP32 once (the conversion runs on the slow FP64 pipe, so it must not sit in
// the per-tap loop).
static void lattice_fp32(Plan& P, int k, const double* qk64, float* uk, cudaStream_t st) {
  GridDims G = dims_of(P, k);
  float* qk = (float*)P.d.tmp[0];  // free between the restriction and the prolongation passes
  klaunch(P.pdl, k_f64_to_f32, blocks_for(grid_points(P, k), 256), 256, 0, st, qk64, qk, grid_points(P, k));
  P.launches += 1;
  LatticeArgs L;
  L.Ex = P.E[0];
  L.Ey = P.E[1];
  L.Ez = P.E[2];
  // one system: the 32 x 16 tile, fixed at compile time, on every level (the
  // runtime-tile kernel is slower per tap than the saving on ragged coarse
  // levels), unless the plan's tuning names another tile for level 0
  lattice_tile_of(P, k, L.txn, L.tyn);
  L.nbz = (int)blocks_for(G.n[2], kLatticeZ);
  L.nsplit = lattice_nsplit(P, k);
  float* up = (float*)P.d.lparts;
  dim3 grid(blocks_for(G.n[0], kLatticeLP * L.txn), blocks_for(G.n[1], 2 * L.tyn), L.nbz * L.nsplit);
  // double-buffered planes and the window offsets (SXw + SY ints)
  const size_t sm = lattice_smem(L.txn, L.tyn, P.E);
  const float scale = (float)std::ldexp(1.0, -k);
  if (L.txn == 4 && L.tyn == 8)
    klaunch(P.pdl, k_lattice_f2<kLatticeLP, 4, 8>, grid, 32 * kLatticeZ, sm, st, qk, uk, up, G, (const Segment2*)P.d.seg2,
                                                                    P.d.seg_start, L, scale);
  else
    klaunch(P.pdl, k_lattice_f2<kLatticeLP, 0, 0>, grid, 32 * kLatticeZ, sm, st, qk, uk, up, G, (const Segment2*)P.d.seg2,
                                                                    P.d.seg_start, L, scale);
  if (L.nsplit > 1) {
    const int64_t np = grid_points(P, k);
    klaunch(P.pdl, k_lattice_reduce<float>, blocks_for(np, 256), 256, 0, st, up, uk, np, L.nsplit);
    P.launches += 1;
  }
}

// Warp tile of the FP32 lattice kernel at level k of a single system: the
// plan's tuned tile on level 0, else 4 x 8 (32 x 16 outputs).
void lattice_tile_of(const Plan& P, int k, int& txn, int& tyn) {
  if (k == 0 && P.lattice_txn > 0) {
    txn = P.lattice_txn;
    tyn = P.lattice_tyn;
  } else {
    txn = 4;
    tyn = 8;
  }
}

// Blocks that share one brick's input planes (FP64: one output's stencil rows)
// at level k: several on small levels, so that the launch still fills the GPU
// (lattice_waves blocks per SM; FP64: 16 warps per SM).
int lattice_nsplit(const Plan& P, int k) {
  if (P.fp64) {
    const int64_t warps = blocks_for(grid_points(P, k), 32);
    return (int)std::min<int64_t>(std::max(P.nlrows, 1), std::max<int64_t>(1, (152 * 16 + warps / 2) / warps));
  }
  GridDims G = dims_of(P, k);
  int txn, tyn;
  lattice_tile_of(P, k, txn, tyn);
  const int64_t bricks = (int64_t)blocks_for(G.n[0], kLatticeLP * txn) * blocks_for(G.n[1], 2 * tyn) *
                         blocks_for(G.n[2], kLatticeZ);
  const int64_t target = (int64_t)P.lattice_waves * 152 * 4 / kLatticeZ;
  return (int)std::min<int64_t>(kLatticeZ + 2 * P.E[2], std::max<int64_t>(1, (target + bricks - 1) / bricks));
}

// Elements of the plan's split-partial buffer: the largest nsplit x points of
// any level whose lattice cutoff is split.
int64_t lattice_parts_elems(const Plan& P) {
  int64_t m = 0;
  for (int k = 0; k + 1 < P.levels; ++k) {
    const int ns = lattice_nsplit(P, k);
    if (ns > 1) m = std::max<int64_t>(m, (int64_t)ns * grid_points(P, k));
  }
  return m;
}

// The FP64 kernel needs no shared memory; the line is that of the stencils its
// plans accept (2a/h up to about 27 spacings), as its 48 KB window once set it.
bool lattice_fits(const Plan& P) {
  if (P.fp64) {
    const int SX = (LBX + 2 * P.E[0] + kSeg) | 1, SY = 8 + 2 * P.E[1];
    return sizeof(double) * SX * SY <= 48 * 1024;
  }
  return lattice_smem(4, 8, P.E) <= kLatticeSmemMax;
}

bool lattice_tile_fits(const Plan& P, int txn, int tyn) {
  return P.fp64 || lattice_smem(txn, tyn, P.E) <= kLatticeSmemMax;
}

cudaError_t launch_lattice(Plan& P, int k, const void* qk, void* uk, cudaStream_t st) {
  P.launches += 1;
  if (P.fp64) lattice_fp64(P, k, (const double*)qk, (double*)uk, st);
  else lattice_fp32(P, k, (const double*)qk, (float*)uk, st);
  return cudaGetLastError();
}

cudaError_t launch_top(Plan& P, const void* qt, void* ut, cudaStream_t st) {
  P.launches += 1;
  int top = P.levels - 1;
  GridDims G = dims_of(P, top);
  unsigned nb = blocks_for(grid_points(P, top), kTopWarps);
  if (P.fp64)
    klaunch(P.pdl, k_top<double>, nb, 32 * kTopWarps, 0, st, (const double*)qt, (double*)ut, P.d.topu, G, P.d.topK,
                                     P.top_table_dims[0], P.top_table_dims[1], P.top_table_dims[2]);
  else
    klaunch(P.pdl, k_top<float>, nb, 32 * kTopWarps, 0, st, (const double*)qt, (float*)ut, P.d.topu, G, P.d.topK,
                                    P.top_table_dims[0], P.top_table_dims[1], P.top_table_dims[2]);
  return cudaGetLastError();
}


#define INTERP_BWD_ARGS(K) \
  K.gfrac, K.gbase, K.perm, K.cell_start, K.AA, K.u0, K.G, K.A, K.phis, K.fs, K.glong, K.gE, K.grad_pos, K.grad_q

// Interpolation arguments of plan P (forward: grid u^0; backward: the adjoint grid).
template <typename T, typename OUT>
InterpKArgs<T, OUT> interp_kargs(Plan& P, bool backward, OUT* phi, OUT* force, const double* gE, OUT* grad_pos,
                                 OUT* grad_q, double* partial, bool batch = false) {
  InterpKArgs<T, OUT> K;
  K.gfrac = (const R4<T>*)P.d.gfrac;
  K.gbase = P.d.gbase;
  K.perm = P.d.perm;
  K.cell_start = P.d.cell_start;
  K.AA = patch_args(P, batch);
  K.u0 = (const T*)(backward ? P.d.au[0] : P.d.gu[0]);
  K.G = dims_of(P, 0);
  K.A = assemble_args(P);
  K.phis = (const T*)P.d.phis;
  K.fs = (R4<T>*)P.d.fs;
  K.glong = (R4<T>*)P.d.glong;
  K.phi_out = phi;
  K.force_out = force;
  K.partial = partial;
  K.gE = gE;
  K.grad_pos = grad_pos;
  K.grad_q = grad_q;
  K.nbx = (int)blocks_for(P.nc[0], K.AA.B);
  K.nby = (int)blocks_for(P.nc[1], K.AA.B);
  return K;
}

cudaError_t launch_interp_gather(Plan& P, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const GridDims G = dims_of(P, 0);
  const AssembleArgs A = assemble_args(P);
  P.launches += 1;
  if (P.fp64) {
    const unsigned nb = blocks_for(n, kWide);
    const R4<double>* f = (const R4<double>*)P.d.gfrac;
    const double* u = (const double*)P.d.gu[0];
    if (P.P.order == 3) klaunch(P.pdl, k_interp_gather64<3>, nb, kWide, 0, st, f, P.d.gbase, (int)n, u, G, A, (R4<double>*)P.d.glong);
    else klaunch(P.pdl, k_interp_gather64<5>, nb, kWide, 0, st, f, P.d.gbase, (int)n, u, G, A, (R4<double>*)P.d.glong);
    return cudaGetLastError();
  }
  AnterpArgs AA = patch_args(P);
  dim3 grid(blocks_for(P.nc[0], AA.B), blocks_for(P.nc[1], AA.B), blocks_for(P.nc[2], AA.B));
  size_t sm = sizeof(float) * (size_t)AA.pd * AA.pd * AA.pd;
  const R4<float>* f = (const R4<float>*)P.d.gfrac;
  const float* u = (const float*)P.d.gu[0];
  if (P.P.order == 3)
    klaunch(P.pdl, k_interp_gather<3>, grid, 256, sm, st, f, P.d.gbase, P.d.cell_start, AA, u, G, A, (R4<float>*)P.d.glong);
  else
    klaunch(P.pdl, k_interp_gather<5>, grid, 256, sm, st, f, P.d.gbase, P.d.cell_start, AA, u, G, A, (R4<float>*)P.d.glong);
  return cudaGetLastError();
}

template <typename OUT>
cudaError_t launch_interp_assemble(Plan& P, int64_t n, double* energy, OUT* phi, OUT* force, cudaStream_t st) {
  const int nb = (int)std::max<int64_t>(0, std::min<int64_t>(P.nblk_partial, (n + 255) / 256));
  const AssembleArgs A = assemble_args(P);
  if (nb > 0) {
    if (P.fp64)
      klaunch(false, k_interp_assemble<double, OUT>, nb, 256, 0, st, n, P.d.perm, (const R4<double>*)P.d.gfrac,
                                                        (const double*)P.d.phis, (const R4<double>*)P.d.fs,
                                                        (const R4<double>*)P.d.react,
                                                        (const R4<double>*)P.d.glong, A, phi, force, P.d.partial,
                                                        P.d.ticket, energy);
    else
      klaunch(false, k_interp_assemble<float, OUT>, nb, 256, 0, st, n, P.d.perm, (const R4<float>*)P.d.gfrac,
                                                       (const float*)P.d.phis, (const R4<float>*)P.d.fs, nullptr,
                                                       (const R4<float>*)P.d.glong, A, phi, force, P.d.partial,
                                                        P.d.ticket, energy);
  }
  if (nb == 0) klaunch(false, k_energy_final, 1, 1024, 0, st, P.d.partial, nb, energy);
  P.launches += 1;
  return cudaGetLastError();
}

template cudaError_t launch_interp_assemble<double>(Plan&, int64_t, double*, double*, double*, cudaStream_t);
template cudaError_t launch_interp_assemble<float>(Plan&, int64_t, double*, float*, float*, cudaStream_t);

template <typename OUT>
cudaError_t launch_interp_backward(Plan& P, int64_t n, const double* gE, OUT* grad_pos, OUT* grad_q,
                                   cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  P.launches += 1;
  if (P.fp64) {
    const unsigned nb = blocks_for(n, kWide);
    const auto K = interp_kargs<double, OUT>(P, true, nullptr, nullptr, gE, grad_pos, grad_q, nullptr);
    if (P.P.order == 3)
      klaunch(P.pdl, k_interp_bwd64<3, OUT>, nb, kWide, 0, st, K.gfrac, K.gbase, K.perm, (int)n, K.u0, K.G, K.A, K.fs,
              (const R4<double>*)P.d.react, K.glong, gE, grad_pos, grad_q);
    else
      klaunch(P.pdl, k_interp_bwd64<5, OUT>, nb, kWide, 0, st, K.gfrac, K.gbase, K.perm, (int)n, K.u0, K.G, K.A, K.fs,
              (const R4<double>*)P.d.react, K.glong, gE, grad_pos, grad_q);
    return cudaGetLastError();
  }
  const auto K = interp_kargs<float, OUT>(P, true, nullptr, nullptr, gE, grad_pos, grad_q, nullptr);
  dim3 grid(K.nbx, K.nby, blocks_for(P.nc[2], K.AA.B));
  size_t sm = sizeof(float) * (size_t)K.AA.pd * K.AA.pd * K.AA.pd;
  if (P.P.order == 3) klaunch(P.pdl, k_interp_bwd<3, OUT>, grid, 256, sm, st, INTERP_BWD_ARGS(K));
  else klaunch(P.pdl, k_interp_bwd<5, OUT>, grid, 256, sm, st, INTERP_BWD_ARGS(K));
  return cudaGetLastError();
}


template cudaError_t launch_interp_backward<double>(Plan&, int64_t, const double*, double*, double*, cudaStream_t);
template cudaError_t launch_interp_backward<float>(Plan&, int64_t, const double*, float*, float*, cudaStream_t);

cudaError_t launch_grid_to_double(Plan& P, const void* src, double* dst, int64_t count, bool is_double,
                                  cudaStream_t st) {
  unsigned nb = blocks_for(count, 256);
  if (count <= 0) return cudaSuccess;
  if (P.fp64 || is_double) klaunch(false, k_to_double<double>, nb, 256, 0, st, (const double*)src, dst, count);
  else klaunch(false, k_to_double<float>, nb, 256, 0, st, (const float*)src, dst, count);
  return cudaGetLastError();
}


// ---- the cutoff method: assembly of phi, F and E from the pair sums ----
// phi_i = k_c u_i, F_i = k_c (pair forces), E = 1/2 k_c sum_i q_i u_i; per-block
// FP64 partials (grid-stride over the sorted atoms) and k_energy_final.
template <typename T, typename OUT>
__global__ void __launch_bounds__(256) k_cutoff_assemble(int64_t n, const int* __restrict__ perm,
                                                         const R4<T>* __restrict__ atoms, const T* __restrict__ phis,
                                                         const R4<T>* __restrict__ fs, T kc, T selfc, OUT* __restrict__ phi_out,
                                                         OUT* __restrict__ force_out, double* __restrict__ partial,
                                                         int* ticket, double* __restrict__ energy) {
  pdl_sync();
  double e = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const R4<T> f = fs[i];
    const T p = short_phi(phis, i, f) - selfc * atoms[i].w;  // selfc: the method's self term (0 for the cutoff method)
    const int o = perm[i];
    if (phi_out) phi_out[o] = (OUT)(kc * p);
    if (force_out) {
      force_out[3 * (size_t)o + 0] = (OUT)(kc * f.x);
      force_out[3 * (size_t)o + 1] = (OUT)(kc * f.y);
      force_out[3 * (size_t)o + 2] = (OUT)(kc * f.z);
    }
    e += (double)(atoms[i].w * (kc * p));
  }
  const double bsum = block_sum<256>(e);
  __syncthreads();  // block_sum's buffer is used again by the last block
  energy_by_last_block(bsum, partial, ticket, energy);
}

template <typename OUT>
cudaError_t launch_cutoff_assemble(Plan& P, int64_t n, double* energy, OUT* phi, OUT* force, cudaStream_t st,
                                   double self_c) {
  const int nb = (int)std::max<int64_t>(0, std::min<int64_t>(P.nblk_partial, (n + 255) / 256));
  if (nb > 0) {
    if (P.fp64)
      klaunch(false, k_cutoff_assemble<double, OUT>, nb, 256, 0, st, n, P.d.perm, (const R4<double>*)P.d.atoms,
                                                        (const double*)P.d.phis, (const R4<double>*)P.d.fs,
                                                        P.P.coulomb_k, self_c, phi, force, P.d.partial, P.d.ticket, energy);
    else
      klaunch(false, k_cutoff_assemble<float, OUT>, nb, 256, 0, st, n, P.d.perm, (const R4<float>*)P.d.atoms,
                                                       (const float*)P.d.phis, (const R4<float>*)P.d.fs,
                                                       (float)P.P.coulomb_k, (float)self_c, phi, force,
                                                       P.d.partial, P.d.ticket, energy);
  }
  if (nb == 0) klaunch(false, k_energy_final, 1, 1024, 0, st, P.d.partial, nb, energy);
  P.launches += 1;
  return cudaGetLastError();
}

template cudaError_t launch_cutoff_assemble<double>(Plan&, int64_t, double*, double*, double*, cudaStream_t, double);
template cudaError_t launch_cutoff_assemble<float>(Plan&, int64_t, double*, float*, float*, cudaStream_t, double);

// ---- batches: every grid pass as one launch over all replicas ----
namespace {

constexpr int kEw = 256;  // threads per block of the batched elementwise kernels

struct ZeroKArgs {
  unsigned* p;
  int64_t words;
};
struct FxKArgs {
  const unsigned long long* gfx;
  double* q0;
  int64_t count;
  const double* dscale;
  double factor;
};
template <typename T>
struct AxisKArgs {
  const T* in;
  T* out;
  AxisArgs A;
  int acc;
};
template <typename T>
struct TileKArgs {
  const T* in;
  T* out;
  Grid3Args A;
};
struct ConvKArgs {
  const double* src;
  float* dst;
  int64_t count;
};
struct AntKArgs {
  const R4<float>* gfrac;
  const int4* gbase;
  const int* cell_start;
  AnterpArgs A;
  GridDims G;
  unsigned long long* gfx;
  int nbx, nby;
};
struct LatKArgs {
  const float* q;
  float* u;
  float* up;  // split partials (nsplit > 1)
  GridDims G;
  const Segment2* seg;
  const int* seg_start;
  LatticeArgs L;
  float scale;
  int nbx, nby;
};
struct TopKArgs {
  const double* qt;
  float* ut;
  double* ut64;
  GridDims G;
  const double* K;
  int tx, ty;
};
struct EnergyKArgs {
  const double* partial;
  int nb;
  double* energy;
};
struct ReduceKArgs {
  const float* up;
  float* u;
  int64_t np;
  int nsplit;
};

__device__ __forceinline__ int64_t ew_index(const int* __restrict__ first, int r) {
  return (int64_t)(blockIdx.x - first[r]) * kEw + threadIdx.x;
}

__global__ void __launch_bounds__(kEw) kb_zero(const ZeroKArgs* __restrict__ tab, const int* __restrict__ first,
                                               int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  const int64_t i = ew_index(first, r);
  if (i < tab[r].words) tab[r].p[i] = 0u;
}

__global__ void __launch_bounds__(kEw) kb_fx_to_f64(const FxKArgs* __restrict__ tab, const int* __restrict__ first,
                                                    int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  const FxKArgs& a = tab[r];
  fx_to_f64_body(a.gfx, a.q0, a.count, a.dscale, a.factor, ew_index(first, r));
}

template <int ORDER>
__global__ void __launch_bounds__(kEw) kb_restrict_axis(const AxisKArgs<double>* __restrict__ tab,
                                                        const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  const AxisKArgs<double>& a = tab[r];
  restrict_axis_body<double, ORDER>(a.in, a.out, a.A, ew_index(first, r));
}

template <int ORDER>
__global__ void __launch_bounds__(256) kb_restrict_tile(const TileKArgs<double>* __restrict__ tab,
                                                        const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  restrict_tile_body<ORDER>(tab[r].in, tab[r].out, tab[r].A, blockIdx.x - first[r]);
}

template <int ORDER>
__global__ void __launch_bounds__(256) kb_prolong_tile(const TileKArgs<float>* __restrict__ tab,
                                                       const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  prolong_tile_body<float, ORDER, 8>(tab[r].in, tab[r].out, tab[r].A, blockIdx.x - first[r]);
}

__global__ void __launch_bounds__(kEw) kb_lattice_reduce(const ReduceKArgs* __restrict__ tab,
                                                         const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  const ReduceKArgs& a = tab[r];
  lattice_reduce_body<float>(a.up, a.u, a.np, a.nsplit, ew_index(first, r));
}

__global__ void __launch_bounds__(kEw) kb_f64_to_f32(const ConvKArgs* __restrict__ tab, const int* __restrict__ first,
                                                     int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  f64_to_f32_body(tab[r].src, tab[r].dst, tab[r].count, ew_index(first, r));
}

template <int ORDER>
__global__ void __launch_bounds__(512, 2) kb_anterp_fx(const AntKArgs* __restrict__ tab, const int* __restrict__ first,
                                                    int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  const AntKArgs& a = tab[r];
  const int b = blockIdx.x - first[r];
  anterp_fx_body<ORDER>(a.gfrac, a.gbase, a.cell_start, a.A, a.G, a.gfx, b % a.nbx, (b / a.nbx) % a.nby,
                        b / (a.nbx * a.nby));
}

__global__ void __launch_bounds__(32 * kLatticeZ, 6) kb_lattice_f2(const LatKArgs* __restrict__ tab,
                                                                   const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  const LatKArgs& a = tab[r];
  const int b = blockIdx.x - first[r];
  lattice_f2_body<kLatticeLP, 0, 0>(a.q, a.u, a.up, a.G, a.seg, a.seg_start, a.L, a.scale, b % a.nbx,
                                    (b / a.nbx) % a.nby, b / (a.nbx * a.nby));
}

__global__ void __launch_bounds__(32 * kTopWarps) kb_top(const TopKArgs* __restrict__ tab,
                                                         const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  const TopKArgs& a = tab[r];
  top_body<float>(a.qt, a.ut, a.ut64, a.G, a.K, a.tx, a.ty,
                  (int64_t)(blockIdx.x - first[r]) * kTopWarps + (threadIdx.x >> 5));
}

template <int ORDER>
__global__ void __launch_bounds__(256, 3) kb_interp_fwd(const InterpKArgs<float, double>* __restrict__ tab,
                                                     const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  const InterpKArgs<float, double>& K = tab[r];
  const int b = blockIdx.x - first[r];
  interp_fwd_call<ORDER, double>(K, b % K.nbx, (b / K.nbx) % K.nby, b / (K.nbx * K.nby), b);
}

template <int ORDER>
__global__ void __launch_bounds__(256, 3) kb_interp_bwd(const InterpKArgs<float, double>* __restrict__ tab,
                                                     const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  const InterpKArgs<float, double>& K = tab[r];
  const int b = blockIdx.x - first[r];
  interp_bwd_call<ORDER, double>(K, b % K.nbx, (b / K.nbx) % K.nby, b / (K.nbx * K.nby));
}

__global__ void __launch_bounds__(1024) kb_energy_final(const EnergyKArgs* __restrict__ tab,
                                                        const int* __restrict__ first, int nrep) {
  const int r = batch_rep(first, nrep, blockIdx.x);
  energy_final_body(tab[r].partial, tab[r].nb, tab[r].energy);
}

int ew_blocks(int64_t count) { return (int)((count + kEw - 1) / kEw); }

}  // namespace

// ---- persistent chains (a measured alternative to one launch per pass) ----
// The restriction and the prolongation of a sweep are chains of small
// dependent passes (three axes per level pair).  A persistent form runs a
// whole chain in one cooperative launch: the co-resident blocks take the
// virtual blocks of each pass in turn (the same tables and element bodies as
// the per-pass launches) and meet at a grid barrier between passes.  The
// barrier is a counter and a generation word in device memory; every wait is
// bounded, and a wait that gives up posts kStatusTimeout and ends its block.
struct PassDesc {
  const void* args;   // the pass's table of per-replica arguments
  const int* first;   // its block offsets
  int nrep;
  int total;          // virtual blocks of kEw elements over all replicas
};
constexpr int kGridSpin = 1 << 22;  // polls of the generation word before a barrier gives up

// All blocks of the grid arrive, the last one releases the others.  bar[0]:
// arrivals of the current barrier, bar[1]: generation.
__device__ bool grid_barrier(unsigned* bar, unsigned nblocks, int* status) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    volatile unsigned* gen = bar + 1;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(bar, 1u) + 1u == nblocks) {
      bar[0] = 0u;  // nobody arrives at the next barrier before the generation moves
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      for (int it = 0; *gen == g; ++it) {
        if (it >= kGridSpin) {
          ok = 0;
          atomicOr(status, kStatusTimeout);
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

template <int ORDER>
__global__ void __launch_bounds__(kEw) kb_restrict_chain(const PassDesc* __restrict__ passes, int npass,
                                                         unsigned* bar, int* status) {
  for (int p = 0; p < npass; ++p) {
    const PassDesc d = passes[p];
    const AxisKArgs<double>* tab = reinterpret_cast<const AxisKArgs<double>*>(d.args);
    for (int b = blockIdx.x; b < d.total; b += gridDim.x) {
      const int r = batch_rep(d.first, d.nrep, b);
      restrict_axis_body<double, ORDER>(tab[r].in, tab[r].out, tab[r].A, (int64_t)(b - d.first[r]) * kEw + threadIdx.x);
    }
    if (p + 1 < npass && !grid_barrier(bar, gridDim.x, status)) return;
  }
}

template <int ORDER>
__global__ void __launch_bounds__(kEw) kb_prolong_chain(const PassDesc* __restrict__ passes, int npass,
                                                        unsigned* bar, int* status) {
  for (int p = 0; p < npass; ++p) {
    const PassDesc d = passes[p];
    const AxisKArgs<float>* tab = reinterpret_cast<const AxisKArgs<float>*>(d.args);
    for (int b = blockIdx.x; b < d.total; b += gridDim.x) {
      const int r = batch_rep(d.first, d.nrep, b);
      prolong_axis_body<float, ORDER>(tab[r].in, tab[r].out, tab[r].A, tab[r].acc,
                                      (int64_t)(b - d.first[r]) * kEw + threadIdx.x);
    }
    if (p + 1 < npass && !grid_barrier(bar, gridDim.x, status)) return;
  }
}

struct GridBatch {
  int order = 3;
  int maxlev = 1;
  bool has_backward = false;
  BatchTable<ZeroKArgs> zero_fx;
  BatchTable<AntKArgs> anterp;
  BatchTable<FxKArgs> fx[2];
  std::vector<BatchTable<AxisKArgs<double>>> restr[2];  // [dir][3 k + axis]
  BatchTable<ConvKArgs> conv[2];
  BatchTable<ReduceKArgs> reduce_u[2];  // split lattice partials -> u, in part order
  float* lparts[2] = {nullptr, nullptr};
  BatchTable<LatKArgs> lattice[2];
  FftBatch* fft[2] = {nullptr, nullptr};  // the FFT form, when every replica's plan took it
  BatchTable<TopKArgs> top[2];
  std::vector<BatchTable<AxisKArgs<float>>> prol[2];  // [dir][3 k + pass] (persistent chains)
  // one launch per level (without persistent chains): restriction where every
  // replica's level is small enough (else the axis passes), prolongation
  std::vector<BatchTable<TileKArgs<double>>> restr_tile[2];
  std::vector<BatchTable<TileKArgs<float>>> prol_tile[2];
  BatchTable<InterpKArgs<float, double>> interp[2];
  BatchTable<EnergyKArgs> energy;
  // persistent chains: pass descriptors of the restriction and prolongation
  // of each direction, barrier words, the status word they post to
  bool persistent = false;
  PassDesc* chain_restr[2] = {nullptr, nullptr};
  PassDesc* chain_prol[2] = {nullptr, nullptr};
  int n_restr = 0, n_prol = 0;
  unsigned* bar = nullptr;
  int* status = nullptr;
  int chain_blocks = 0;
  // the adjoint direction's temporaries, one block per replica
  std::vector<void*> scratch1;
};

void grid_batch_free(GridBatch* b) {
  if (!b) return;
  b->zero_fx.release();
  b->anterp.release();
  for (int d = 0; d < 2; ++d) {
    b->fx[d].release();
    for (auto& t : b->restr[d]) t.release();
    b->conv[d].release();
    b->reduce_u[d].release();
    if (b->lparts[d]) cudaFree(b->lparts[d]);
    b->lattice[d].release();
    fft_batch_free(b->fft[d]);
    b->top[d].release();
    for (auto& t : b->prol[d]) t.release();
    for (auto& t : b->restr_tile[d]) t.release();
    for (auto& t : b->prol_tile[d]) t.release();
    b->interp[d].release();
  }
  b->energy.release();
  for (int d = 0; d < 2; ++d) {
    if (b->chain_restr[d]) cudaFree(b->chain_restr[d]);
    if (b->chain_prol[d]) cudaFree(b->chain_prol[d]);
  }
  if (b->bar) cudaFree(b->bar);
  for (void* p : b->scratch1) cudaFree(p);
  delete b;
}

cudaError_t grid_batch_build(const std::vector<BatchRep>& reps, bool backward, GridBatch** out) {
  *out = nullptr;
  GridBatch* B = new (std::nothrow) GridBatch();
  if (!B) return cudaErrorMemoryAllocation;
  const int R = (int)reps.size();
  B->order = reps.empty() ? 3 : reps[0].plan->P.order;
  B->has_backward = backward;
  const bool chains = !reps.empty() && reps[0].plan->batch_persistent;  // restriction and prolongation
  for (const BatchRep& r : reps) B->maxlev = std::max(B->maxlev, r.plan->levels);
  cudaError_t e = cudaSuccess;
  auto chk = [&](cudaError_t x) {
    if (e == cudaSuccess) e = x;
  };
  {  // anterpolation into the fixed-point grids (tmp[0]); the same kernels for both directions
    std::vector<ZeroKArgs> za;
    std::vector<AntKArgs> aa;
    std::vector<int> zb, ab;
    size_t sm = 0;
    for (const BatchRep& r : reps) {
      Plan& P = *r.plan;
      const int64_t np = grid_points(P, 0);
      za.push_back(ZeroKArgs{(unsigned*)P.d.tmp[0], 2 * np});
      zb.push_back(ew_blocks(2 * np));
      AntKArgs a;
      a.gfrac = (const R4<float>*)P.d.gfrac;
      a.gbase = P.d.gbase;
      a.cell_start = P.d.cell_start;
      a.A = patch_args(P, true);
      a.G = dims_of(P, 0);
      a.gfx = (unsigned long long*)P.d.tmp[0];
      a.nbx = (int)blocks_for(P.nc[0], a.A.B);
      a.nby = (int)blocks_for(P.nc[1], a.A.B);
      aa.push_back(a);
      ab.push_back(r.n > 0 ? a.nbx * a.nby * (int)blocks_for(P.nc[2], a.A.B) : 0);
      sm = std::max(sm, 2 * sizeof(int) * (size_t)a.A.pd * a.A.pd * a.A.pd);
    }
    chk(make_table(B->zero_fx, za, zb));
    chk(make_table(B->anterp, aa, ab, sm));
  }
  // the adjoint direction's own temporaries (restriction and prolongation,
  // the FFT workspace or the stencil's FP32 charges, the top level's FP64
  // values), so that its level chain can run beside the forward's
  struct Scratch {
    void* tmp[2] = {nullptr, nullptr};
    void* fftw = nullptr;
    double* topu = nullptr;
  };
  std::vector<Scratch> S1(reps.size());
  if (backward)
    for (size_t i = 0; i < reps.size() && e == cudaSuccess; ++i) {
      Plan& P = *reps[i].plan;
      size_t lat = 0;
      for (int k = 0; k + 1 < P.levels; ++k) lat += (size_t)grid_points(P, k);
      const size_t tmpb = sizeof(double) * (size_t)P.tmp_elems, fftb = P.lattice_fft ? 16 * lat : 0;
      const size_t topb = sizeof(double) * (size_t)grid_points(P, P.levels - 1);
      char* base = nullptr;
      chk(cudaMalloc((void**)&base, 2 * tmpb + fftb + topb));
      if (e != cudaSuccess) break;
      B->scratch1.push_back(base);
      S1[i].tmp[0] = base;
      S1[i].tmp[1] = base + tmpb;
      S1[i].fftw = base + 2 * tmpb;
      S1[i].topu = reinterpret_cast<double*>(base + 2 * tmpb + fftb);
    }
  for (int dir = 0; dir < (backward ? 2 : 1); ++dir) {
    // this direction's temporaries of replica r
    auto tmp_of = [&](const BatchRep& r, int i) -> void* {
      return dir ? S1[&r - &reps[0]].tmp[i] : r.plan->d.tmp[i];
    };
    std::vector<FxKArgs> fa;
    std::vector<int> fb;
    for (const BatchRep& r : reps) {
      Plan& P = *r.plan;
      const int64_t np = grid_points(P, 0);
      fa.push_back(FxKArgs{(const unsigned long long*)P.d.tmp[0], (double*)(dir ? P.d.aq[0] : P.d.gq[0]), np,
                           dir ? r.grad_energy : nullptr, dir ? 0.5 : 1.0});
      fb.push_back(ew_blocks(np));
    }
    chk(make_table(B->fx[dir], fa, fb));
    // restriction k -> k+1, FP64: tiles (one launch) where every replica's level
    // is small enough, else three axis passes (fine -> tmp[0] -> tmp[1] -> coarse),
    // which the persistent chains take on every level
    B->restr[dir].resize(3 * std::max(B->maxlev - 1, 0));
    B->restr_tile[dir].resize(std::max(B->maxlev - 1, 0));
    B->prol_tile[dir].resize(std::max(B->maxlev - 1, 0));
    for (int k = 0; k + 1 < B->maxlev; ++k) {
      bool small = !chains;
      for (const BatchRep& r : reps)
        if (k + 1 < r.plan->levels) small = small && restrict_by_tiles(grid_points(*r.plan, k + 1));
      for (int ax = 0; ax < 3 && !small; ++ax) {
        std::vector<AxisKArgs<double>> ra;
        std::vector<int> rb;
        for (const BatchRep& r : reps) {
          Plan& P = *r.plan;
          AxisKArgs<double> a{};
          int nb = 0;
          if (k + 1 < P.levels) {
            void* const* q = dir ? P.d.aq : P.d.gq;
            const double* src[3] = {(const double*)q[k], (const double*)tmp_of(r, 0), (const double*)tmp_of(r, 1)};
            double* dst[3] = {(double*)tmp_of(r, 0), (double*)tmp_of(r, 1), (double*)q[k + 1]};
            int cur[3] = {P.n[k][0], P.n[k][1], P.n[k][2]};
            for (int a2 = 0; a2 < ax; ++a2) cur[a2] = P.n[k + 1][a2];
            for (int d = 0; d < 3; ++d) a.A.nin[d] = cur[d];
            cur[ax] = P.n[k + 1][ax];
            for (int d = 0; d < 3; ++d) a.A.nout[d] = cur[d];
            a.A.axis = ax;
            a.A.lo_in = P.lo[k][ax];
            a.A.lo_out = P.lo[k + 1][ax];
            a.A.periodic = P.P.periodic;
            a.in = src[ax];
            a.out = dst[ax];
            a.acc = 0;
            nb = ew_blocks((int64_t)cur[0] * cur[1] * cur[2]);
          }
          ra.push_back(a);
          rb.push_back(nb);
        }
        chk(make_table(B->restr[dir][3 * k + ax], ra, rb));
      }
      if (chains) continue;  // restriction and prolongation run as persistent chains
      std::vector<TileKArgs<double>> ra;
      std::vector<TileKArgs<float>> pa;
      std::vector<int> rb, pb;
      for (const BatchRep& r : reps) {
        Plan& P = *r.plan;
        TileKArgs<double> a{};
        TileKArgs<float> p{};
        int na = 0, np = 0;
        if (k + 1 < P.levels) {
          void* const* q = dir ? P.d.aq : P.d.gq;
          void* const* u = dir ? P.d.au : P.d.gu;
          a = TileKArgs<double>{(const double*)q[k], (double*)q[k + 1], grid3_args(P, k, k + 1)};
          na = (int)restrict_tiles(P.n[k + 1]);
          p = TileKArgs<float>{(const float*)u[k + 1], (float*)u[k], grid3_args(P, k + 1, k)};
          np = (int)prolong_tiles(P.n[k], 8);
        }
        ra.push_back(a);
        rb.push_back(na);
        pa.push_back(p);
        pb.push_back(np);
      }
      if (small) chk(make_table(B->restr_tile[dir][k], ra, rb));
      chk(make_table(B->prol_tile[dir][k], pa, pb));
    }
    // lattice cutoff of every level below the top.  FFT form (every plan
    // periodic and built with it): five launches over all levels of all
    // replicas, level k of a replica working at offset sum_{j<k} N_j of its
    // plan's complex workspace
    bool all_fft = true;
    for (const BatchRep& r : reps) all_fft = all_fft && r.plan->lattice_fft;
    if (all_fft) {
      std::vector<FftBatchItem> items;
      for (const BatchRep& r : reps) {
        Plan& P = *r.plan;
        void* const* q = dir ? P.d.aq : P.d.gq;
        void* const* u = dir ? P.d.au : P.d.gu;
        int64_t off = 0;
        for (int k = 0; k + 1 < P.levels; ++k) {
          void* work = dir ? S1[&r - &reps[0]].fftw : P.d.fft_work;
          items.push_back(FftBatchItem{&P.fftl[k], (const double*)q[k], u[k],
                                       (char*)work + 2 * sizeof(float) * (size_t)off});
          off += grid_points(P, k);
        }
      }
      chk(fft_batch_build(items, false, &B->fft[dir]));
    }
    // otherwise the stencil, all in one launch: FP32 copies of the charges at
    // offsets of tmp[0], the outputs zeroed where several blocks add into them
    if (!all_fft) {
      std::vector<ConvKArgs> ca;
      std::vector<LatKArgs> la;
      std::vector<int> cb, lb;
      size_t sm = 0;
      for (const BatchRep& r : reps) {
        Plan& P = *r.plan;
        void* const* q = dir ? P.d.aq : P.d.gq;
        void* const* u = dir ? P.d.au : P.d.gu;
        int64_t off = 0;
        for (int k = 0; k + 1 < P.levels; ++k) {
          const int64_t np = grid_points(P, k);
          float* qf = (float*)tmp_of(r, 0) + off;
          off += np;
          ca.push_back(ConvKArgs{(const double*)q[k], qf, np});
          cb.push_back(ew_blocks(np));
          GridDims G = dims_of(P, k);
          LatKArgs a;
          if (k == 0 && P.lattice_txn > 0) {  // the plan's tuned tile on its finest level
            a.L.txn = P.lattice_txn;
            a.L.tyn = P.lattice_tyn;
          } else {
            lattice_tile(G.n[0], G.n[1], P.E, a.L.txn, a.L.tyn);
          }
          const int TW = kLatticeLP * a.L.txn, LBY = 2 * a.L.tyn;
          a.q = qf;
          a.u = (float*)u[k];
          a.G = G;
          a.seg = (const Segment2*)P.d.seg2;
          a.seg_start = P.d.seg_start;
          a.L.Ex = P.E[0];
          a.L.Ey = P.E[1];
          a.L.Ez = P.E[2];
          a.L.nbz = (int)blocks_for(G.n[2], kLatticeZ);
          a.nbx = (int)blocks_for(G.n[0], TW);
          a.nby = (int)blocks_for(G.n[1], LBY);
          a.L.nsplit = 1;  // set below, once the bricks of every replica and level are known
          a.scale = (float)std::ldexp(1.0, -k);
          a.up = nullptr;
          la.push_back(a);
          lb.push_back(a.nbx * a.nby * a.L.nbz);
          sm = std::max(sm, lattice_smem(a.L.txn, a.L.tyn, P.E));
        }
      }
      // one launch holds the bricks of every replica and level, so the input
      // planes are split over several blocks only while the whole launch
      // falls short of lattice_waves blocks per SM
      int64_t bricks = 0;
      for (int b : lb) bricks += b;
      const int64_t target = (int64_t)reps[0].plan->lattice_waves * 152 * 4 / kLatticeZ;
      const int nsplit = (int)std::max<int64_t>(1, (target + bricks - 1) / std::max<int64_t>(bricks, 1));
      // split grids write their parts to one buffer of the graph, reduced in
      // part order afterwards (reproducible sums)
      int64_t elems = 0;
      for (size_t i = 0; i < la.size(); ++i) {
        la[i].L.nsplit = std::min(nsplit, kLatticeZ + 2 * la[i].L.Ez);
        lb[i] *= la[i].L.nsplit;
        if (la[i].L.nsplit > 1) elems += (int64_t)la[i].L.nsplit * la[i].G.n[0] * la[i].G.n[1] * la[i].G.n[2];
      }
      if (elems > 0) chk(cudaMalloc((void**)&B->lparts[dir], sizeof(float) * (size_t)elems));
      std::vector<ReduceKArgs> ra;
      std::vector<int> rb;
      int64_t off = 0;
      for (size_t i = 0; i < la.size(); ++i) {
        const int64_t np = (int64_t)la[i].G.n[0] * la[i].G.n[1] * la[i].G.n[2];
        if (la[i].L.nsplit > 1 && B->lparts[dir]) {
          la[i].up = B->lparts[dir] + off;
          ra.push_back(ReduceKArgs{la[i].up, la[i].u, np, la[i].L.nsplit});
          rb.push_back(ew_blocks(np));
          off += (int64_t)la[i].L.nsplit * np;
        }
      }
      chk(make_table(B->conv[dir], ca, cb));
      chk(make_table(B->lattice[dir], la, lb, sm));
      chk(make_table(B->reduce_u[dir], ra, rb));
    }
    {  // top level of every replica
      std::vector<TopKArgs> ta;
      std::vector<int> tb;
      for (const BatchRep& r : reps) {
        Plan& P = *r.plan;
        const int top = P.levels - 1;
        void* const* q = dir ? P.d.aq : P.d.gq;
        void* const* u = dir ? P.d.au : P.d.gu;
        ta.push_back(TopKArgs{(const double*)q[top], (float*)u[top], dir ? S1[&r - &reps[0]].topu : P.d.topu,
                              dims_of(P, top), P.d.topK,
                              P.top_table_dims[0], P.top_table_dims[1]});
        tb.push_back((int)blocks_for(grid_points(P, top), kTopWarps));
      }
      chk(make_table(B->top[dir], ta, tb));
    }
    // prolongation k+1 -> k in the persistent chains: three passes (coarse ->
    // tmp[0] -> tmp[1] -> fine, the last one adding), FP32
    B->prol[dir].resize(3 * std::max(B->maxlev - 1, 0));
    for (int k = B->maxlev - 2; k >= 0 && chains; --k)
      for (int i = 0; i < 3; ++i) {
        std::vector<AxisKArgs<float>> pa;
        std::vector<int> pb;
        for (const BatchRep& r : reps) {
          Plan& P = *r.plan;
          AxisKArgs<float> a{};
          int nb = 0;
          if (k + 1 < P.levels) {
            void* const* u = dir ? P.d.au : P.d.gu;
            const float* src[3] = {(const float*)u[k + 1], (const float*)tmp_of(r, 0), (const float*)tmp_of(r, 1)};
            float* dst[3] = {(float*)tmp_of(r, 0), (float*)tmp_of(r, 1), (float*)u[k]};
            int cur[3] = {P.n[k + 1][0], P.n[k + 1][1], P.n[k + 1][2]};
            for (int j = 0; j < i; ++j) cur[2 - j] = P.n[k][2 - j];
            const int ax = 2 - i;  // z, then y, then x
            for (int d = 0; d < 3; ++d) a.A.nin[d] = cur[d];
            cur[ax] = P.n[k][ax];
            for (int d = 0; d < 3; ++d) a.A.nout[d] = cur[d];
            a.A.axis = ax;
            a.A.lo_in = P.lo[k + 1][ax];
            a.A.lo_out = P.lo[k][ax];
            a.A.periodic = P.P.periodic;
            a.in = src[i];
            a.out = dst[i];
            a.acc = (i == 2) ? 1 : 0;
            nb = ew_blocks((int64_t)cur[0] * cur[1] * cur[2]);
          }
          pa.push_back(a);
          pb.push_back(nb);
        }
        chk(make_table(B->prol[dir][3 * k + i], pa, pb));
      }
    {  // interpolation and assembly
      std::vector<InterpKArgs<float, double>> ia;
      std::vector<int> ib;
      std::vector<EnergyKArgs> ea;
      std::vector<int> eb;
      size_t sm = 0;
      for (const BatchRep& r : reps) {
        Plan& P = *r.plan;
        auto K = dir ? interp_kargs<float, double>(P, true, nullptr, nullptr, r.grad_energy, r.grad_pos, r.grad_q,
                                                   nullptr, true)
                     : interp_kargs<float, double>(P, false, r.phi, r.force, nullptr, nullptr, nullptr, P.d.partial,
                                                   true);
        const int nb = K.nbx * K.nby * (int)blocks_for(P.nc[2], K.AA.B);
        ia.push_back(K);
        ib.push_back(r.n > 0 ? nb : 0);
        sm = std::max(sm, sizeof(float) * (size_t)K.AA.pd * K.AA.pd * K.AA.pd);
        ea.push_back(EnergyKArgs{P.d.partial, r.n > 0 ? nb : 0, r.energy});
        eb.push_back(1);
      }
      chk(make_table(B->interp[dir], ia, ib, sm));
      if (dir == 0) chk(make_table(B->energy, ea, eb));
    }
  }
  (void)R;
  // persistent chains (replica 0's plan asks for them): one cooperative launch
  // per chain, as many blocks as are co-resident
  if (e == cudaSuccess && chains) {
    const bool o3 = B->order == 3;
    int dev = 0, nsm = 0, per_r = 0, per_p = 0;
    chk(cudaGetDevice(&dev));
    chk(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    chk(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_r, (const void*)(o3 ? kb_restrict_chain<3> : kb_restrict_chain<5>), kEw, 0));
    chk(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_p, (const void*)(o3 ? kb_prolong_chain<3> : kb_prolong_chain<5>), kEw, 0));
    B->chain_blocks = nsm * std::max(1, std::min(per_r, per_p));
    for (int dir = 0; dir < (backward ? 2 : 1) && e == cudaSuccess; ++dir) {
      std::vector<PassDesc> rd, pd;
      for (int k = 0; k + 1 < B->maxlev; ++k)
        for (int ax = 0; ax < 3; ++ax) {
          const auto& t = B->restr[dir][3 * k + ax];
          if (t.total > 0) rd.push_back(PassDesc{t.args, t.first, t.nrep, t.total});
        }
      for (int k = B->maxlev - 2; k >= 0; --k)
        for (int i = 0; i < 3; ++i) {
          const auto& t = B->prol[dir][3 * k + i];
          if (t.total > 0) pd.push_back(PassDesc{t.args, t.first, t.nrep, t.total});
        }
      B->n_restr = (int)rd.size();
      B->n_prol = (int)pd.size();
      chk(cudaMalloc((void**)&B->chain_restr[dir], sizeof(PassDesc) * std::max<size_t>(1, rd.size())));
      chk(cudaMalloc((void**)&B->chain_prol[dir], sizeof(PassDesc) * std::max<size_t>(1, pd.size())));
      if (e == cudaSuccess && !rd.empty())
        chk(cudaMemcpy(B->chain_restr[dir], rd.data(), sizeof(PassDesc) * rd.size(), cudaMemcpyHostToDevice));
      if (e == cudaSuccess && !pd.empty())
        chk(cudaMemcpy(B->chain_prol[dir], pd.data(), sizeof(PassDesc) * pd.size(), cudaMemcpyHostToDevice));
    }
    chk(cudaMalloc((void**)&B->bar, 2 * sizeof(unsigned)));
    if (e == cudaSuccess) chk(cudaMemset(B->bar, 0, 2 * sizeof(unsigned)));
    B->status = reps[0].plan->d.status;
    B->persistent = true;
  }
  if (e != cudaSuccess) {
    grid_batch_free(B);
    return e;
  }
  *out = B;
  return cudaSuccess;
}

// One chain as a cooperative launch.
template <typename K>
cudaError_t launch_chain(GridBatch* B, K kernel, PassDesc* passes, int npass, cudaStream_t st) {
  if (npass == 0) return cudaSuccess;
  void* args[] = {(void*)&passes, (void*)&npass, (void*)&B->bar, (void*)&B->status};
  return cudaLaunchCooperativeKernel((const void*)kernel, dim3(B->chain_blocks), dim3(kEw), args, 0, st);
}

template <typename A, typename K>
void launch_table(const BatchTable<A>& t, K kernel, int threads, cudaStream_t st) {
  if (t.total > 0) kernel<<<t.total, threads, t.smem, st>>>(t.args, t.first, t.nrep);
}

cudaError_t grid_batch_front(GridBatch* B, bool backward, cudaStream_t st) {
  if (backward && !B->has_backward) return cudaErrorInvalidValue;
  const bool o3 = B->order == 3;
  launch_table(B->zero_fx, kb_zero, kEw, st);
  launch_table(B->anterp, o3 ? kb_anterp_fx<3> : kb_anterp_fx<5>, 512, st);
  launch_table(B->fx[0], kb_fx_to_f64, kEw, st);
  if (backward) launch_table(B->fx[1], kb_fx_to_f64, kEw, st);
  return cudaGetLastError();
}

bool grid_batch_persistent(const GridBatch* B) { return B->persistent; }

cudaError_t grid_batch_levels(GridBatch* B, int d, cudaStream_t st) {
  if (d == 1 && !B->has_backward) return cudaErrorInvalidValue;
  const bool o3 = B->order == 3;
  if (B->persistent) {
    cudaError_t e = launch_chain(B, o3 ? kb_restrict_chain<3> : kb_restrict_chain<5>, B->chain_restr[d], B->n_restr, st);
    if (e != cudaSuccess) return e;
  } else {
    for (int k = 0; k + 1 < B->maxlev; ++k) {
      if (B->restr_tile[d][k].total > 0) {
        launch_table(B->restr_tile[d][k], o3 ? kb_restrict_tile<3> : kb_restrict_tile<5>, 256, st);
        continue;
      }
      for (int ax = 0; ax < 3; ++ax)
        launch_table(B->restr[d][3 * k + ax], o3 ? kb_restrict_axis<3> : kb_restrict_axis<5>, kEw, st);
    }
  }
  if (B->fft[d]) {
    cudaError_t e = fft_batch_launch(B->fft[d], st);
    if (e != cudaSuccess) return e;
  } else {
    launch_table(B->conv[d], kb_f64_to_f32, kEw, st);
    launch_table(B->lattice[d], kb_lattice_f2, 32 * kLatticeZ, st);
    launch_table(B->reduce_u[d], kb_lattice_reduce, kEw, st);
  }
  launch_table(B->top[d], kb_top, 32 * kTopWarps, st);
  if (B->persistent) {
    cudaError_t e = launch_chain(B, o3 ? kb_prolong_chain<3> : kb_prolong_chain<5>, B->chain_prol[d], B->n_prol, st);
    if (e != cudaSuccess) return e;
  } else {
    for (int k = B->maxlev - 2; k >= 0; --k)
      launch_table(B->prol_tile[d][k], o3 ? kb_prolong_tile<3> : kb_prolong_tile<5>, 256, st);
  }
  return cudaGetLastError();
}

cudaError_t grid_batch_interp(GridBatch* B, bool backward, cudaStream_t st) {
  const bool o3 = B->order == 3;
  if (backward) {
    if (!B->has_backward) return cudaErrorInvalidValue;
    launch_table(B->interp[1], o3 ? kb_interp_bwd<3> : kb_interp_bwd<5>, 256, st);
  } else {
    launch_table(B->interp[0], o3 ? kb_interp_fwd<3> : kb_interp_fwd<5>, 256, st);
    launch_table(B->energy, kb_energy_final, 1024, st);
  }
  return cudaGetLastError();
}

// Opts the patch kernels into more than 48 KB of dynamic shared memory.  Done
// once per process when the first plan is built, so that no configuration call
// happens while a stream is being captured into a graph.
cudaError_t configure_kernels() {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* f) {
    cudaError_t r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLatticeSmemMax);
    if (r != cudaSuccess) e = r;
  };
  set((const void*)k_interp_gather<3>);
  set((const void*)k_interp_gather<5>);
  set((const void*)k_lattice_f2<kLatticeLP, 4, 8>);
  set((const void*)k_lattice_f2<kLatticeLP, 0, 0>);
  set((const void*)kb_lattice_f2);
  set((const void*)kb_anterp_fx<3>);
  set((const void*)kb_anterp_fx<5>);
  set((const void*)kb_interp_fwd<3>);
  set((const void*)kb_interp_fwd<5>);
  set((const void*)kb_interp_bwd<3>);
  set((const void*)kb_interp_bwd<5>);
  set((const void*)k_anterp_fx<3>);
  set((const void*)k_anterp_fx<5>);
  set((const void*)k_interp_bwd<3, double>);
  set((const void*)k_interp_bwd<3, float>);
  set((const void*)k_interp_bwd<5, double>);
  set((const void*)k_interp_bwd<5, float>);
  if (e == cudaSuccess) e = configure_fft_kernels();
  if (e == cudaSuccess) e = configure_pair64_kernels();
  return e;
}

}  // namespace msm
