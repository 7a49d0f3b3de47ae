// kernels_pair64.cu -- the short-range pair sums of FP64 plans (the same sums
// as kernels_pair.cu, every pair function in FP64).
//
// This GPU issues FP64 at 1/64 of the FP32 rate (2 lanes per SM and clock), so
// the kernel is bound by the number of FP64 instructions and nothing else:
// 22 per MSM pair seen from one atom, 27 for both atoms at once, and only pairs
// inside the cutoff are worth them.  The candidates of a target's neighbourhood
// are ~2,000 sources (culled against the bounding box of a warp's targets),
// ~750 of them inside a 12 A cutoff at water density.  So the kernel separates
// finding from evaluating:
//   - sources are staged 32 at a time in a ring of shared memory (FP64
//     coordinates in the targets' frame, and their FP32 truncation), and every
//     lane tests every staged source against its own target in FP32, with a
//     margin for the truncation; a hit goes onto the lane's own list (one byte,
//     the ring slot).  This costs ~10 FP32-rate instructions per source, under
//     5 % of the FP64 time.
//   - the lanes then pop their lists in step and evaluate one pair each, all
//     lanes on real pairs.  The cutoff and r > 0 are decided again in FP64 (on
//     the bit patterns, which order like the values and cost no FP64
//     instruction).  Lists of different lanes fill unevenly as the walk passes
//     through the neighbourhood; the ring keeps up to 256 sources alive so that
//     a lane ahead of the others still has entries.
// An MSM pair is evaluated once: of two groups of targets the one that
// takes_pair() names meets the other's atoms, and adds to their reaction sums
// with FP64 reductions (fire and forget; at most 4 per 27 FP64 instructions, and
// gathering them to whole sectors first made no difference).  An atom has two
// reaction sums, for near and far pairs (kNear2), beside its own total: the many
// small terms of the far pairs would else round onto the few large ones (force
// error of 3,000 atoms 4.3e-16 with every pair from both atoms, 6.8e-16 with one
// sum that also took the atom's own total, 4.4e-16 with the three, at the same
// speed).  Against each atom for itself: 1,066,628 atoms (a = 12) 36.4 -> 24.0 ms
// (the FP64 pipe alone would take 18.4), 100,000 (a = 10) 2.63 -> 1.63 ms, 23,558
// 735 -> 533 us, 3,000 open 154 -> 114 us.  The choice by group index halves the
// sources staged and tested too.  At a million atoms where it takes 20.9 ms, "the
// earlier atom" takes 25.6 (an atom at the top of its cell has far fewer later
// neighbours than one at the bottom, and the lanes wait for the fullest list), and
// a choice by atom parity 21.5 (the ring fills with sources few lanes take; 3,000
// atoms 140 against 110 us).
// The reciprocal square root is seeded by the FP32 one and refined once by
// Halley's third-order iteration (5 FP64 instructions, error below 1 ulp).
//
// A group of T = 8 or 16 consecutive sorted atoms is a warp's targets,
// 32 / T lanes sharing one (each tests every (32 / T)-th source); small systems
// also split a group's sources over 2 to 8 warps of a block, combined in a
// fixed order.  Groups are cut into pieces of one cell row as the target runs
// of kernels_pair.cu are.
#include <algorithm>
#include <cstring>

#include "pair_common.h"

namespace msm {

namespace {

constexpr int kRing = 256;   // staged sources (a list entry is one byte)
constexpr int kChunk = 32;   // sources staged together
constexpr int kMaxSplit = 8; // warps sharing a group
constexpr int kShift0 = 3;   // index of offset 0 in the shift tables
// Near pairs: r^2 <= kNear2 a^2.  In a CPU model of the sums' order (water, a
// gas and like charges, 420 to 750 pairs an atom) the rounding error of force
// and potential is 0.4 to 1.0 of that of every pair from both atoms for 0.14 to
// 0.22, up to 1.6 below 0.05 and 1.2 at 0.36; one reaction sum has 1.5 to 2.0.
constexpr double kNear2 = 0.1875;

struct Pair64Args {
  PairKArgs g;  // geometry: cell widths and cutoff in FP32, scaled by 2^esc (a in [1, 2))
  const R4<double>* atoms;
  R4<double>* fs;     // force sums, potential of the pairs an atom's own group evaluates
  R4<double>* react;  // [2 i], [2 i + 1]: the same from the other pairs, near and far (both_sides)
  double a2;
  double G[4], D[3];  // pot = 1/r + sum_k G[k] r2^k, f' = 1/r^3 + sum_k D[k] r2^k
  WolfC<double> W;
  double shx[8], shy[8], shz[8];  // offset (index - kShift0) times the cell width
  int near_hi;                    // high word of the near pairs' largest r^2
  float a2test;                   // scaled cutoff^2 with the margin of the FP32 test
  int esc;                        // exponent added to coordinates before the FP32 test
  int lt;                         // log2 of the targets per group
  int nsplit;                     // warps sharing a group (1: a block's warps take groups of their own)
};

struct alignas(16) Warp64 {
  double src[kRing][4];  // x, y, z, q in the piece's frame
  float4 f[kRing];       // their FP32 truncations and the source's index
  unsigned char list[kRing][32];
  SegList segs;
};

// x 2^esc truncated to FP32 (integer operations only: conversions from FP64
// run at the FP64 rate).
__device__ __forceinline__ float trunc_scaled(double x, int esc) {
  const int hi = __double2hiint(x);
  const int e = ((hi >> 20) & 0x7ff) - 896 + esc;
  if (e <= 0) return 0.f;
  return __int_as_float((hi & 0x80000000) | (e << 23) | ((hi & 0xfffff) << 3) |
                        (int)((unsigned)__double2loint(x) >> 29));
}

// 1 / sqrt(x), x > 0 and normal: the FP32 approximation of the mantissa, its
// exponent halved with integers, then y (1 + r/2 + 3 r^2/8), r = 1 - x y^2
// (Halley's iteration; the next term, 5 r^3/16 with |r| < 2^-21, is below
// 2^-64).  The rounding of x y and the last one are half an ulp each at most.
__device__ __forceinline__ double rsqrt_halley(double x) {
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) - 1023, odd = e & 1;
  const float m = __int_as_float(((127 + odd) << 23) | ((hi & 0xfffff) << 3) |
                                 (int)((unsigned)__double2loint(x) >> 29));
  float s;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(m));
  const int sb = __float_as_int(s);
  const double y = __hiloint2double((sb >> 3) + ((896 - ((e - odd) >> 1)) << 20), sb << 29);
  const double r = fma(-(x * y), y, 1.0);
  return fma(y * r, fma(0.375, r, 0.5), y);
}

// MSM pairs are evaluated once, for both atoms, with reductions into the sums
// (their order varies, as that of the FP64 anterpolation's does); the cutoff
// and Wolf methods evaluate each pair for either atom and store, so that their
// results repeat bit for bit.
__host__ __device__ constexpr bool both_sides(int kind) { return kind == kPairMSM; }

// Adds (x, y, z, w) to one atom's sums.
__device__ __forceinline__ void add_sums(R4<double>* s, double x, double y, double z, double w) {
  atomicAdd(&s->x, x);
  atomicAdd(&s->y, y);
  atomicAdd(&s->z, z);
  atomicAdd(&s->w, w);
}

// Which of two groups (atoms of a group) i != j evaluates their pairs: the later
// one if the numbers have the same parity, else the earlier one.
__device__ __forceinline__ bool takes_pair(int i, int j) { return ((((j - i) >> 31) ^ i ^ j) & 1) != 0; }

// One pair: q_j times the pair potential onto phi, f' (r_i - r_j) onto
// (px, py, pz), with the force on i being q_i times that sum.  BOTH: q_i q_j f'
// (r_i - r_j) onto (px, py, pz), and the same for atom j onto its reaction sums
// sj (5 more FP64 instructions against the 22 of a second visit).
template <int M, int K>
__device__ __forceinline__ void pair64(const Pair64Args& A, double tx, double ty, double tz, double tq,
                                       const double* src, double& phi, double& px, double& py, double& pz,
                                       R4<double>* sj) {
  constexpr bool BOTH = both_sides(K);
  const double2 xy = *reinterpret_cast<const double2*>(src), zq = *reinterpret_cast<const double2*>(src + 2);
  const double dx = tx - xy.x, dy = ty - xy.y, dz = tz - zq.x;
  const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
  const long long rb = __double_as_longlong(r2);
  const bool ok = rb < __double_as_longlong(A.a2) && rb > 0;  // inside the cutoff, not the atom itself
  const double r2s = ok ? r2 : A.a2, q = ok ? zq.y : 0.0;
  const double ri = rsqrt_halley(r2s);
  double f;
  if (K == kPairMSM) {
    double g = A.G[M];
#pragma unroll
    for (int k = M - 1; k >= 0; --k) g = fma(g, r2s, A.G[k]);
    double d = A.D[M - 1];
#pragma unroll
    for (int k = M - 2; k >= 0; --k) d = fma(d, r2s, A.D[k]);
    const double v = ri + g;
    phi = fma(q, v, phi);
    f = q * fma(ri * ri, ri, d);
    if constexpr (BOTH) {
      const double w = -tq * f;
      const double wx = w * dx, wy = w * dy, wz = w * dz;
      px -= wx;
      py -= wy;
      pz -= wz;
      if (ok && sj) add_sums(sj + (__double2hiint(r2) > A.near_hi), wx, wy, wz, tq * v);
      return;
    }
  } else if (K == kPairWolf) {
    const double r = r2s * ri;
    const double e = d_erfc(A.W.alpha * r) * ri, x = A.W.c2 * d_exp(-A.W.alpha2 * r2s);
    phi = fma(q, e - A.W.vR + A.W.c1 * (r - A.W.R), phi);
    f = q * ((e + x) * ri * ri - A.W.c1 * ri);
  } else {
    phi = fma(q, ri, phi);
    f = q * (ri * ri * ri);
  }
  px = fma(f, dx, px);
  py = fma(f, dy, py);
  pz = fma(f, dz, pz);
}

template <int M, int K>
__global__ void __launch_bounds__(32 * kMaxSplit) k_pair64(const __grid_constant__ Pair64Args A) {
  constexpr bool BOTH = both_sides(K);
  pdl_sync();
  extern __shared__ __align__(16) unsigned char smem64[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  Warp64& S = reinterpret_cast<Warp64*>(smem64)[warp];
  const PairKArgs& g = A.g;
  const int T = 1 << A.lt, t = lane & (T - 1), h = lane >> A.lt, lpt = 32 >> A.lt;
  const bool split = A.nsplit > 1;
  const int group = split ? blockIdx.x : blockIdx.x * (blockDim.x >> 5) + warp, part = split ? warp : 0;
  const int s0 = group << A.lt;
  if (s0 >= g.natoms) return;  // warp-uniform; block-uniform where the block shares the group
  const int nval = min(T, g.natoms - s0);
  const int ncx = g.A.nc[0], ncy = g.A.nc[1];
  const float FAR = 1e6f;
  const bool sv = t < nval;
  const int mycell = sv ? g.scell[s0 + t] : INT_MAX;
  const R4<double> me = sv ? A.atoms[s0 + t] : R4<double>{0.0, 0.0, 0.0, 0.0};
  for (int l0 = 0; l0 < nval;) {  // one piece per step (the same for every warp of the group)
    const int c0 = __shfl_sync(kFull, mycell, l0);
    const int cx = c0 % ncx, cy = (c0 / ncx) % ncy, cz = c0 / (ncx * ncy);
    const int climit = c0 + min(g.maxspan, ncx - 1 - cx);
    const bool inp = t >= l0 && mycell <= climit;
    const unsigned pb = __ballot_sync(kFull, inp) & (kFull >> (32 - T));
    const int l1 = 32 - __clz(pb);
    const int span = __shfl_sync(kFull, mycell, l1 - 1) - c0;
    // the home block: the atoms of the piece's cells
    const int h0 = g.cell_start[c0], h1 = g.cell_start[c0 + span + 1];
    const double tx = me.x + A.shx[(inp ? mycell - c0 : 0) + kShift0], ty = me.y, tz = me.z;
    const float ux = trunc_scaled(tx, A.esc), uy = trunc_scaled(ty, A.esc), uz = trunc_scaled(tz, A.esc);
    const float lx = warp_min(inp ? ux : FAR), ly = warp_min(inp ? uy : FAR), lz = warp_min(inp ? uz : FAR);
    const float hx = warp_max(inp ? ux : -FAR), hy = warp_max(inp ? uy : -FAR), hz = warp_max(inp ? uz : -FAR);
    // the ranges of sources: the home block, then the neighbour rows
    const int nseg = build_segments(S.segs, g, cx, cy, cz, span, lx, ly, lz, hx, hy, hz, lane);
    int seg = -1, jb = h0 + kChunk * part, je = h1, xb = -cx, oyz = kShift0 | (kShift0 << 4);
    auto settle = [&]() -> bool {  // at the next 32 sources of this warp, in a later range if this one has ended
      while (jb >= je) {
        const int skip = (jb - je) / kChunk;  // chunks of the following ranges that are the other warps'
        if (++seg >= nseg) return false;
        const int4 r = S.segs.rec[seg];
        jb = r.x + kChunk * skip;
        je = r.y;
        xb = r.z;
        oyz = r.w;
      }
      return true;
    };
    bool more = settle();
    double phi = 0.0, px = 0.0, py = 0.0, pz = 0.0;
    unsigned staged = 0, oldest = 0;  // sources staged so far; the oldest one a list still names
    unsigned head = 0, tail = 0;      // the lane's list: entries popped, entries pushed
    for (;;) {
      // find: stage chunks while the ring has room, test the new sources
      while (more && staged - oldest <= kRing - kChunk) {
        const int j = jb + lane;
        R4<double> a = {0.0, 0.0, 0.0, 0.0};
        bool keep = j < je && (!BOTH || (j >> A.lt) == group || takes_pair(group, j >> A.lt));
        if (keep) {
          a = A.atoms[j];
          a.x += A.shx[(int)g.cellx[j] + xb + kShift0];
          a.y += A.shy[oyz & 15];
          a.z += A.shz[oyz >> 4];
        }
        jb += kChunk * A.nsplit;
        more = settle();
        const float ax = trunc_scaled(a.x, A.esc), ay = trunc_scaled(a.y, A.esc), az = trunc_scaled(a.z, A.esc);
        const float ex = fmaxf(fmaxf(lx - ax, ax - hx), 0.f);
        const float ey = fmaxf(fmaxf(ly - ay, ay - hy), 0.f);
        const float ez = fmaxf(fmaxf(lz - az, az - hz), 0.f);
        keep = keep && ex * ex + ey * ey + ez * ez < A.a2test;
        const unsigned bal = __ballot_sync(kFull, keep);
        if (keep) {
          const int p = (staged + __popc(bal & ((1u << lane) - 1u))) & (kRing - 1);
          S.f[p] = make_float4(ax, ay, az, __int_as_float(j));
          *reinterpret_cast<double2*>(&S.src[p][0]) = make_double2(a.x, a.y);
          *reinterpret_cast<double2*>(&S.src[p][2]) = make_double2(a.z, a.w);
        }
        __syncwarp();
        const unsigned end = staged + __popc(bal);
#pragma unroll 4
        for (unsigned s = staged + ((h - staged) & (lpt - 1)); s < end; s += lpt) {
          const int p = s & (kRing - 1);
          const float4 b = S.f[p];
          const float dx = ux - b.x, dy = uy - b.y, dz = uz - b.z;
          const int j = __float_as_int(b.w);
          const bool mine = !BOTH || (j >> A.lt) != group || j == s0 + t || takes_pair(s0 + t, j);
          if (inp && mine && dx * dx + dy * dy + dz * dz < A.a2test) S.list[tail++ & (kRing - 1)][lane] = (unsigned char)p;
        }
        staged = end;
      }
      // evaluate: every lane pops its own list; while more sources follow, as
      // many steps as all lanes have entries for (at least 8, so that the
      // ring's oldest source is let go)
      const unsigned have = tail - head;
      const unsigned steps = more ? max(8u, __reduce_min_sync(kFull, inp ? have : 0xffffffffu))
                                  : __reduce_max_sync(kFull, have);
      double sphi = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
      for (unsigned k = 0; k < steps; ++k)
        if (head < tail) {
          const int p = S.list[head++ & (kRing - 1)][lane];
          const int j = BOTH ? __float_as_int(S.f[p].w) : 0;
          // (an image of the atom itself is one-sided: the mirror image is met too)
          pair64<M, K>(A, tx, ty, tz, me.w, S.src[p], sphi, sx, sy, sz, j != s0 + t ? A.react + 2 * (int64_t)j : nullptr);
        }
      phi += sphi;
      px += sx;
      py += sy;
      pz += sz;
      if (!more) break;
      // the ring index of the lane's next entry lies 1 .. kRing sources back
      const unsigned back = head < tail ? ((staged - 1u - S.list[head & (kRing - 1)][lane]) & (kRing - 1)) + 1u : 0u;
      oldest = staged - __reduce_max_sync(kFull, back);
      __syncwarp();
    }
    // the lanes of a target, then the parts of a group, in a fixed order
    for (int o = T; o < 32; o <<= 1) {
      phi += __shfl_xor_sync(kFull, phi, o);
      px += __shfl_xor_sync(kFull, px, o);
      py += __shfl_xor_sync(kFull, py, o);
      pz += __shfl_xor_sync(kFull, pz, o);
    }
    if (split) {
      __syncwarp();
      if (lane < T) {
        S.src[lane][0] = phi;
        S.src[lane][1] = px;
        S.src[lane][2] = py;
        S.src[lane][3] = pz;
      }
      __syncthreads();
      if (part == 0 && lane < T)
        for (int p = 1; p < A.nsplit; ++p) {
          const double* o = reinterpret_cast<Warp64*>(smem64)[p].src[lane];
          phi += o[0];
          px += o[1];
          py += o[2];
          pz += o[3];
        }
      __syncthreads();
    }
    if (part == 0 && h == 0 && inp) {
      const int i = s0 + t;
      A.fs[i] = BOTH ? R4<double>{px, py, pz, phi} : R4<double>{me.w * px, me.w * py, me.w * pz, phi};
    }
    __syncwarp();
    l0 = l1;
  }
}

// Targets per group and warps per group: groups of 16 once they make 152 SMs x
// 8 warps, else groups of 8, then several warps per group.  Pair sums alone with
// groups of 8, 16 and 32: 12,000 atoms 320, 439 and 716 us, 23,558 502, 533 and 798
// (groups of 8 stage each source for fewer targets, and beside the grid passes an
// evaluation with gradients takes 663 against 653 us), 50,000 942, 1,004 and 1,233,
// 100,000 1.65, 1.63 and 1.87 ms, 200,000 3.12, 2.92 and 3.12, 1,066,628 25.5, 24.0
// and 24.1 (groups of 32 leave the chip waiting for its last warps).  Warps per
// group of 8, 1, 2, 4 and 8: 3,000 atoms 231, 135, 113 and 117 us; 6,000 262, 191,
// 206 and 214.
void group_shape(int64_t n, int& lt, int& nsplit) {
  constexpr int64_t kFill = 152 * 8;
  lt = (n + 15) >> 4 >= kFill ? 4 : 3;
  nsplit = 1;
  while (nsplit < kMaxSplit && ((n + (1 << lt) - 1) >> lt) * nsplit < kFill * 3 / 4) nsplit *= 2;
}

Pair64Args pair64_args(const Plan& P, int64_t n, double alpha) {
  Pair64Args A;
  const double a = P.P.cutoff;
  A.g = pair_kargs(P);
  A.g.natoms = (int)n;
  A.esc = -std::ilogb(a);
  const double sc = std::ldexp(1.0, A.esc);
  A.g.cwx = (float)(P.cw[0] * sc);
  A.g.cwy = (float)(P.cw[1] * sc);
  A.g.cwz = (float)(P.cw[2] * sc);
  // a coordinate lies within X = 8 cell widths of the origin and its
  // truncation is off by at most 2^-23 X, a difference by three times that
  // (with its own rounding): r^2 near a^2 by 2 sqrt(3) a 3 2^-23 X (1 + small)
  double X = 0.0;
  for (int d = 0; d < 3; ++d) X = std::max(X, 8.0 * P.cw[d] * sc);
  const double as = a * sc;
  const double a2t = as * as + 16.0 * as * X * std::ldexp(1.0, -23) + 16.0 * X * X * std::ldexp(1.0, -46);
  A.a2test = (float)(a2t * (1.0 + 1e-6));
  A.g.A.a2f = A.a2test;
  A.atoms = (const R4<double>*)P.d.atoms;
  A.fs = (R4<double>*)P.d.fs;
  A.react = (R4<double>*)P.d.react;
  A.a2 = a * a;
  const double near2 = kNear2 * A.a2;
  uint64_t near_bits;
  std::memcpy(&near_bits, &near2, sizeof near_bits);
  A.near_hi = (int)(near_bits >> 32);
  static const double cf[4][4] = {{0, 0, 0, 0}, {1.5, -0.5, 0, 0}, {1.875, -1.25, 0.375, 0},
                                  {2.1875, -2.1875, 1.3125, -0.3125}};
  const int m = P.P.splitting;
  for (int k = 0; k < 4; ++k) A.G[k] = k <= m ? -cf[m][k] / std::pow(a, 2 * k + 1) : 0.0;
  for (int k = 0; k < 3; ++k) A.D[k] = k + 1 <= m ? 2.0 * (k + 1) * cf[m][k + 1] / std::pow(a, 2 * k + 3) : 0.0;
  A.W = wolf_consts<double>(alpha, a);
  for (int o = 0; o < 8; ++o) {
    A.shx[o] = (o - kShift0) * P.cw[0];
    A.shy[o] = (o - kShift0) * P.cw[1];
    A.shz[o] = (o - kShift0) * P.cw[2];
  }
  group_shape(n, A.lt, A.nsplit);
  return A;
}

template <int M, int K>
cudaError_t launch_k(const Plan& P, const Pair64Args& A, cudaStream_t st) {
  const int64_t groups = ((int64_t)A.g.natoms + (1 << A.lt) - 1) >> A.lt;
  const int warps = A.nsplit > 1 ? A.nsplit : 2;
  const unsigned blocks = (unsigned)(A.nsplit > 1 ? groups : (groups + warps - 1) / warps);
  return klaunch(P.pdl, k_pair64<M, K>, blocks, 32 * warps, warps * sizeof(Warp64), st, A);
}

template <int M, int K>
cudaError_t set_smem() {
  return cudaFuncSetAttribute((const void*)k_pair64<M, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(kMaxSplit * sizeof(Warp64)));
}

}  // namespace

cudaError_t configure_pair64_kernels() {
  cudaError_t e = set_smem<1, kPairMSM>();
  if (e == cudaSuccess) e = set_smem<2, kPairMSM>();
  if (e == cudaSuccess) e = set_smem<3, kPairMSM>();
  if (e == cudaSuccess) e = set_smem<2, kPairCutoff>();
  if (e == cudaSuccess) e = set_smem<2, kPairWolf>();
  return e;
}

cudaError_t launch_pair64(Plan& P, int kind, int64_t n, double alpha, cudaStream_t st) {
  const Pair64Args A = pair64_args(P, n, alpha);
  if (kind == kPairCutoff) return launch_k<2, kPairCutoff>(P, A, st);  // M unused
  if (kind == kPairWolf) return launch_k<2, kPairWolf>(P, A, st);
  if (P.P.splitting == 1) return launch_k<1, kPairMSM>(P, A, st);
  if (P.P.splitting == 2) return launch_k<2, kPairMSM>(P, A, st);
  return launch_k<3, kPairMSM>(P, A, st);
}

}  // namespace msm
