// Escape physics of the cluster (Sec. 2.2; Sec. 3.1 footnote on r_t):
//
// * boundedness: particle i is bound when kin |v_i|^2 - sum_{j != i} G m_j / r_ij < 0
//   in the cluster frame, the sum an unsoftened direct summation over every
//   particle of its progenitor;
// * the energy-based Lagrange radius r_x: the k-th smallest cluster-frame radius
//   among the bound particles, k = ceil(frac n_bound); the coefficient set of
//   Eq. 3b is r <= r_x;
// * tidal scales at the centre R: T_ij = -d^2 psi_host/dx_i dx_j, its eigenvalues,
//   the tidal radius r_t = (G M_c / (l1 - (l2 + l3)/2))^(1/3) and the
//   integration timestep dt_int = sqrt(eta) (|T|_F^2 / 6)^(-1/4).
//
// Kernels:
//   k_bound_pairs  O(N^2) pair sums, every unordered pair once: chunk A of a
//                  progenitor's particles against chunk B = A + r (round r),
//                  one 1/r for both particles.  The i-particles (A) sit in
//                  registers; the j-particles (B) are dealt one pair a lane and
//                  their sums travel around the warp with them.  Double precision
//                  evaluates the pair terms in float-float arithmetic
//                  (k_bound_pairs_ff).
//   k_bound_ordered, _ff  every ordered pair, for small samples.
//   k_bound_finish one thread per particle: adds the slots in order, forms
//                  E_i and the bound flag, and the radius key (bits of r^2).
//   k_select       one block, or a cluster of eight, per progenitor: bound count
//                  and mass, radix selection of the k-th smallest key (8 passes
//                  of 8 bits over shared-memory histograms of integer counts),
//                  the mask.
//   k_tidal        one thread per progenitor.
// Every sum has a fixed order, so results are bitwise reproducible.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cooperative_groups.h>
#include <math_constants.h>

#include "scf_device.cuh"

#include "scf_escape.h"

namespace {

namespace cg = cooperative_groups;

constexpr int kPairThreads = 128;
constexpr int kPairWarps = kPairThreads / 32;

template <typename V4>
struct Elem;
template <>
struct Elem<float4> {
  static constexpr int I = 4;     // i-particles per thread
};
template <>
struct Elem<ScfD4> {
  static constexpr int I = 2;
};
template <typename V4>
constexpr int kPairChunk = kPairThreads * Elem<V4>::I;  // particles of a chunk

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 neg(float2 x) { return make_float2(-x.x, -x.y); }
__device__ __forceinline__ float2 rotate(float2 x, int lane) {  // from the next lane
  return make_float2(__shfl_sync(0xffffffffu, x.x, (lane + 1) & 31), __shfl_sync(0xffffffffu, x.y, (lane + 1) & 31));
}
__device__ __forceinline__ bool finite2(float2 x) { return isfinite(x.x) && isfinite(x.y); }

// 1/sqrt(r2) of single-precision pairs by the hardware approximation
// (rsqrt.approx.ftz.f32, a few ulp).  A pair that adds nothing (r2 zero, below
// the smallest normal float, which the approximation flushes to zero, or NaN)
// gives an infinity or NaN: SAFE replaces it by 0, the fast form leaves it to
// show in the sums, which are then formed again by SAFE.  r2 = inf gives 0.
template <bool SAFE>
__device__ __forceinline__ float2 pair_inv_r(float2 r2) {
  float2 y = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
  if (SAFE) {
    y.x = r2.x >= 1.17549435e-38f ? y.x : 0.f;
    y.y = r2.y >= 1.17549435e-38f ? y.y : 0.f;
  }
  return y;
}

// Single precision.  A lane's i-particles, each coordinate in both halves of a
// packed operand (negated: separations are sums).
struct PairI {
  float2 x[4], y[4], z[4], m[4];
};

// One rotation: the warp's 128 i-particles against 64 j-particles, two a lane at a
// time (xy, zm: (x, x', y, y') and (z, z', m, m') of 32 pairs).  part[q] += m_j / r
// over the lane's 32 steps, sj = the j sums sum m_i / r, back at their home lane.
// Bound by the FP32 pipe: 12 additions, 12 products and 9 accumulations, packed,
// for eight unordered pairs (the special-function unit a third busy).
template <bool SAFE>
__device__ __forceinline__ void rotation(const PairI& pi, const float4* xy, const float4* zm, int lane, float2* part,
                                         float2& sj) {
  sj = dup(0.f);
#pragma unroll 4
  for (int s = 0; s < 32; ++s) {
    const int k = (lane + s) & 31;
    const float4 a = xy[k], b = zm[k];
    const float2 xj = make_float2(a.x, a.y), yj = make_float2(a.z, a.w), zj = make_float2(b.x, b.y),
                 mj = make_float2(b.z, b.w);
    float2 t = dup(0.f);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float2 dx = __fadd2_rn(xj, pi.x[q]), dy = __fadd2_rn(yj, pi.y[q]), dz = __fadd2_rn(zj, pi.z[q]);
      const float2 ri = pair_inv_r<SAFE>(__ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx))));
      part[q] = __ffma2_rn(mj, ri, part[q]);
      t = q == 0 ? __fmul2_rn(pi.m[q], ri) : __ffma2_rn(pi.m[q], ri, t);
    }
    sj = rotate(__fadd2_rn(sj, t), lane);
  }
}

// Pair sums over the rounds [r0, r0 + gridDim.z R): block (A, progenitor, g) takes
// the R rounds from r0 + g R.  Round r pairs chunk A with chunk B = A + r (mod P),
// r = 1 .. P/2 (r = P/2 of an even P for A < P/2 only); round 0 is the chunk with
// itself, every ordered pair, done by block g = 0 of the first launch.  A slot of
// part has one writer per element and launch: slot g the i sums of group g, slot
// gridDim.z + g R + k the j sums of its k-th round; launches follow one another,
// so every sum has a fixed order.
__global__ void __launch_bounds__(kPairThreads) k_bound_pairs(BoundArgs a) {
  constexpr int C = kPairChunk<float4>, I = 4;
  __shared__ float4 s_xy[C / 2], s_zm[C / 2];
  __shared__ float s_sum[kPairWarps][C];
  const float4* pos = reinterpret_cast<const float4*>(a.pos);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, A = blockIdx.x;
  for (int p = blockIdx.y; p < a.n_prog; p += gridDim.y) {
    const int64_t o0 = a.prog_off[p], n = a.prog_off[p + 1] - o0;
    const int P = (int)((n + C - 1) / C);
    if (A >= P) continue;  // the same for every thread of the block
    PairI pi;
    double acc[I];
#pragma unroll
    for (int q = 0; q < I; ++q) {
      const int64_t i = (int64_t)A * C + warp * (32 * I) + q * 32 + lane;
      // a particle past the end: far from everything, no mass
      const float4 x = i < n ? pos[o0 + i] : make_float4(1e18f, 0.f, 0.f, 0.f);
      pi.x[q] = dup(-x.x);
      pi.y[q] = dup(-x.y);
      pi.z[q] = dup(-x.z);
      pi.m[q] = dup(x.w);
      acc[q] = 0.0;
    }
    const int rb = a.round0 + blockIdx.z * a.rounds;
    for (int rr = rb == 1 && a.round0 == 1 ? -1 : 0; rr < a.rounds; ++rr) {
      const bool self = rr < 0;  // the first launch's block g = 0 starts with round 0
      const int r = self ? 0 : rb + rr;
      if (r > P / 2 || (2 * r == P && A >= r)) break;
      const int B = A + r < P ? A + r : A + r - P;
      __syncthreads();
      for (int k = tid; k < C / 2; k += kPairThreads) {
        const int64_t j = (int64_t)B * C + 2 * k;
        const float4 far = make_float4(-1e18f, 0.f, 0.f, 0.f);
        const float4 u = j < n ? pos[o0 + j] : far, v = j + 1 < n ? pos[o0 + j + 1] : far;
        s_xy[k] = make_float4(u.x, v.x, u.y, v.y);
        s_zm[k] = make_float4(u.z, v.z, u.w, v.w);
      }
      __syncthreads();
      float2 part[I];
      for (int c = 0; c < C / 64; ++c) {
        // blocks of 64 terms (two rotations of 32, two lanes) before the double add
        float2 was[I], sj;
#pragma unroll
        for (int q = 0; q < I; ++q) {
          if (c % 2 == 0) part[q] = dup(0.f);
          was[q] = part[q];
        }
        bool ok = !self;
        if (!self) {
          rotation<false>(pi, s_xy + 32 * c, s_zm + 32 * c, lane, part, sj);
          ok = finite2(sj) && finite2(part[0]) && finite2(part[1]) && finite2(part[2]) && finite2(part[3]);
        }
        if (__any_sync(0xffffffffu, !ok)) {
#pragma unroll
          for (int q = 0; q < I; ++q) part[q] = was[q];
          rotation<true>(pi, s_xy + 32 * c, s_zm + 32 * c, lane, part, sj);
        }
        if (c % 2 == 1)
#pragma unroll
          for (int q = 0; q < I; ++q) acc[q] += (double)part[q].x + (double)part[q].y;
        *reinterpret_cast<float2*>(&s_sum[warp][64 * c + 2 * lane]) = sj;
      }
      __syncthreads();
      if (!self) {
        double* out = a.part + (size_t)(gridDim.z + blockIdx.z * a.rounds + rr) * (size_t)a.n_total + o0 + (int64_t)B * C;
        for (int k = tid; k < C && (int64_t)B * C + k < n; k += kPairThreads) {
          double v = 0.0;
#pragma unroll
          for (int w = 0; w < kPairWarps; ++w) v += (double)s_sum[w][k];
          out[k] += v;
        }
      }
    }
#pragma unroll
    for (int q = 0; q < I; ++q) {
      const int64_t i = (int64_t)A * C + warp * (32 * I) + q * 32 + lane;
      if (i < n) a.part[(size_t)blockIdx.z * (size_t)a.n_total + (size_t)(o0 + i)] += acc[q];
    }
    __syncthreads();
  }
}

// Double-precision pair sums in float-float arithmetic ("double-single"):
// GB300 retires 64 single-precision FMAs for each double one, and a pair term
// carried as unevaluated sums of two floats (Dekker 1971; Knuth's TwoSum and
// the FMA-based exact product) costs tens of single-precision operations
// against 11 double ones, so it runs several times faster at a relative error
// near 1e-13.  Positions and masses are split once into hi + lo floats when
// they are staged (48 of a double's 53 bits: a pair term's relative error
// grows like 2^-48 |x| / r_ij for pairs far closer together than their
// distance from the centre); separations are exact differences of the hi
// parts plus the difference of the lo parts; r^2 keeps each square's
// rounding error; 1/r is
// the hardware estimate refined by one Newton step whose residual 1 - r^2 y^2
// is formed in float-float; m / r is added to float-float sums, folded into
// doubles after every rotation.  Two j-particles at a time in packed operations
// (the _rn intrinsics are never contracted, which would break the transformations).
struct FF2 {
  float2 h, l;
};
__device__ __forceinline__ FF2 two_sum2(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b);
  const float2 bb = __fadd2_rn(s, neg(a));
  return {s, __fadd2_rn(__fadd2_rn(a, neg(__fadd2_rn(s, neg(bb)))), __fadd2_rn(b, neg(bb)))};
}
// s += (h, l)
__device__ __forceinline__ void add_ff(FF2& s, float2 h, float2 l) {
  const FF2 t = two_sum2(s.h, h);
  s.h = t.h;
  s.l = __fadd2_rn(s.l, __fadd2_rn(t.l, l));
}
// m / r as a pair: m (hi, lo) times y (hi, lo)
__device__ __forceinline__ FF2 mul_ff(float2 mh, float2 ml, float2 yh, float2 yl) {
  const float2 p = __fmul2_rn(mh, yh);
  return {p, __ffma2_rn(mh, yl, __ffma2_rn(ml, yh, __ffma2_rn(mh, yh, neg(p))))};
}

struct SplitF {
  float h, l;
};
__device__ __forceinline__ SplitF split_double(double x) {
  const float h = __double2float_rn(x);
  return {h, __double2float_rn(x - (double)h)};
}

// A lane's i-particles: hi and lo parts, coordinates negated.
struct PairIFF {
  float2 xh[2], xl[2], yh[2], yl[2], zh[2], zl[2], mh[2], ml[2];
};

// 64 i-particles of a warp (two a lane) against 64 j-particles, as rotation().
template <bool SAFE>
__device__ __forceinline__ void rotation_ff(const PairIFF& pi, const float4* hxy, const float4* hzm, const float4* lxy,
                                            const float4* lzm, int lane, FF2* part, FF2& sj) {
#pragma unroll
  for (int q = 0; q < 2; ++q) part[q] = {dup(0.f), dup(0.f)};
  sj = {dup(0.f), dup(0.f)};
  const float2 half = dup(0.5f), one = dup(1.f);
#pragma unroll 1
  for (int s = 0; s < 32; ++s) {
    const int k = (lane + s) & 31;
    const float4 ha = hxy[k], hb = hzm[k], la = lxy[k], lb = lzm[k];
    const float2 mjh = make_float2(hb.z, hb.w), mjl = make_float2(lb.z, lb.w);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      // separation: exact difference of the hi parts + difference of the lo parts
      const FF2 dx = two_sum2(make_float2(ha.x, ha.y), pi.xh[q]), dy = two_sum2(make_float2(ha.z, ha.w), pi.yh[q]),
                dz = two_sum2(make_float2(hb.x, hb.y), pi.zh[q]);
      const float2 lx = __fadd2_rn(dx.l, __fadd2_rn(make_float2(la.x, la.y), pi.xl[q]));
      const float2 ly = __fadd2_rn(dy.l, __fadd2_rn(make_float2(la.z, la.w), pi.yl[q]));
      const float2 lz = __fadd2_rn(dz.l, __fadd2_rn(make_float2(lb.x, lb.y), pi.zl[q]));
      // r^2 = sum (h + l)^2 = sum h^2 + (2h + l) l, with the exact rounding
      // error of each h^2, renormalised (all of r^2 may sit in the l parts)
      const float2 px = __fmul2_rn(dx.h, dx.h), py = __fmul2_rn(dy.h, dy.h), pz = __fmul2_rn(dz.h, dz.h);
      const float2 cx = __ffma2_rn(__fadd2_rn(__fadd2_rn(dx.h, dx.h), lx), lx, __ffma2_rn(dx.h, dx.h, neg(px)));
      const float2 cy = __ffma2_rn(__fadd2_rn(__fadd2_rn(dy.h, dy.h), ly), ly, __ffma2_rn(dy.h, dy.h, neg(py)));
      const float2 cz = __ffma2_rn(__fadd2_rn(__fadd2_rn(dz.h, dz.h), lz), lz, __ffma2_rn(dz.h, dz.h, neg(pz)));
      const FF2 s1 = two_sum2(px, py);
      const FF2 s2 = two_sum2(s1.h, pz);
      const FF2 r2 = two_sum2(s2.h, __fadd2_rn(__fadd2_rn(s1.l, s2.l), __fadd2_rn(__fadd2_rn(cx, cy), cz)));
      // 1/r: one Newton step y0 (1 + d/2), d = 1 - r^2 y0^2 in float-float
      const float2 y0 = make_float2(rsqrt_approx(r2.h.x), rsqrt_approx(r2.h.y));
      const float2 t = __fmul2_rn(y0, y0), te = __ffma2_rn(y0, y0, neg(t));
      const float2 u = __fmul2_rn(r2.h, t);
      const float2 ue = __ffma2_rn(r2.l, t, __ffma2_rn(r2.h, te, __ffma2_rn(r2.h, t, neg(u))));
      const float2 d = __fadd2_rn(__fadd2_rn(one, neg(u)), neg(ue));
      const float2 corr = __fmul2_rn(__fmul2_rn(half, y0), d);
      float2 yh = __fadd2_rn(y0, corr), yl = __fadd2_rn(corr, neg(__fadd2_rn(yh, neg(y0))));
      if (SAFE) {  // pairs outside the normal range add nothing
        const bool ok0 = r2.h.x >= 1.17549435e-38f && r2.h.x <= 3.40282347e38f;
        const bool ok1 = r2.h.y >= 1.17549435e-38f && r2.h.y <= 3.40282347e38f;
        yh = make_float2(ok0 ? yh.x : 0.f, ok1 ? yh.y : 0.f);
        yl = make_float2(ok0 ? yl.x : 0.f, ok1 ? yl.y : 0.f);
      }
      const FF2 wi = mul_ff(mjh, mjl, yh, yl), wj = mul_ff(pi.mh[q], pi.ml[q], yh, yl);
      add_ff(part[q], wi.h, wi.l);
      add_ff(sj, wj.h, wj.l);
    }
    sj.h = rotate(sj.h, lane);
    sj.l = rotate(sj.l, lane);
  }
}

__global__ void __launch_bounds__(kPairThreads) k_bound_pairs_ff(BoundArgs a) {
  constexpr int C = kPairChunk<ScfD4>, I = 2;
  __shared__ float4 s_hxy[C / 2], s_hzm[C / 2], s_lxy[C / 2], s_lzm[C / 2];
  __shared__ double s_sum[kPairWarps][C];
  const ScfD4* pos = reinterpret_cast<const ScfD4*>(a.pos);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, A = blockIdx.x;
  for (int p = blockIdx.y; p < a.n_prog; p += gridDim.y) {
    const int64_t o0 = a.prog_off[p], n = a.prog_off[p + 1] - o0;
    const int P = (int)((n + C - 1) / C);
    if (A >= P) continue;  // the same for every thread of the block
    PairIFF pi;
    double acc[I];
#pragma unroll
    for (int q = 0; q < I; ++q) {
      const int64_t i = (int64_t)A * C + warp * (32 * I) + q * 32 + lane;
      const ScfD4 v = i < n ? pos[o0 + i] : ScfD4{1e18, 0.0, 0.0, 0.0};
      const SplitF x = split_double(-v.x), y = split_double(-v.y), z = split_double(-v.z), m = split_double(v.w);
      pi.xh[q] = dup(x.h), pi.xl[q] = dup(x.l);
      pi.yh[q] = dup(y.h), pi.yl[q] = dup(y.l);
      pi.zh[q] = dup(z.h), pi.zl[q] = dup(z.l);
      pi.mh[q] = dup(m.h), pi.ml[q] = dup(m.l);
      acc[q] = 0.0;
    }
    const int rb = a.round0 + blockIdx.z * a.rounds;
    for (int rr = rb == 1 && a.round0 == 1 ? -1 : 0; rr < a.rounds; ++rr) {
      const bool self = rr < 0;
      const int r = self ? 0 : rb + rr;
      if (r > P / 2 || (2 * r == P && A >= r)) break;
      const int B = A + r < P ? A + r : A + r - P;
      __syncthreads();
      for (int k = tid; k < C; k += kPairThreads) {
        const int64_t j = (int64_t)B * C + k;
        const ScfD4 v = j < n ? pos[o0 + j] : ScfD4{-1e18, 0.0, 0.0, 0.0};
        const SplitF x = split_double(v.x), y = split_double(v.y), z = split_double(v.z), m = split_double(v.w);
        float *hxy = reinterpret_cast<float*>(&s_hxy[k / 2]) + (k & 1), *hzm = reinterpret_cast<float*>(&s_hzm[k / 2]) + (k & 1),
              *lxy = reinterpret_cast<float*>(&s_lxy[k / 2]) + (k & 1), *lzm = reinterpret_cast<float*>(&s_lzm[k / 2]) + (k & 1);
        hxy[0] = x.h, hxy[2] = y.h, hzm[0] = z.h, hzm[2] = m.h;
        lxy[0] = x.l, lxy[2] = y.l, lzm[0] = z.l, lzm[2] = m.l;
      }
      __syncthreads();
      for (int c = 0; c < C / 64; ++c) {
        FF2 part[I], sj;
        bool ok = !self;
        if (!self) {
          rotation_ff<false>(pi, s_hxy + 32 * c, s_hzm + 32 * c, s_lxy + 32 * c, s_lzm + 32 * c, lane, part, sj);
          ok = finite2(sj.h) && finite2(sj.l) && finite2(part[0].h) && finite2(part[0].l) && finite2(part[1].h) &&
               finite2(part[1].l);
        }
        if (__any_sync(0xffffffffu, !ok))
          rotation_ff<true>(pi, s_hxy + 32 * c, s_hzm + 32 * c, s_lxy + 32 * c, s_lzm + 32 * c, lane, part, sj);
#pragma unroll
        for (int q = 0; q < I; ++q)
          acc[q] += ((double)part[q].h.x + (double)part[q].l.x) + ((double)part[q].h.y + (double)part[q].l.y);
        *reinterpret_cast<double2*>(&s_sum[warp][64 * c + 2 * lane]) =
            make_double2((double)sj.h.x + (double)sj.l.x, (double)sj.h.y + (double)sj.l.y);
      }
      __syncthreads();
      if (!self) {
        double* out = a.part + (size_t)(gridDim.z + blockIdx.z * a.rounds + rr) * (size_t)a.n_total + o0 + (int64_t)B * C;
        for (int k = tid; k < C && (int64_t)B * C + k < n; k += kPairThreads) {
          double v = 0.0;
#pragma unroll
          for (int w = 0; w < kPairWarps; ++w) v += s_sum[w][k];
          out[k] += v;
        }
      }
    }
#pragma unroll
    for (int q = 0; q < I; ++q) {
      const int64_t i = (int64_t)A * C + warp * (32 * I) + q * 32 + lane;
      if (i < n) a.part[(size_t)blockIdx.z * (size_t)a.n_total + (size_t)(o0 + i)] += acc[q];
    }
    __syncthreads();
  }
}

// Ordered pairs, for samples too small to fill the chip with rounds of chunks (scf_bound_plan):
// block (i-chunk, progenitor, segment) stages its segment of the j-particles through shared
// memory and evaluates every pair of it for the i-particle alone, so a chunk's work is as many
// independent blocks as there are slots, each with a short chain; slot s holds segment s.
// King N = 4096 (us a call): mixed 43, rounds of chunks 80; float-float 102 and 134.
constexpr int kPairSub = 64;  // pair terms summed in single precision (or float-float) before the double add

__device__ __forceinline__ float pair_inv_r1(float r2) {
  const float y = rsqrt_approx(r2);
  return r2 >= 1.17549435e-38f ? y : 0.f;  // as pair_inv_r<true>
}

__global__ void __launch_bounds__(kPairThreads) k_bound_ordered(BoundArgs a) {
  constexpr int kPairI = Elem<float4>::I;
  __shared__ float4 s_j[kPairThreads];
  const float4* pos = reinterpret_cast<const float4*>(a.pos);
  for (int p = blockIdx.y; p < a.n_prog; p += gridDim.y) {
    const int64_t o0 = a.prog_off[p], o1 = a.prog_off[p + 1];
    const int64_t ib = o0 + (int64_t)blockIdx.x * (kPairThreads * kPairI);
    if (ib >= o1) continue;  // the same for every thread of the block
    const int64_t seg = (o1 - o0 + a.slots - 1) / a.slots;
    const int64_t j0 = min(o1, o0 + (int64_t)blockIdx.z * seg), j1 = min(o1, j0 + seg);
    float xi[kPairI], yi[kPairI], zi[kPairI];
    double acc[kPairI];
#pragma unroll
    for (int q = 0; q < kPairI; ++q) {
      const int64_t i = ib + threadIdx.x + q * kPairThreads;
      const float4 pi = i < o1 ? pos[i] : float4{};
      xi[q] = pi.x;
      yi[q] = pi.y;
      zi[q] = pi.z;
      acc[q] = 0.0;
    }
    for (int64_t jb = j0; jb < j1; jb += kPairThreads) {
      const int cnt = (int)min((int64_t)kPairThreads, j1 - jb);
      __syncthreads();
      if ((int)threadIdx.x < cnt) s_j[threadIdx.x] = pos[jb + threadIdx.x];
      __syncthreads();
      for (int s = 0; s < cnt; s += kPairSub) {
        const int e = min(cnt, s + kPairSub);
        float part[kPairI];
#pragma unroll
        for (int q = 0; q < kPairI; ++q) part[q] = 0.f;
#pragma unroll 4
        for (int jj = s; jj < e; ++jj) {
          const float4 pj = s_j[jj];
#pragma unroll
          for (int q = 0; q < kPairI; ++q) {
            const float dx = pj.x - xi[q], dy = pj.y - yi[q], dz = pj.z - zi[q];
            const float r2 = dx * dx + dy * dy + dz * dz;
            // the self pair (and any coincident pair, and non-finite r2) adds nothing
            const float ri = pair_inv_r1(r2);
            part[q] += pj.w * ri;
          }
        }
#pragma unroll
        for (int q = 0; q < kPairI; ++q) acc[q] += (double)part[q];
      }
    }
#pragma unroll
    for (int q = 0; q < kPairI; ++q) {
      const int64_t i = ib + threadIdx.x + q * kPairThreads;
      if (i < o1) a.part[(size_t)blockIdx.z * (size_t)a.n_total + (size_t)i] = acc[q];
    }
  }
}

__device__ __forceinline__ SplitF two_sum1(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__global__ void __launch_bounds__(kPairThreads) k_bound_ordered_ff(BoundArgs a) {
  constexpr int kPairI = Elem<ScfD4>::I;
  __shared__ float4 s_hi[kPairThreads], s_lo[kPairThreads];
  const ScfD4* pos = reinterpret_cast<const ScfD4*>(a.pos);
  for (int p = blockIdx.y; p < a.n_prog; p += gridDim.y) {
    const int64_t o0 = a.prog_off[p], o1 = a.prog_off[p + 1];
    const int64_t ib = o0 + (int64_t)blockIdx.x * (kPairThreads * kPairI);
    if (ib >= o1) continue;  // the same for every thread of the block
    const int64_t seg = (o1 - o0 + a.slots - 1) / a.slots;
    const int64_t j0 = min(o1, o0 + (int64_t)blockIdx.z * seg), j1 = min(o1, j0 + seg);
    SplitF xi[kPairI], yi[kPairI], zi[kPairI];
    double acc[kPairI];
#pragma unroll
    for (int q = 0; q < kPairI; ++q) {
      const int64_t i = ib + threadIdx.x + q * kPairThreads;
      const ScfD4 pi = i < o1 ? pos[i] : ScfD4{};
      xi[q] = split_double(pi.x);
      yi[q] = split_double(pi.y);
      zi[q] = split_double(pi.z);
      acc[q] = 0.0;
    }
    for (int64_t jb = j0; jb < j1; jb += kPairThreads) {
      const int cnt = (int)min((int64_t)kPairThreads, j1 - jb);
      __syncthreads();
      if ((int)threadIdx.x < cnt) {
        const ScfD4 pj = pos[jb + threadIdx.x];
        const SplitF x = split_double(pj.x), y = split_double(pj.y), z = split_double(pj.z), m = split_double(pj.w);
        s_hi[threadIdx.x] = make_float4(x.h, y.h, z.h, m.h);
        s_lo[threadIdx.x] = make_float4(x.l, y.l, z.l, m.l);
      }
      __syncthreads();
      for (int s = 0; s < cnt; s += kPairSub) {
        const int e = min(cnt, s + kPairSub);
        SplitF sum[kPairI];
#pragma unroll
        for (int q = 0; q < kPairI; ++q) sum[q] = {0.f, 0.f};
#pragma unroll 2
        for (int jj = s; jj < e; ++jj) {
          const float4 hj = s_hi[jj], lj = s_lo[jj];
#pragma unroll
          for (int q = 0; q < kPairI; ++q) {
            // separation: exact difference of the hi parts + difference of the lo parts
            const SplitF dx = two_sum1(hj.x, -xi[q].h), dy = two_sum1(hj.y, -yi[q].h), dz = two_sum1(hj.z, -zi[q].h);
            const float lx = __fadd_rn(dx.l, __fsub_rn(lj.x, xi[q].l));
            const float ly = __fadd_rn(dy.l, __fsub_rn(lj.y, yi[q].l));
            const float lz = __fadd_rn(dz.l, __fsub_rn(lj.z, zi[q].l));
            // r^2 = sum (h + l)^2 = sum h^2 + (2h + l) l, with the exact rounding
            // error of each h^2, renormalised (all of r^2 may sit in the l parts)
            const float px = __fmul_rn(dx.h, dx.h), py = __fmul_rn(dy.h, dy.h), pz = __fmul_rn(dz.h, dz.h);
            const float cx = fmaf(__fadd_rn(__fadd_rn(dx.h, dx.h), lx), lx, fmaf(dx.h, dx.h, -px));
            const float cy = fmaf(__fadd_rn(__fadd_rn(dy.h, dy.h), ly), ly, fmaf(dy.h, dy.h, -py));
            const float cz = fmaf(__fadd_rn(__fadd_rn(dz.h, dz.h), lz), lz, fmaf(dz.h, dz.h, -pz));
            const SplitF s1 = two_sum1(px, py);
            const SplitF s2 = two_sum1(s1.h, pz);
            const SplitF r2 = two_sum1(s2.h, __fadd_rn(__fadd_rn(s1.l, s2.l), __fadd_rn(__fadd_rn(cx, cy), cz)));
            const float r2h = r2.h, r2l = r2.l;
            // 1/r: one Newton step y0 (1 + d/2), d = 1 - r^2 y0^2 in float-float
            const float y0 = rsqrt_approx(r2h);
            const float t = __fmul_rn(y0, y0), te = fmaf(y0, y0, -t);
            const float u = __fmul_rn(r2h, t);
            const float ue = fmaf(r2l, t, fmaf(r2h, te, fmaf(r2h, t, -u)));
            const float d = __fsub_rn(__fsub_rn(1.f, u), ue);
            const float corr = __fmul_rn(__fmul_rn(0.5f, y0), d);
            const float yh = __fadd_rn(y0, corr), yl = __fsub_rn(corr, __fsub_rn(yh, y0));
            // m / r into the float-float sum; pairs outside the normal range add nothing
            const bool ok = r2h >= 1.17549435e-38f && r2h <= 3.40282347e38f;
            const float ph = ok ? __fmul_rn(hj.w, yh) : 0.f;
            const float pe = ok ? fmaf(hj.w, yl, fmaf(lj.w, yh, fmaf(hj.w, yh, -ph))) : 0.f;
            const SplitF ns = two_sum1(sum[q].h, ph);
            sum[q] = {ns.h, __fadd_rn(sum[q].l, __fadd_rn(ns.l, pe))};
          }
        }
#pragma unroll
        for (int q = 0; q < kPairI; ++q) acc[q] += (double)sum[q].h + (double)sum[q].l;
      }
    }
#pragma unroll
    for (int q = 0; q < kPairI; ++q) {
      const int64_t i = ib + threadIdx.x + q * kPairThreads;
      if (i < o1) a.part[(size_t)blockIdx.z * (size_t)a.n_total + (size_t)i] = acc[q];
    }
  }
}

template <typename V4>
__global__ void k_bound_finish(BoundArgs a) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n_total) return;
  double pot = 0.0;
  for (int s = 0; s < a.slots; ++s) pot += a.part[(size_t)s * (size_t)a.n_total + (size_t)i];
  const V4 v = reinterpret_cast<const V4*>(a.vel)[i];
  const V4 p = reinterpret_cast<const V4*>(a.pos)[i];
  const double vx = v.x, vy = v.y, vz = v.z;
  const double E = a.kin * (vx * vx + vy * vy + vz * vz) - a.G * pot;
  if (a.E_out) a.E_out[i] = E;
  a.bound[i] = E < 0.0 ? 1 : 0;
  // r^2 = (x x + y y) + z z without contraction, the same rounding as a plain
  // evaluation of that expression; for r^2 >= 0 its bits order like its value
  const double x = p.x, y = p.y, z = p.z;
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z));
  a.key[i] = (unsigned long long)__double_as_longlong(r2);
}

// NB blocks of NT threads per progenitor (select_launch says which): the blocks'
// histograms and sums meet through distributed shared memory, so a radix pass is
// one sweep of the cluster's threads over the particles.
template <int NB>
__device__ __forceinline__ void select_sync() {
  if constexpr (NB == 1) __syncthreads();
  else cg::this_cluster().sync();
}
template <int NB, typename T>
__device__ __forceinline__ T* of_block(T* p, int b) {  // p of the cluster's block b
  if constexpr (NB == 1) return p;
  else return cg::this_cluster().map_shared_rank(p, b);
}
template <typename V4, int NT, int NB>
__global__ void __cluster_dims__(NB, 1, 1) __launch_bounds__(NT) k_select(BoundArgs a) {
  constexpr int NW = NT / 32;
  __shared__ unsigned s_hist[2][256];   // alternating: a pass is read remotely while the next is cleared
  __shared__ unsigned s_scan[256];
  __shared__ double s_m[NW], s_mb;
  __shared__ unsigned long long s_c[NW], s_n;
  __shared__ unsigned s_digit, s_below;
  const int rank = (int)blockIdx.x % NB;
  const int p = blockIdx.x / NB, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t o0 = a.prog_off[p], o1 = a.prog_off[p + 1];
  const int64_t first = o0 + (int64_t)rank * NT + tid;
  constexpr int64_t kStride = (int64_t)NT * NB;
  const V4* pos = reinterpret_cast<const V4*>(a.pos);
  const uint8_t* bound = a.bound;
  const unsigned long long* key = a.key;

  // bound count and bound mass (fixed order: thread strides, shuffle tree, warps and blocks in order)
  unsigned long long c = 0;
  double m = 0.0;
  for (int64_t k = first; k < o1; k += kStride)
    if (bound[k]) {
      ++c;
      m += (double)pos[k].w;
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    c += __shfl_xor_sync(0xffffffffu, c, o);
    m += __shfl_xor_sync(0xffffffffu, m, o);
  }
  if (lane == 0) {
    s_c[warp] = c;
    s_m[warp] = m;
  }
  __syncthreads();
  if (tid == 0) {
    unsigned long long nb = 0;
    double mb = 0.0;
    for (int w = 0; w < NW; ++w) {
      nb += s_c[w];
      mb += s_m[w];
    }
    s_n = nb;
    s_mb = mb;
  }
  select_sync<NB>();
  unsigned long long nb = 0;
  double mb = 0.0;
  for (int b = 0; b < NB; ++b) {
    nb += *of_block<NB>(&s_n, b);
    mb += *of_block<NB>(&s_mb, b);
  }
  unsigned long long krem = 0, prefix = 0;
  if (nb > 0) {
    const double kk = ceil(a.frac * (double)nb);
    krem = kk < 1.0 ? 1ull : (unsigned long long)kk;
    if (krem > nb) krem = nb;
    // radix selection of the k-th smallest key among the bound particles
    for (int pass = 0; pass < 8; ++pass) {
      const int shift = 56 - 8 * pass;
      const unsigned long long hi = pass == 0 ? 0ull : (~0ull << (shift + 8));
      unsigned* hist = s_hist[pass & 1];
      if (tid < 256) hist[tid] = 0u;
      __syncthreads();
      for (int64_t k = first; k < o1; k += kStride) {
        if (!bound[k]) continue;
        const unsigned long long kk2 = key[k];
        if ((kk2 & hi) == prefix) atomicAdd(&hist[(kk2 >> shift) & 255ull], 1u);
      }
      select_sync<NB>();
      // every block adds all the blocks' counts and finds the digit by a scan
      unsigned v = 0, t = 0;
      if (tid < 256) {
        for (int b = 0; b < NB; ++b) v += *of_block<NB>(&hist[tid], b);
        t = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned u = __shfl_up_sync(0xffffffffu, t, o);
          if (lane >= o) t += u;
        }
        if (lane == 31) s_scan[warp] = t;
      }
      __syncthreads();
      if (tid < 256) {
        for (int w = 0; w < warp; ++w) t += s_scan[w];
        if (t >= krem && t - v < krem) {
          s_digit = (unsigned)tid;
          s_below = t - v;
        }
      }
      __syncthreads();
      prefix |= (unsigned long long)s_digit << shift;
      krem -= s_below;
    }
  }
  // key of r_x^2 (0 = the bits of +0.0 when nothing is bound)
  const unsigned long long kx = nb > 0 ? prefix : 0ull;

  // the coefficient set r <= r_x, and its size
  unsigned long long cm = 0;
  for (int64_t k = first; k < o1; k += kStride) {
    const bool in = key[k] <= kx;
    if (a.mask) a.mask[k] = in ? 1 : 0;
    cm += in ? 1ull : 0ull;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cm += __shfl_xor_sync(0xffffffffu, cm, o);
  select_sync<NB>();  // s_n has been read by every block
  if (lane == 0) s_c[warp] = cm;
  __syncthreads();
  if (tid == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < NW; ++w) t += s_c[w];
    s_n = t;
  }
  select_sync<NB>();
  if (rank == 0 && tid == 0) {
    unsigned long long n_in = 0;
    for (int b = 0; b < NB; ++b) n_in += *of_block<NB>(&s_n, b);
    double* st = a.stats + 4 * (size_t)p;
    st[0] = (double)nb;
    st[1] = mb;
    st[2] = sqrt(__longlong_as_double((long long)kx));
    st[3] = (double)n_in;
  }
  select_sync<NB>();  // no block leaves while its shared memory is read
}

// Eigenvalues l1 >= l2 >= l3 of a symmetric 3x3 matrix S (row-major) by the
// trigonometric solution of its characteristic cubic (Smith, Comm. ACM 4, 168,
// 1961): with q = tr S / 3 and p = sqrt(tr((S - qI)^2) / 6), the eigenvalues
// are q + 2p cos(phi + 2 pi j / 3), phi = acos(det((S - qI)/p) / 2) / 3.
__device__ void sym3_eigen(const double* S, double* lam) {
  const double p1 = S[1] * S[1] + S[2] * S[2] + S[5] * S[5];
  const double q = (S[0] + S[4] + S[8]) / 3.0;
  if (p1 == 0.0) {
    double d0 = S[0], d1 = S[4], d2 = S[8], t;
    if (d0 < d1) { t = d0; d0 = d1; d1 = t; }
    if (d1 < d2) { t = d1; d1 = d2; d2 = t; }
    if (d0 < d1) { t = d0; d0 = d1; d1 = t; }
    lam[0] = d0;
    lam[1] = d1;
    lam[2] = d2;
    return;
  }
  const double a0 = S[0] - q, a4 = S[4] - q, a8 = S[8] - q;
  const double p2 = a0 * a0 + a4 * a4 + a8 * a8 + 2.0 * p1;
  const double p = sqrt(p2 / 6.0);
  const double b0 = a0 / p, b4 = a4 / p, b8 = a8 / p, b1 = S[1] / p, b2 = S[2] / p, b5 = S[5] / p;
  const double det = b0 * (b4 * b8 - b5 * b5) - b1 * (b1 * b8 - b5 * b2) + b2 * (b1 * b5 - b4 * b2);
  double r = 0.5 * det;
  r = r < -1.0 ? -1.0 : (r > 1.0 ? 1.0 : r);
  const double phi = acos(r) / 3.0;
  const double two_pi_3 = 2.0943951023931954923;  // 2 pi / 3
  lam[0] = q + 2.0 * p * cos(phi);
  lam[2] = q + 2.0 * p * cos(phi + two_pi_3);
  lam[1] = 3.0 * q - lam[0] - lam[2];
}

__global__ void k_tidal(TidalArgs a) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= a.n_prog) return;
  double R[3] = {0.0, 0.0, 0.0};
  if (a.com)
    for (int i = 0; i < 3; ++i) R[i] = a.com[6 * (size_t)p + i];
  double T[9];
  for (int j = 0; j < 3; ++j) {  // column j: derivative of a_host along x_j (dual numbers)
    Dual x(R[0], j == 0 ? 1.0 : 0.0), y(R[1], j == 1 ? 1.0 : 0.0), z(R[2], j == 2 ? 1.0 : 0.0);
    Dual ax, ay, az;
    scf_host_accel_t<Dual>(a.host, x, y, z, ax, ay, az);
    T[0 + j] = ax.d;
    T[3 + j] = ay.d;
    T[6 + j] = az.d;
  }
  double S[9], lam[3], fro2 = 0.0;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      S[3 * i + j] = 0.5 * (T[3 * i + j] + T[3 * j + i]);
      fro2 += T[3 * i + j] * T[3 * i + j];
    }
  sym3_eigen(S, lam);
  const double fro = sqrt(fro2);
  const double l1e = lam[0] - 0.5 * (lam[1] + lam[2]);
  const double Mc = a.M_c ? a.M_c[(size_t)p * a.M_stride] : 0.0;
  double* o = a.out + 16 * (size_t)p;
  for (int i = 0; i < 9; ++i) o[i] = T[i];
  o[9] = lam[0];
  o[10] = lam[1];
  o[11] = lam[2];
  o[12] = fro;
  o[13] = l1e;
  o[14] = l1e > 0.0 ? cbrt(a.G * Mc / l1e) : CUDART_INF;
  o[15] = fro > 0.0 ? sqrt(a.eta) / sqrt(fro / sqrt(6.0)) : CUDART_INF;
}

}  // namespace

static int64_t scf_bound_chunk(int f32) { return f32 ? kPairChunk<float4> : kPairChunk<ScfD4>; }

// Rounds of chunks or ordered pairs.  Both evaluate about 3e12 pairs a second in single
// precision and 3.6e11 in float-float when the chip is full, of C^2 (P + P (P - 1) / 2) for the
// P chunks of a progenitor and of C P n, and a call over rounds takes the time of kLag pairs more:
// its shortest chain is a chunk against itself and one other.  Calls, ordered / rounds (us):
//   mixed  1 x 8000 72/87, 12000 107/99, 16384 163/124; 4 x 3000 46/79, 8000 146/109; 16 x 3000 90/88;
//          64 x 1000 54/76, 2000 138/127; 304 x 1000 150/154; 2048 x 64 136/290, 700 637/697, 1000 869/733
//   double 1 x 4096 102/134, 6000 170/151; 4 x 1000 46/128, 3000 169/147; 64 x 300 65/128, 1000 259/248;
//          2048 x 300 997/1403, 700 3192/2494
BoundPlan scf_bound_plan(const int64_t* offsets, int n_prog, int f32, int n_sm) {
  BoundPlan pl;
  const int64_t C = scf_bound_chunk(f32);
  const double kLag = f32 ? 6e7 : 1.2e7;
  double ordered = 0.0, rounds = kLag;
  for (int p = 0; p < n_prog; ++p) {
    const int64_t n = offsets[p + 1] - offsets[p], P = (n + C - 1) / C;
    pl.chunks += P;
    pl.max_chunks = std::max(pl.max_chunks, P);
    ordered += (double)C * P * n;
    rounds += (double)C * C * (P + 0.5 * P * (P - 1.0));
  }
  pl.ordered = ordered <= rounds;
  if (pl.ordered) {  // about four blocks an SM
    const int64_t s = pl.chunks > 0 ? (4 * (int64_t)n_sm + pl.chunks - 1) / pl.chunks : 1;
    pl.slots = (int)std::min<int64_t>(s, kBoundMaxSegments);
  } else {
    // Blocks of a launch: as many groups as leave about 32 blocks an SM, a few waves of short
    // blocks (with eight, King N = 1e5 in double precision ran 1.5 waves a launch).  Rounds a
    // block: so many that a launch takes about 2 ms, since its start and end cost some 10 us (one
    // round a block took 144.5 ms at N = 1e6 in single precision where 20 took 140.1, and 14.68
    // ms where 14.45 for ten progenitors of 1e5); each takes a slot, 8 N bytes that every call
    // clears and reads.
    const int64_t total = pl.max_chunks / 2, groups = (32 * (int64_t)n_sm + pl.chunks - 1) / pl.chunks;
    pl.groups = (int)std::max<int64_t>(1, std::min({groups, total, (int64_t)kBoundMaxSlots / 2}));
    const int64_t per = (int64_t)((f32 ? 6e9 : 7.2e8) / ((double)pl.chunks * pl.groups * C * C)) + 1;
    const int64_t most = std::min<int64_t>(kBoundMaxSlots / pl.groups - 1, (total + pl.groups - 1) / pl.groups);
    pl.rounds = (int)std::max<int64_t>(1, std::min(per, most));
    pl.slots = pl.groups * (1 + pl.rounds);
  }
  return pl;
}

// A progenitor's selection is ten sweeps over its particles with block barriers between
// them.  A cluster of eight blocks has an eighth of the sweep and dearer barriers, and
// takes eight blocks' room (two blocks of 1024 threads an SM): it pays for a large
// progenitor while the clusters run in a few waves.  Whole calls, one block / cluster
// (us): mixed 1 x 4096 43/52, 12000 107/107, 16384 163/156, 65536 1930/1812, 4 x 8000
// 146/148, 16 x 12000 995/1005, 24000 3289/3276, 64 x 8000 1513/1561, 2048 x 64 136/1678.
// Up to 1024 particles a block of 256 threads leaves nobody idle and eight fit an SM:
// 304 x 64 27 against 35, 2048 x 300 171 against 239, 1 x 2000 36 against 33.
template <typename V4>
static void select_launch(const BoundArgs& a, cudaStream_t s) {
  const int64_t waves = (8 * (int64_t)a.n_prog + 2 * a.n_sm - 1) / (2 * a.n_sm);
  if (waves < 8 && a.max_n * (8 - waves) >= 156000 * waves - 58500) k_select<V4, 1024, 8><<<8 * a.n_prog, 1024, 0, s>>>(a);
  else if (a.max_n > 1024) k_select<V4, 1024, 1><<<a.n_prog, 1024, 0, s>>>(a);
  else k_select<V4, 256, 1><<<a.n_prog, 256, 0, s>>>(a);
}

cudaError_t scf_bound_launch(const BoundArgs& a, const BoundPlan& pl, cudaStream_t s) {
  if (a.n_total > 0) {
    const unsigned gy = (unsigned)(a.n_prog < 65535 ? a.n_prog : 65535);
    if (pl.ordered) {
      const dim3 grid((unsigned)pl.max_chunks, gy, (unsigned)pl.slots);
      if (a.f32) k_bound_ordered<<<grid, kPairThreads, 0, s>>>(a);
      else k_bound_ordered_ff<<<grid, kPairThreads, 0, s>>>(a);
    } else {
      cudaError_t e = cudaMemsetAsync(a.part, 0, sizeof(double) * (size_t)a.slots * (size_t)a.n_total, s);
      if (e != cudaSuccess) return e;
      const int64_t total = pl.max_chunks / 2;  // rounds of the largest progenitor
      BoundArgs b = a;
      b.rounds = pl.rounds;
      for (int64_t r = 1; r == 1 || r <= total; r += (int64_t)pl.groups * pl.rounds) {
        b.round0 = (int)r;
        const dim3 grid((unsigned)pl.max_chunks, gy, (unsigned)pl.groups);
        if (a.f32) k_bound_pairs<<<grid, kPairThreads, 0, s>>>(b);
        else k_bound_pairs_ff<<<grid, kPairThreads, 0, s>>>(b);
      }
    }
    const unsigned fb = (unsigned)((a.n_total + 255) / 256);
    if (a.f32) k_bound_finish<float4><<<fb, 256, 0, s>>>(a);
    else k_bound_finish<ScfD4><<<fb, 256, 0, s>>>(a);
  }
  return scf_select_launch(a, s);
}

cudaError_t scf_select_launch(const BoundArgs& a, cudaStream_t s) {
  if (a.f32) select_launch<float4>(a, s);
  else select_launch<ScfD4>(a, s);
  return cudaGetLastError();
}

namespace {
// Complete refresh: b = r_50 / div, the scale of the lowest-order density of
// the radial family whose half-mass radius is the bound stars' energy-based
// one (stats from a selection at frac = 0.5); unchanged for a progenitor with
// nothing bound.
__global__ void k_retune_b(const double* stats, double* b_prog, int n_prog, double div) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_prog) return;
  const double* st = stats + 4 * (size_t)p;
  if (st[0] > 0.0 && st[2] > 0.0) b_prog[p] = st[2] / div;
}
}  // namespace

double scf_half_mass_divisor(double alpha) {
  // enclosed mass of the lowest-order density: (t/(1+t))^(alpha+1), t = (r/b)^(1/alpha)
  if (alpha == 1.0) return 1.0 + 1.4142135623730950488;  // Hernquist
  return std::pow(std::pow(2.0, 1.0 / (alpha + 1.0)) - 1.0, -alpha);
}

cudaError_t scf_retune_b_launch(const double* stats, double* b_prog, int n_prog, double alpha, cudaStream_t s) {
  k_retune_b<<<(n_prog + 127) / 128, 128, 0, s>>>(stats, b_prog, n_prog, scf_half_mass_divisor(alpha));
  return cudaGetLastError();
}

cudaError_t scf_tidal_launch(const TidalArgs& a, cudaStream_t s) {
  k_tidal<<<(a.n_prog + 127) / 128, 128, 0, s>>>(a);
  return cudaGetLastError();
}
