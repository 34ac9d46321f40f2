// Radial bins (scf_bins.h): moments of the angular factors over the particles of
// a bin,  M[d][lm] = sum_k tau_k^d  m_k s^l q^((2l+1) alpha) Pb_lm W_m.
//
// One block per task (particles of one bin); its warps take tiles of 32 particles
// in turn, without a block barrier until their sums are added: the lanes form
// the angular columns of 32 particles (one particle a lane, the Legendre
// recurrence along l at fixed m, so two values are live), leave them in the
// warp's shared-memory rows, then turn into columns and add tau^d times them to
// their register sums.  GL lanes cover the columns, 32 / GL sub-groups take
// different particles; their sums are added by shuffles at the end.
//
// Single precision: columns are read four particles at a time (rows of 36
// floats, an odd number of 16-byte words: conflict-free) and the T sums of a
// column run as packed FMAs over particle pairs; bound by shared memory
// (a column value is written and read once: 121 + 128 wavefronts per 32
// particles at lmax = 10) with the FMA pipe close behind.  Double precision:
// bound by the FP64 pipe, T FMAs a column and particle.
#include <type_traits>

#include "scf_bins.h"

static __constant__ ScfBinConst c_leg;

cudaError_t scf_upload_const_bin_moments(const ScfBinConst* t) { return cudaMemcpyToSymbol(c_leg, t, sizeof(*t)); }

namespace {

template <typename T> struct Elem;
template <> struct Elem<double> {
  using V4 = ScfD4;
  static constexpr int kPad = 34, kVec = 2;   // row length, particles per column load
};
template <> struct Elem<float> {
  using V4 = float4;
  static constexpr int kPad = 36, kVec = 4;
};

// Lanes that cover the columns: fewest padded columns at a register count that fits.
__host__ __device__ constexpr int lanes_of(int L) { return L <= 6 ? 8 : 32; }
__host__ __device__ constexpr int cols_per_lane(int L) { return (scf_bin_cols(L) + lanes_of(L) - 1) / lanes_of(L); }

// Warps of a block; rows of a warp: the columns, tau (single) or tau^1..tau^(T-1) (double).
constexpr int warps_of(bool f32) { return f32 ? 4 : 2; }
template <typename T, int L, int NT>
constexpr size_t warp_elems() {
  return (size_t)(scf_bin_cols(L) + (sizeof(T) == 8 ? NT - 1 : 1)) * Elem<T>::kPad;
}

__device__ __forceinline__ float power(float x, float y) { return powf(x, y); }
__device__ __forceinline__ double power(double x, double y) { return pow(x, y); }

// Columns of one particle: Y[l^2 + m] = pre_l P_lm C_m, Y[l^2 + l + m] = pre_l P_lm S_m (P: Ph in
// single, Pb in double precision),
// pre_l = m_k qa (s qa^2)^l folded into the Legendre recurrence.
template <typename T, int L>
__device__ __forceinline__ void columns(T* Y, T pre, T sq2, T u, T v, T c) {
  constexpr int PAD = Elem<T>::kPad;
  const T cS = c * sq2, S2 = sq2 * sq2;
  T Wc = 1, Ws = 0;
#pragma unroll
  for (int m = 0; m <= L; ++m) {
    T p2 = 0, p1 = pre;
    if constexpr (sizeof(T) == 8) p1 *= c_leg.ldiag[m];
#pragma unroll
    for (int l = 0; l <= L; ++l) {
      if (l < m) continue;
      T p = p1;
      if (l > m) {
        const int i = scf_lm(l, m);
        if constexpr (sizeof(T) == 8) {
          p = (c_leg.la[i] * cS) * p1;
          if (l > m + 1) p -= (c_leg.lb[i] * S2) * p2;
        } else {
          p = cS * p1;
          if (l > m + 1) {
            const T t = S2 * p2;
            p -= c_leg.gamf[i] * t;
            if (m == 0) p -= c_leg.gamlo[i] * t;  // a rounded constant leaks the monopole into the even degrees
          }
        }
        p2 = p1;
        p1 = p;
      }
      if (m == 0) {
        Y[(l * l) * PAD] = p;
      } else {
        Y[(l * l + m) * PAD] = p * Wc;
        Y[(l * l + l + m) * PAD] = p * Ws;
      }
    }
    pre *= sq2;
    const T wc = Wc * u - Ws * v;
    Ws = Wc * v + Ws * u;
    Wc = wc;
  }
}

template <typename T, int L, int NT>
__global__ void __launch_bounds__(32 * warps_of(sizeof(T) == 4), 3) k_moments(MomentArgs a) {
  using V4 = typename Elem<T>::V4;
  constexpr int PAD = Elem<T>::kPad, VEC = Elem<T>::kVec;
  constexpr int COLS = scf_bin_cols(L), CP = scf_bin_colpad(L);
  constexpr int GL = lanes_of(L), NG = 32 / GL, CPL = cols_per_lane(L);
  constexpr int W = warps_of(sizeof(T) == 4);
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  T* Y = reinterpret_cast<T*>(smem) + warp * warp_elems<T, L, NT>();
  const int p = a.blk_prog[blockIdx.x], K = a.K;
  const unsigned* ts = a.task_start + (size_t)p * (K + 1);
  const unsigned task = (unsigned)a.blk_task[blockIdx.x];
  if (task >= ts[K]) return;
  // the bin with ts[bin] <= task < ts[bin + 1]: every lane looks at its share at once
  int lo = 0;
  for (int i = lane; i < K; i += 32)
    if (ts[i] <= task && task < ts[i + 1]) lo = i;
  lo = __reduce_max_sync(0xffffffffu, lo);
  const unsigned* bs = a.bin_start + (size_t)p * (K + 1);
  const unsigned nb = bs[lo + 1] - bs[lo], nt = ts[lo + 1] - ts[lo], it = task - ts[lo];
  // the bin's particles in nt near-equal runs of whole tiles
  const unsigned per = ((nb + nt - 1) / nt + 31) / 32 * 32;
  const unsigned k0 = min(nb, it * per), k1 = min(nb, k0 + per);
  // sorted records: ScfBinRec (position first) or ScfD4
  using Rec = typename std::conditional<sizeof(T) == 4, ScfBinRec, ScfD4>::type;
  const Rec* sp = reinterpret_cast<const Rec*>(a.spos) + a.prog_off[p] + bs[lo];
  T qc, inv;
  if constexpr (sizeof(T) == 8) {
    const double2 f = reinterpret_cast<const double2*>(a.frame)[lo];
    qc = f.x;
    inv = f.y;
  } else {
    const float2 f = reinterpret_cast<const float2*>(a.frame)[lo];
    qc = f.x;
    inv = f.y;
  }
  const T binv = (T)a.binv[p];

  const int gl = lane % GL, sg = lane / GL;
  const T* Yc[CPL];  // this lane's columns (columns past the last repeat column 0 and are not written)
#pragma unroll
  for (int j = 0; j < CPL; ++j) Yc[j] = Y + (gl + GL * j < COLS ? gl + GL * j : 0) * PAD;
  T* tau_row = Y + COLS * PAD;
  float2 acc2[sizeof(T) == 4 ? CPL : 1][NT];
  double acc[sizeof(T) == 8 ? CPL : 1][NT];
#pragma unroll
  for (int j = 0; j < CPL; ++j)
#pragma unroll
    for (int d = 0; d < NT; ++d) {
      if constexpr (sizeof(T) == 4) acc2[j][d] = make_float2(0.f, 0.f);
      else acc[j][d] = 0.0;
    }

  V4 next{};  // the next tile's particle, loaded while this tile's columns are summed
  if (k0 + 32 * warp + lane < k1) next = *reinterpret_cast<const V4*>(sp + k0 + 32 * warp + lane);
  for (unsigned base = k0 + 32 * warp; base < k1; base += 32 * W) {
    const unsigned k = base + lane;
    const V4 q = next;
    if (k + 32 * W < k1) next = *reinterpret_cast<const V4*>(sp + k + 32 * W);
    T x = 0, y = 0, z = 0, mass = 0;
    if (k < k1) {
      if (scf_finite3(q.x, q.y, q.z) && isfinite(q.w)) {
        x = q.x;
        y = q.y;
        z = q.z;
        mass = q.w;
      }
    }
    {
      // (the correctly rounded root and reciprocal: an approximation's bias would
      // leak the monopole into l = 2)
      const T r = sqrt(x * x + y * y + z * z);
      const T rinv = r > (T)0 ? (T)1 / r : (T)0;
      const T s = r * binv;
      T t = s, qa;
      const bool gen = sizeof(T) == 8 ? a.alpha != 1.0 : a.alphaf != 1.f;
      if (gen) t = power(s, sizeof(T) == 8 ? (T)a.inv_alpha : (T)a.inv_alphaf);
      const T q = (T)1 / ((T)1 + t);
      qa = q;
      if (gen) qa = power(q, sizeof(T) == 8 ? (T)a.alpha : (T)a.alphaf);
      T tau = (qc - q) * inv;
      if (!(mass != (T)0)) tau = 0;  // lanes past the end and masked or skipped particles add zeros
      if constexpr (sizeof(T) == 4) {
        tau_row[lane] = tau;
      } else {
        T w = tau;
#pragma unroll
        for (int d = 1; d < NT; ++d) {
          tau_row[(d - 1) * PAD + lane] = w;
          w *= tau;
        }
      }
      columns<T, L>(Y + lane, mass * qa, s * qa * qa, x * rinv, y * rinv, z * rinv);
    }
    __syncwarp();
    const int groups = (int)(min(32u, k1 - base) + VEC - 1) / VEC;
    for (int g0 = 0; g0 < groups; g0 += NG) {
      const int g = g0 + sg;
      if (NG > 1 && g >= groups) break;
      if constexpr (sizeof(T) == 4) {
        float2 pw[NT][2];  // tau^d of the four particles (d >= 1)
        const float4 t4 = *reinterpret_cast<const float4*>(tau_row + 4 * g);
        pw[1][0] = make_float2(t4.x, t4.y);
        pw[1][1] = make_float2(t4.z, t4.w);
#pragma unroll
        for (int d = 2; d < NT; ++d) {
          pw[d][0] = __fmul2_rn(pw[d - 1][0], pw[1][0]);
          pw[d][1] = __fmul2_rn(pw[d - 1][1], pw[1][1]);
        }
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
          const float4 y4 = *reinterpret_cast<const float4*>(Yc[j] + 4 * g);
          const float2 ya = make_float2(y4.x, y4.y), yb = make_float2(y4.z, y4.w);
          acc2[j][0] = __fadd2_rn(acc2[j][0], __fadd2_rn(ya, yb));
#pragma unroll
          for (int d = 1; d < NT; ++d) {
            acc2[j][d] = __ffma2_rn(ya, pw[d][0], acc2[j][d]);
            acc2[j][d] = __ffma2_rn(yb, pw[d][1], acc2[j][d]);
          }
        }
      } else {
        double2 pw[NT];
#pragma unroll
        for (int d = 1; d < NT; ++d) pw[d] = *reinterpret_cast<const double2*>(tau_row + (d - 1) * PAD + 2 * g);
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
          const double2 y2 = *reinterpret_cast<const double2*>(Yc[j] + 2 * g);
          acc[j][0] += y2.x + y2.y;
#pragma unroll
          for (int d = 1; d < NT; ++d) {
            acc[j][d] += y2.x * pw[d].x;
            acc[j][d] += y2.y * pw[d].y;
          }
        }
      }
    }
    __syncwarp();
  }
  // the warps' sums, added in warp order (a warp's rows hold NT CP values)
  static_assert(warp_elems<T, L, NT>() >= (size_t)NT * CP, "");
#pragma unroll
  for (int j = 0; j < CPL; ++j) {
    const int col = gl + GL * j;
#pragma unroll
    for (int d = 0; d < NT; ++d) {
      T v;
      if constexpr (sizeof(T) == 4) v = acc2[j][d].x + acc2[j][d].y;
      else v = acc[j][d];
#pragma unroll
      for (int o = GL; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (sg == 0 && col < CP) Y[d * CP + col] = v;
    }
  }
  __syncthreads();
  T* row = reinterpret_cast<T*>(a.rows) + (size_t)(a.row_off[p] + task) * NT * CP;
  const T* Y0 = reinterpret_cast<const T*>(smem);
  for (int e = threadIdx.x; e < NT * CP; e += 32 * W) {
    T v = Y0[e];
#pragma unroll
    for (int w = 1; w < W; ++w) v += Y0[w * warp_elems<T, L, NT>() + e];
    row[e] = v;
  }
}

template <typename T, int L, int NT>
cudaError_t launch(const MomentArgs* a, int blocks, cudaStream_t s) {
  constexpr int W = warps_of(sizeof(T) == 4);
  constexpr size_t sm = sizeof(T) * W * warp_elems<T, L, NT>();
  if (!a) return cudaFuncSetAttribute(k_moments<T, L, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_moments<T, L, NT><<<blocks, 32 * W, sm, s>>>(*a);
  return cudaGetLastError();
}

template <typename T, int NT>
cudaError_t by_degree(int L, const MomentArgs* a, int blocks, cudaStream_t s) {
  switch (L) {
    case 4: return launch<T, 4, NT>(a, blocks, s);
    case 5: return launch<T, 5, NT>(a, blocks, s);
    case 6: return launch<T, 6, NT>(a, blocks, s);
    case 8: return launch<T, 8, NT>(a, blocks, s);
    case 10: return launch<T, 10, NT>(a, blocks, s);
    case 12: return launch<T, 12, NT>(a, blocks, s);
    default: return cudaErrorInvalidValue;
  }
}

// The shape's kernel: launched, or (no arguments) given its shared memory.
cudaError_t by_shape(int f32, const ScfBinShape& sh, const MomentArgs* a, int blocks, cudaStream_t s) {
  if (f32) return sh.T == 6 ? by_degree<float, 6>(sh.L, a, blocks, s) : by_degree<float, 8>(sh.L, a, blocks, s);
  return sh.T == 8 ? by_degree<double, 8>(sh.L, a, blocks, s) : by_degree<double, 10>(sh.L, a, blocks, s);
}

}  // namespace

cudaError_t scf_moments_prepare(int f32, const ScfBinShape& sh) { return by_shape(f32, sh, nullptr, 0, nullptr); }

cudaError_t scf_moments_launch(int f32, const ScfBinShape& sh, const MomentArgs& a, int blocks, cudaStream_t s) {
  return by_shape(f32, sh, &a, blocks, s);
}
