// Radial bins (scf_bins.h): kernel 3 over particles sorted by radius.
//
// One thread per particle.  Per (l, m >= 1) a thread evaluates the (cosine, sine)
// pair of the polynomial sum_n F_nlm C_n(xi) and its derivative by Horner's rule.
// The order is m outside, l inside: the sums over l at fixed m,
//   a = sum Pt Z, f = sum (l - m) Pt Z (running sums of a), h = sum Pt Z',
//   d = -sum kap Pt_{l,m+1} Z,
// with Pt = k_l Ph_lm, k_l = (1/b) s^(l-1) qa^(2l+1) folded into the Legendre
// recurrence, meet W_m only once:
//   psi += r Re(a W),  A_z += Re(d W),
//   A_n += Re(((1 - 2 s w) f - (2 m + 1) s w a + g h - c d) W),
//   (A_x, A_y) += m (a_c C_{m-1} + a_s S_{m-1}, a_s C_{m-1} - a_c S_{m-1}),
// g = s q w inv / alpha (l - (2l+1) s w is the radial factor's own derivative);
// only two Legendre columns are live.  l = 0 (whose k_0 is singular at the
// origin) is added by itself.
//
// Single precision: blocks of kBinFieldThreads particles of one bin, the bin's
// row staged in shared memory (one broadcast load serves a warp), all the work of
// a (cosine, sine) pair in packed FMAs.  Bound by the FP32 pipe and issue.
// Double precision: bound by the FP64 pipe (2 FMAs per clock and SM), so rows
// come straight from L1 / L2 (the lanes are neighbours in radius: one or two
// rows a warp) and blocks are one warp, which spreads the last wave evenly.
#include "scf_bins.h"

static __constant__ ScfBinConst c_leg;

cudaError_t scf_upload_const_bin_field(const ScfBinConst* t) { return cudaMemcpyToSymbol(c_leg, t, sizeof(*t)); }

namespace {

template <typename T> struct Vec;
template <> struct Vec<double> { using V4 = ScfD4; using V2 = double2; };
template <> struct Vec<float> { using V4 = float4; using V2 = float2; };

__device__ __forceinline__ float power(float x, float y) { return powf(x, y); }
__device__ __forceinline__ double power(double x, double y) { return pow(x, y); }

// (cosine, sine) pairs: packed FMAs in single precision.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) { return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)); }
__device__ __forceinline__ double2 mul2(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 dup(double x) { return make_double2(x, x); }

template <typename T> __device__ __forceinline__ T c_gam(int i) { return sizeof(T) == 8 ? (T)c_leg.gam[i] : (T)c_leg.gamf[i]; }
template <typename T> __device__ __forceinline__ T c_kap(int i) { return sizeof(T) == 8 ? (T)c_leg.kap[i] : (T)c_leg.kapf[i]; }

// NT (cosine, sine) pairs of a row.
template <int NT>
__device__ __forceinline__ void load_pairs(const float* p, float2* c) {
#pragma unroll
  for (int i = 0; i < NT / 2; ++i) {
    const float4 v = *(reinterpret_cast<const float4*>(p) + i);
    c[2 * i] = make_float2(v.x, v.y);
    c[2 * i + 1] = make_float2(v.z, v.w);
  }
}
template <int NT>
__device__ __forceinline__ void load_pairs(const double* p, double2* c) {
#pragma unroll
  for (int i = 0; i < NT; ++i) c[i] = __ldg(reinterpret_cast<const double2*>(p) + i);
}
template <int NT>
__device__ __forceinline__ void load_row(const float* p, float* c) {
#pragma unroll
  for (int i = 0; i < NT / 2; ++i) {
    const float2 v = *(reinterpret_cast<const float2*>(p) + i);
    c[2 * i] = v.x;
    c[2 * i + 1] = v.y;
  }
}
template <int NT>
__device__ __forceinline__ void load_row(const double* p, double* c) {
#pragma unroll
  for (int i = 0; i < NT / 2; ++i) {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p) + i);
    c[2 * i] = v.x;
    c[2 * i + 1] = v.y;
  }
}

// Value z0 and derivative z1 of sum_d c_d tau^d.
template <int NT, typename V>
__device__ __forceinline__ void horner2(const V* c, V tau, V& z0, V& z1) {
  z1 = c[NT - 1];
  z0 = fma2(z1, tau, c[NT - 2]);
#pragma unroll
  for (int d = NT - 3; d >= 0; --d) {
    z1 = fma2(z1, tau, z0);
    z0 = fma2(z0, tau, c[d]);
  }
}
template <int NT, typename T>
__device__ __forceinline__ void horner1(const T* c, T tau, T& z0, T& z1) {
  z1 = c[NT - 1];
  z0 = z1 * tau + c[NT - 2];
#pragma unroll
  for (int d = NT - 3; d >= 0; --d) {
    z1 = z1 * tau + z0;
    z0 = z0 * tau + c[d];
  }
}

// Column m of Pt, l = m .. L, from Pt_mm = K (constant trip counts, so that
// the unrolled accesses stay in registers).
template <typename T, int L>
__device__ __forceinline__ void column(int m, T K, T cS, T S2, T* col) {
#pragma unroll
  for (int l = 1; l <= L; ++l) {
    if (l == m) col[l] = K;
    else if (l == m + 1) col[l] = cS * col[l - 1];
    else if (l > m + 1) col[l] = cS * col[l - 1] - c_gam<T>(scf_lm(l, m)) * (S2 * col[l - 2]);
  }
}

// The block's host values: in single precision as floats (a conversion from
// double runs on the FP64 pipe), with the tidal difference's R-only values.
template <typename T> struct FieldHost;
template <> struct FieldHost<double> {
  double R[3], aR[3], inv_alpha, half_dt;
};
template <> struct FieldHost<float> {
  ScfHostParamsF host;
  float tid[SCF_HOST_CAP][SCF_TIDAL_W];
  float R[3], inv_alpha, alpha, half_dt, binv;
};

// Field of one particle from its bin's row: writes the acceleration (with the
// tide) and the closing kick.
template <typename T, int L, int NT>
__device__ __forceinline__ void field_of(const BinFieldArgs& a, typename Vec<T>::V4 p, int idx,
                                         typename Vec<T>::V2 frame, const T* row, T binv, bool has_host,
                                         const FieldHost<T>& fh, typename Vec<T>::V4 vel) {
  using V4 = typename Vec<T>::V4;
  using V2 = typename Vec<T>::V2;
  const bool finite = scf_finite3(p.x, p.y, p.z);
  if (!finite) atomicOr(a.status, 1u);
  const T x = finite ? p.x : (T)0, y = finite ? p.y : (T)0, z = finite ? p.z : (T)0;
  const T r = sqrt(x * x + y * y + z * z);
  const T rinv = r > (T)0 ? (T)1 / r : (T)0;
  const T u = x * rinv, v = y * rinv, c = z * rinv;
  const T s = r * binv;
  T t = s, w, qa;
  bool gen;
  if constexpr (sizeof(T) == 8) gen = a.alpha != 1.0;
  else gen = fh.alpha != 1.f;
  const T ia = (T)fh.inv_alpha;
  if (gen) t = power(s, ia);
  const T q = (T)1 / ((T)1 + t);
  qa = w = q;
  if (gen) {
    if constexpr (sizeof(T) == 8) qa = power(q, a.alpha);
    else qa = power(q, fh.alpha);
    w = s > (T)0 ? q * power(s, ia - (T)1) : (T)0;
  }
  const T tau = (frame.x - q) * frame.y;
  const T sw = s * w;
  const T gq = ia * q * w * frame.y;  // g = s gq
  const T g = s * gq;
  const T S = s * qa * qa, S2 = S * S, cS = c * S;
  const V2 tau2 = dup(tau);

  T An, Az, pot;
  T nxt[L + 1];
  T K = binv * qa * qa * qa;  // k_1
  {  // m = 0, and the column m = 1
    column<T, L>(1, K, cS, S2, nxt);
    T cf[NT], z0, z1;
    load_row<NT>(row, cf);
    horner1<NT>(cf, tau, z0, z1);
    pot = qa * z0;
    An = binv * qa * (gq * z1 - w * z0);
    T P[L + 1];
    P[1] = c * K;
    if (L >= 2) P[2] = cS * P[1] - c_gam<T>(scf_lm(2, 0)) * (S * K);
#pragma unroll
    for (int l = 3; l <= L; ++l) P[l] = cS * P[l - 1] - c_gam<T>(scf_lm(l, 0)) * (S2 * P[l - 2]);
    T a0 = 0, f0 = 0, h0 = 0, d0 = 0;
#pragma unroll
    for (int l = L; l >= 1; --l) {
      load_row<NT>(row + l * NT, cf);
      horner1<NT>(cf, tau, z0, z1);
      a0 += P[l] * z0;
      f0 += a0;  // sum over l of l Pt z0, as running sums from the top degree
      h0 += P[l] * z1;
      d0 -= (c_kap<T>(scf_lm(l, 0)) * nxt[l]) * z0;
    }
    pot += r * a0;
    An += ((T)1 - 2 * sw) * f0 - sw * a0 + g * h0 - c * d0;
    Az = d0;
  }
  V2 W = dup((T)0);  // W_{m-1}
  W.x = 1;
  const V2 e_f = dup((T)1 - 2 * sw), e_h = dup(g), e_d = dup(-c);
  // (cosine, sine) parts of the sums over m
  V2 tn = dup((T)0), tp = tn, tz = tn, tx = tn, ty = tn;
#pragma unroll
  for (int m = 1; m <= L; ++m) {
    T cur[L + 1];
#pragma unroll
    for (int l = 1; l <= L; ++l) cur[l] = nxt[l];
    K *= S;  // k_{m+1}
    if (m < L) column<T, L>(m + 1, K, cS, S2, nxt);
    V2 sa = dup((T)0), sf = sa, sh = sa, sd = sa;
#pragma unroll
    for (int l = L; l >= 1; --l) {
      if (l < m) continue;
      V2 cf[NT], z0, z1;
      load_pairs<NT>(row + scf_bin_off(L, NT, l, m), cf);
      horner2<NT>(cf, tau2, z0, z1);
      const V2 P = dup(cur[l]);
      sa = fma2(P, z0, sa);
      if (l > m) sf = add2(sf, sa);  // sum of (l - m) Pt Z
      sh = fma2(P, z1, sh);
      if (l > m) sd = fma2(dup(-c_kap<T>(scf_lm(l, m)) * nxt[l]), z0, sd);
    }
    V2 V;  // W_m
    V.x = W.x * u - W.y * v;
    V.y = W.x * v + W.y * u;
    // (1 - 2 s w) (sf + m a) - (s w + m) a = (1 - 2 s w) sf - (2 m + 1) s w a
    const V2 e = fma2(e_f, sf, fma2(dup(-(T)(2 * m + 1) * sw), sa, fma2(e_h, sh, mul2(e_d, sd))));
    tn = fma2(e, V, tn);
    tp = fma2(sa, V, tp);
    tz = fma2(sd, V, tz);
    const V2 am = mul2(dup((T)m), sa);
    tx = fma2(am, W, tx);
    ty.x += am.y * W.x;
    ty.y += am.x * W.y;
    W = V;
  }
  An += tn.x + tn.y;
  pot += r * (tp.x + tp.y);
  Az += tz.x + tz.y;
  const T Ax = tx.x + tx.y, Ay = ty.x - ty.y;
  V4 out;
  out.x = -(An * u + Ax);
  out.y = -(An * v + Ay);
  out.z = -(An * c + Az);
  if (has_host) {  // a_host(R + x) - a_host(R), as in the direct kernel
    if constexpr (sizeof(T) == 8) {
      double hx, hy, hz;
      scf_host_accel(a.host, fh.R[0] + p.x, fh.R[1] + p.y, fh.R[2] + p.z, hx, hy, hz);
      out.x += hx - fh.aR[0];
      out.y += hy - fh.aR[1];
      out.z += hz - fh.aR[2];
    } else {
      float tx, ty, tz;
      scf_tidal_f32(fh.host, fh.tid, fh.R[0], fh.R[1], fh.R[2], p.x, p.y, p.z, tx, ty, tz);
      out.x += tx;
      out.y += ty;
      out.z += tz;
    }
  }
  out.w = pot;
  if (!(isfinite(out.x) && isfinite(out.y) && isfinite(out.z))) atomicOr(a.status, 2u);
  if constexpr (sizeof(T) == 8) {
    if (a.mode == SCF_MODE_ADJ_J) {  // xbar_k += m_k f(x_k; A^J), then the drift is undone, as in the direct kernel
      ScfD4* xb = reinterpret_cast<ScfD4*>(a.adj.xbar) + idx;
      ScfD4 X = *xb;
      X.x += p.w * out.x;
      X.y += p.w * out.y;
      X.z += p.w * out.z;
      *xb = X;
      if (a.adj.drift) {
        ScfD4* vb = reinterpret_cast<ScfD4*>(a.adj.vbar) + idx;
        ScfD4 V = *vb;
        V.x += a.dt * X.x;
        V.y += a.dt * X.y;
        V.z += a.dt * X.z;
        *vb = V;
      }
      return;
    }
  }
  reinterpret_cast<V4*>(a.acc)[idx] = out;
  if (a.mode == SCF_MODE_STEP) {
    const T h = (T)fh.half_dt;
    vel.x += h * out.x;
    vel.y += h * out.y;
    vel.z += h * out.z;
    reinterpret_cast<V4*>(a.vel)[idx] = vel;
  }
}

// The velocity to kick (step mode).
template <typename V4>
__device__ __forceinline__ V4 load_vel(const BinFieldArgs& a, int idx) {
  V4 v{};
  if (a.mode == SCF_MODE_STEP) v = reinterpret_cast<const V4*>(a.vel_in ? a.vel_in : a.vel)[idx];
  return v;
}

// Single precision.
template <int L, int NT>
__global__ void __launch_bounds__(kBinFieldThreads) k_field(BinFieldArgs a) {
  constexpr int ROW = scf_bin_row(L, NT);
  __shared__ __align__(16) float s_row[ROW];
  __shared__ FieldHost<float> s_h;
  __shared__ int s_bin;
  const int tid = threadIdx.x, K = a.K;
  const int prog = a.blk_prog[blockIdx.x];
  const unsigned task = (unsigned)a.blk_task[blockIdx.x];
  const unsigned* fs = a.field_start + (size_t)prog * (K + 1);
  if (task >= fs[K]) return;
  for (int i = tid; i < K; i += kBinFieldThreads)  // the bin with fs[bin] <= task < fs[bin + 1]
    if (fs[i] <= task && task < fs[i + 1]) s_bin = i;
  __syncthreads();
  const int bin = s_bin;
  const unsigned* bs = a.bin_start + (size_t)prog * (K + 1);
  // sorted particles of this block, from the progenitor's first
  const unsigned k0 = bs[bin] + (task - fs[bin]) * kBinFieldTask, k1 = min(bs[bin + 1], k0 + kBinFieldTask);
  const float4* row = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(a.P) + ((size_t)prog * K + bin) * ROW);
  for (int i = tid; i < ROW / 4; i += kBinFieldThreads) reinterpret_cast<float4*>(s_row)[i] = row[i];
  const bool has_host = a.host.n > 0 && a.com != nullptr;
  if (has_host) {
    if (tid < 3) s_h.R[tid] = (float)a.com[6 * prog + tid];
    if (tid < SCF_HOST_CAP) scf_host_f32(a.host, tid, &s_h.host);
    if (tid < a.host.n * SCF_TIDAL_W) (&s_h.tid[0][0])[tid] = a.tid[(size_t)prog * SCF_HOST_CAP * SCF_TIDAL_W + tid];
  }
  if (tid == 32) {
    s_h.inv_alpha = (float)a.inv_alpha;
    s_h.alpha = (float)a.alpha;
    s_h.half_dt = (float)(0.5 * a.dt);
    s_h.binv = (float)a.binv[prog];
  }
  const float2 frame = reinterpret_cast<const float2*>(a.frame)[bin];
  const int64_t o = a.prog_off[prog];
  const ScfBinRec* rec = reinterpret_cast<const ScfBinRec*>(a.spos) + o;
  unsigned k = k0 + tid;
  int idx = 0;
  float4 pos{}, vel{};
  if (k < k1) {  // the first particle's records arrive while the row is staged
    pos = rec[k].p;
    idx = rec[k].key.x;
    vel = load_vel<float4>(a, idx);
  }
  __syncthreads();
  while (k < k1) {
    field_of<float, L, NT>(a, pos, idx, frame, s_row, s_h.binv, has_host, s_h, vel);
    k += kBinFieldThreads;
    if (k < k1) {
      pos = rec[k].p;
      idx = rec[k].key.x;
      vel = load_vel<float4>(a, idx);
    }
  }
}

// Double precision.
template <int L, int NT>
__global__ void __launch_bounds__(kBinField64Threads) k_field64(BinFieldArgs a) {
  const int prog = a.blk_prog[blockIdx.x];
  const int64_t k = a.blk_begin[blockIdx.x] + threadIdx.x;
  if (k >= a.blk_end[blockIdx.x]) return;
  const int2 key = a.skey[k];
  const bool has_host = a.host.n > 0 && a.com != nullptr;
  FieldHost<double> fh{};
  fh.inv_alpha = a.inv_alpha;
  fh.half_dt = 0.5 * a.dt;
  if (has_host)
    for (int d = 0; d < 3; ++d) {
      fh.R[d] = a.com[6 * prog + d];
      fh.aR[d] = a.aR[4 * prog + d];
    }
  const double* row = reinterpret_cast<const double*>(a.P) + ((size_t)prog * a.K + key.y) * scf_bin_row(L, NT);
  field_of<double, L, NT>(a, reinterpret_cast<const ScfD4*>(a.spos)[k], key.x,
                          __ldg(reinterpret_cast<const double2*>(a.frame) + key.y), row, a.binv[prog], has_host, fh,
                          load_vel<ScfD4>(a, key.x));
}

template <typename T, int L, int NT>
cudaError_t launch(const BinFieldArgs& a, int blocks, cudaStream_t s) {
  if constexpr (sizeof(T) == 8) {
    k_field64<L, NT><<<blocks, kBinField64Threads, 0, s>>>(a);
  } else {
    k_field<L, NT><<<blocks, kBinFieldThreads, 0, s>>>(a);
  }
  return cudaGetLastError();
}

template <typename T, int NT>
cudaError_t by_degree(int L, const BinFieldArgs& a, int blocks, cudaStream_t s) {
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

}  // namespace

cudaError_t scf_bin_field_launch(int f32, const ScfBinShape& sh, const BinFieldArgs& a, int blocks, cudaStream_t s) {
  if (f32) return sh.T == 6 ? by_degree<float, 6>(sh.L, a, blocks, s) : by_degree<float, 8>(sh.L, a, blocks, s);
  return sh.T == 8 ? by_degree<double, 8>(sh.L, a, blocks, s) : by_degree<double, 10>(sh.L, a, blocks, s);
}
