// Radial bins (scf_bins.h): the adjoint's two dual-number passes (scf_adjoint.cu)
// over particles sorted by radius, alpha = 1, double precision.
//
// Both are bound by the FP64 pipe (2 FMAs per clock and SM), so what counts is
// the number of FP64 operations a particle.  The direct dual passes spend 8 FMAs
// (field) and 4 (coefficients) per (n, l, m) and a Gegenbauer recurrence in dual
// numbers; here the radial sums are polynomials of NT terms in the bin's
// coordinate tau, which needs no dual arithmetic: with z0, z1 and z2 the
// polynomial, its derivative and half its second derivative, the dual numbers of
// the sum and of its derivative are (z0, z1 tau.d) and (z1, 2 z2 tau.d).
// King N = 20000 (20,8), GB300: field 265 us, moments 201 us (62% and 47% of the
// FP64 pipe: four or five warps an SM); a run of four steps forward and backward
// 15.3 ms with the direct dual passes, 8.3 ms with these.
#include <type_traits>

#include "scf_adjoint.cuh"
#include "scf_bins.h"

static __constant__ ScfBinConst c_leg;

cudaError_t scf_upload_const_bin_adjoint(const ScfBinConst* t) { return cudaMemcpyToSymbol(c_leg, t, sizeof(*t)); }

namespace {

// Geometry of one particle in dual numbers: n_hat = (u, v, c), s = r / b, q = 1 / (1 + s).
struct Geom {
  Dual r, u, v, c, s, q;
};
__device__ __forceinline__ Geom geometry(Dual x, Dual y, Dual z, double binv) {
  Geom g;
  g.r = sqrt(x * x + y * y + z * z);
  const Dual rinv = g.r.v > 0.0 ? Dual(1.0) / g.r : Dual(0.0);
  g.u = x * rinv;
  g.v = y * rinv;
  g.c = z * rinv;
  g.s = g.r * binv;
  g.q = Dual(1.0) / (Dual(1.0) + g.s);
  return g;
}

// ---------------------------------------------------------------------------
// Field: xbar_k += d/deps a(x_k + eps d_k) at fixed coefficients, the sums of
// scf_bins_field.cu in dual numbers.  One thread per particle, blocks of one warp.
// ---------------------------------------------------------------------------
struct Pair {  // (cosine, sine)
  Dual c, s;
};
__device__ __forceinline__ void add(Pair& a, Dual p, Pair z) {
  a.c += p * z.c;
  a.s += p * z.s;
}

// z0, z1 = sum_d c_d tau^d and its derivative, as dual numbers.
template <int NT, int STEP>
__device__ __forceinline__ void horner(const double* c, Dual tau, Dual& z0, Dual& z1) {
  double p0 = c[(NT - 1) * STEP], p1 = 0.0, p2 = 0.0;
#pragma unroll
  for (int d = NT - 2; d >= 0; --d) {
    p2 = p2 * tau.v + p1;
    p1 = p1 * tau.v + p0;
    p0 = p0 * tau.v + c[d * STEP];
  }
  z0 = Dual(p0, p1 * tau.d);
  z1 = Dual(p1, p2 * (2.0 * tau.d));
}
template <int N>
__device__ __forceinline__ void load(const double* p, double* c) {
  static_assert(N % 2 == 0, "");
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p) + i);
    c[2 * i] = v.x;
    c[2 * i + 1] = v.y;
  }
}

// Column m of Pt, l = m .. L, from Pt_mm = K.
template <int L>
__device__ __forceinline__ void column(int m, Dual K, Dual cS, Dual S2, Dual* col) {
#pragma unroll
  for (int l = 1; l <= L; ++l) {
    if (l == m) col[l] = K;
    else if (l == m + 1) col[l] = cS * col[l - 1];
    else if (l > m + 1) col[l] = cS * col[l - 1] - c_leg.gam[scf_lm(l, m)] * (S2 * col[l - 2]);
  }
}

template <int L, int NT>
__device__ __forceinline__ void field_dual(const Geom& g, double2 frame, const double* row, double binv, double& ax,
                                           double& ay, double& az) {
  const Dual q = g.q, sw = g.s * q, S = sw * q, S2 = S * S, cS = g.c * S;
  const Dual tau((frame.x - q.v) * frame.y, -q.d * frame.y);
  const Dual gq = frame.y * (q * q), gg = g.s * gq;
  const Dual e_f = Dual(1.0) - 2.0 * sw;
  Dual An, Az, z0, z1, nxt[L + 1];
  Dual K = binv * (q * q * q);
  {  // m = 0, and the column m = 1
    column<L>(1, K, cS, S2, nxt);
    double cf[NT];
    load<NT>(row, cf);
    horner<NT, 1>(cf, tau, z0, z1);
    An = binv * (q * (gq * z1 - q * z0));
    Dual P[L + 1];
    P[1] = g.c * K;
    if (L >= 2) P[2] = cS * P[1] - c_leg.gam[scf_lm(2, 0)] * (S * K);
#pragma unroll
    for (int l = 3; l <= L; ++l) P[l] = cS * P[l - 1] - c_leg.gam[scf_lm(l, 0)] * (S2 * P[l - 2]);
    Dual a0, f0, h0, d0;
#pragma unroll
    for (int l = L; l >= 1; --l) {
      load<NT>(row + l * NT, cf);
      horner<NT, 1>(cf, tau, z0, z1);
      a0 += P[l] * z0;
      f0 += a0;
      h0 += P[l] * z1;
      d0 -= (c_leg.kap[scf_lm(l, 0)] * nxt[l]) * z0;
    }
    An += e_f * f0 - sw * a0 + gg * h0 - g.c * d0;
    Az = d0;
  }
  Dual Wc(1.0), Ws(0.0), Ax, Ay;  // W_{m-1}
#pragma unroll
  for (int m = 1; m <= L; ++m) {
    Dual cur[L + 1];
#pragma unroll
    for (int l = 1; l <= L; ++l) cur[l] = nxt[l];
    K *= S;
    if (m < L) column<L>(m + 1, K, cS, S2, nxt);
    Pair sa{}, sf{}, sh{}, sd{};
#pragma unroll
    for (int l = L; l >= 1; --l) {
      if (l < m) continue;
      double cf[2 * NT];
      load<2 * NT>(row + scf_bin_off(L, NT, l, m), cf);
      Pair Z0, Z1;
      horner<NT, 2>(cf, tau, Z0.c, Z1.c);
      horner<NT, 2>(cf + 1, tau, Z0.s, Z1.s);
      add(sa, cur[l], Z0);
      if (l > m) {
        sf.c += sa.c;
        sf.s += sa.s;
      }
      add(sh, cur[l], Z1);
      if (l > m) add(sd, -c_leg.kap[scf_lm(l, m)] * nxt[l], Z0);
    }
    const Dual Vc = Wc * g.u - Ws * g.v, Vs = Wc * g.v + Ws * g.u;  // W_m
    const Dual e_a = -(2.0 * m + 1.0) * sw;
    An += (e_f * sf.c + e_a * sa.c + gg * sh.c - g.c * sd.c) * Vc + (e_f * sf.s + e_a * sa.s + gg * sh.s - g.c * sd.s) * Vs;
    Az += sd.c * Vc + sd.s * Vs;
    Ax += (double)m * (sa.c * Wc + sa.s * Ws);
    Ay += (double)m * (sa.s * Wc - sa.c * Ws);
    Wc = Vc;
    Ws = Vs;
  }
  ax = -(An * g.u + Ax).d;
  ay = -(An * g.v + Ay).d;
  az = -(An * g.c + Az).d;
}

template <int L, int NT>
__global__ void __launch_bounds__(kBinField64Threads) k_field_dual(BinFieldArgs a) {
  static_assert(kBinField64Threads == 32, "one warp a block: the partials are summed by shuffles");
  const int prog = a.blk_prog[blockIdx.x], lane = threadIdx.x;
  const int64_t k = a.blk_begin[blockIdx.x] + lane;
  const bool has_host = a.host.n > 0 && a.com != nullptr;
  double acc[SCF_ADJ_Q];
#pragma unroll
  for (int i = 0; i < SCF_ADJ_Q; ++i) acc[i] = 0.0;
  if (k < a.blk_end[blockIdx.x]) {
    const int2 key = a.skey[k];
    const ScfD4 p = reinterpret_cast<const ScfD4*>(a.spos)[k], vb = reinterpret_cast<const ScfD4*>(a.adj.vbar)[key.x];
    if (scf_finite3(p.x, p.y, p.z) && scf_finite3(vb.x, vb.y, vb.z)) {
      const double w = a.adj.weight, dx = w * vb.x, dy = w * vb.y, dz = w * vb.z;
      const double binv = a.binv[prog];
      const double* row = reinterpret_cast<const double*>(a.P) + ((size_t)prog * a.K + key.y) * scf_bin_row(L, NT);
      double gx, gy, gz;
      field_dual<L, NT>(geometry(Dual(p.x, dx), Dual(p.y, dy), Dual(p.z, dz), binv),
                        __ldg(reinterpret_cast<const double2*>(a.frame) + key.y), row, binv, gx, gy, gz);
      if (has_host)
        scf_adj_tide(a.host, a.com[6 * prog] + p.x, a.com[6 * prog + 1] + p.y, a.com[6 * prog + 2] + p.z, dx, dy, dz, gx,
                     gy, gz, acc);
      if (!(isfinite(gx) && isfinite(gy) && isfinite(gz))) atomicOr(a.status, 2u);
      ScfD4* xb = reinterpret_cast<ScfD4*>(a.adj.xbar) + key.x;
      ScfD4 X = *xb;
      X.x += gx;
      X.y += gy;
      X.z += gz;
      *xb = X;
    } else {
      atomicOr(a.status, 1u);
    }
  }
  if (!has_host) return;
#pragma unroll
  for (int i = 0; i < SCF_ADJ_Q; ++i) {
    double v = acc[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) a.adj.part[(size_t)blockIdx.x * SCF_ADJ_Q + i] = v;
  }
}

// ---------------------------------------------------------------------------
// Coefficients: rows of d/deps sum_k tau_k^d Y_lm(x_k + eps d_k), unit masses,
//   sum_k tau^d (Y.d) + d tau^(d-1) (tau.d Y.v).
// One block, a warp, per task.  The lanes form the columns of 32 particles (Y.d
// and tau.d Y.v, two rows of shared memory a column), then turn into columns and
// add 2 FMAs a term, column and particle to their register sums.  Rows of 33
// doubles: the lanes of both phases hit different banks.
// ---------------------------------------------------------------------------
constexpr int kPad = 33;
__host__ __device__ constexpr int lanes_of(int L) { return L <= 6 ? 8 : 32; }
template <int L, int NT>
constexpr size_t dual_smem() {
  return sizeof(double) * kPad * (2 * (size_t)scf_bin_cols(L) + 2 * NT - 3);
}

template <int L>
__device__ __forceinline__ void store(double* Y, int col, Dual y, double taud) {
  Y[2 * col * kPad] = y.d;
  Y[(2 * col + 1) * kPad] = y.v * taud;
}

template <int L, int NT>
__global__ void __launch_bounds__(32) k_moments_dual(MomentDualArgs a) {
  constexpr int COLS = scf_bin_cols(L), CP = scf_bin_colpad(L);
  constexpr int GL = lanes_of(L), NG = 32 / GL, CPL = (COLS + GL - 1) / GL;
  extern __shared__ __align__(16) double Y[];
  double* Tau = Y + 2 * COLS * kPad;             // tau^1 .. tau^(NT-1)
  double* Slope = Tau + (NT - 1) * kPad;         // 2 tau .. (NT-1) tau^(NT-2)
  const int lane = threadIdx.x, p = a.m.blk_prog[blockIdx.x], K = a.m.K;
  const unsigned* ts = a.m.task_start + (size_t)p * (K + 1);
  const unsigned task = (unsigned)a.m.blk_task[blockIdx.x];
  if (task >= ts[K]) return;
  int bin = 0;  // ts[bin] <= task < ts[bin + 1]
  for (int i = lane; i < K; i += 32)
    if (ts[i] <= task && task < ts[i + 1]) bin = i;
  bin = __reduce_max_sync(0xffffffffu, bin);
  const unsigned* bs = a.m.bin_start + (size_t)p * (K + 1);
  const unsigned nb = bs[bin + 1] - bs[bin], nt = ts[bin + 1] - ts[bin], it = task - ts[bin];
  const unsigned per = ((nb + nt - 1) / nt + 31) / 32 * 32;
  const unsigned k0 = min(nb, it * per), k1 = min(nb, k0 + per);
  const int64_t first = a.m.prog_off[p] + bs[bin];
  const ScfD4* sp = reinterpret_cast<const ScfD4*>(a.m.spos) + first;
  const int2* key = a.skey + first;
  const ScfD4* vbar = reinterpret_cast<const ScfD4*>(a.adj.vbar);
  const double2 frame = reinterpret_cast<const double2*>(a.m.frame)[bin];
  const double binv = a.m.binv[p], w = a.adj.weight;
  const int gl = lane % GL, sg = lane / GL;
  const double* Yc[CPL];  // columns past the last repeat column 0 and are not written
#pragma unroll
  for (int j = 0; j < CPL; ++j) Yc[j] = Y + 2 * (gl + GL * j < COLS ? gl + GL * j : 0) * kPad;
  double acc[CPL][NT];
#pragma unroll
  for (int j = 0; j < CPL; ++j)
#pragma unroll
    for (int d = 0; d < NT; ++d) acc[j][d] = 0.0;

  for (unsigned base = k0; base < k1; base += 32) {
    const unsigned k = base + lane;
    Dual x, y, z;
    if (k < k1) {
      const ScfD4 q = sp[k], vb = vbar[key[k].x];
      if (scf_finite3(q.x, q.y, q.z) && scf_finite3(vb.x, vb.y, vb.z)) {
        x = Dual(q.x, w * vb.x);
        y = Dual(q.y, w * vb.y);
        z = Dual(q.z, w * vb.z);
      }
    }
    {
      const Geom g = geometry(x, y, z, binv);
      const double tau = (frame.x - g.q.v) * frame.y, taud = -g.q.d * frame.y;
      double t = 1.0;
#pragma unroll
      for (int d = 1; d < NT; ++d) {
        if (d > 1) Slope[(d - 2) * kPad + lane] = d * t;
        t *= tau;
        Tau[(d - 1) * kPad + lane] = t;
      }
      const Dual sq2 = g.s * g.q * g.q, cS = g.c * sq2, S2 = sq2 * sq2;
      Dual pre = g.q, Wc(1.0), Ws(0.0);
      double* Yl = Y + lane;
#pragma unroll
      for (int m = 0; m <= L; ++m) {
        Dual p2(0.0), p1 = pre * c_leg.ldiag[m];
#pragma unroll
        for (int l = 0; l <= L; ++l) {
          if (l < m) continue;
          Dual f = p1;
          if (l > m) {
            const int i = scf_lm(l, m);
            f = (c_leg.la[i] * cS) * p1;
            if (l > m + 1) f -= (c_leg.lb[i] * S2) * p2;
            p2 = p1;
            p1 = f;
          }
          if (m == 0) {
            store<L>(Yl, l * l, f, taud);
          } else {
            store<L>(Yl, l * l + m, f * Wc, taud);
            store<L>(Yl, l * l + l + m, f * Ws, taud);
          }
        }
        pre *= sq2;
        const Dual wc = Wc * g.u - Ws * g.v;
        Ws = Wc * g.v + Ws * g.u;
        Wc = wc;
      }
    }
    __syncwarp();
    const int n = (int)min(32u, k1 - base);
    for (int i = sg; i < n; i += NG) {
      double t[NT], e[NT];
#pragma unroll
      for (int d = 1; d < NT; ++d) t[d] = Tau[(d - 1) * kPad + i];
#pragma unroll
      for (int d = 2; d < NT; ++d) e[d] = Slope[(d - 2) * kPad + i];
#pragma unroll
      for (int j = 0; j < CPL; ++j) {
        const double yd = Yc[j][i], yv = Yc[j][kPad + i];
        acc[j][0] += yd;
        acc[j][1] += t[1] * yd + yv;
#pragma unroll
        for (int d = 2; d < NT; ++d) {
          acc[j][d] += t[d] * yd;
          acc[j][d] += e[d] * yv;
        }
      }
    }
    __syncwarp();
  }
  double* row = reinterpret_cast<double*>(a.m.rows) + (size_t)(a.m.row_off[p] + task) * NT * CP;
#pragma unroll
  for (int j = 0; j < CPL; ++j) {
    const int col = gl + GL * j;
#pragma unroll
    for (int d = 0; d < NT; ++d) {
      double v = acc[j][d];
#pragma unroll
      for (int o = GL; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (sg == 0 && col < CP) row[d * CP + col] = v;
    }
  }
}

template <int L, int NT>
cudaError_t moments(const MomentDualArgs* a, int blocks, cudaStream_t s) {
  constexpr size_t sm = dual_smem<L, NT>();
  if (!a) return cudaFuncSetAttribute(k_moments_dual<L, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_moments_dual<L, NT><<<blocks, 32, sm, s>>>(*a);
  return cudaGetLastError();
}

template <int L, int NT>
cudaError_t field(const BinFieldArgs* a, int blocks, cudaStream_t s) {
  k_field_dual<L, NT><<<blocks, kBinField64Threads, 0, s>>>(*a);
  return cudaGetLastError();
}

template <int NT, typename A>
cudaError_t by_degree(int L, const A* a, int blocks, cudaStream_t s) {
  auto run = [&](auto deg) -> cudaError_t {
    constexpr int D = decltype(deg)::value;
    if constexpr (std::is_same<A, BinFieldArgs>::value) return field<D, NT>(a, blocks, s);
    else return moments<D, NT>(a, blocks, s);
  };
  switch (L) {
    case 4: return run(std::integral_constant<int, 4>());
    case 5: return run(std::integral_constant<int, 5>());
    case 6: return run(std::integral_constant<int, 6>());
    case 8: return run(std::integral_constant<int, 8>());
    case 10: return run(std::integral_constant<int, 10>());
    case 12: return run(std::integral_constant<int, 12>());
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t scf_moments_dual_prepare(const ScfBinShape& sh) {
  const MomentDualArgs* none = nullptr;
  return sh.T == 8 ? by_degree<8>(sh.L, none, 0, nullptr) : by_degree<10>(sh.L, none, 0, nullptr);
}

cudaError_t scf_moments_dual_launch(const ScfBinShape& sh, const MomentDualArgs& a, int blocks, cudaStream_t s) {
  return sh.T == 8 ? by_degree<8>(sh.L, &a, blocks, s) : by_degree<10>(sh.L, &a, blocks, s);
}

cudaError_t scf_bin_field_dual_launch(const ScfBinShape& sh, const BinFieldArgs& a, int blocks, cudaStream_t s) {
  return sh.T == 8 ? by_degree<8>(sh.L, &a, blocks, s) : by_degree<10>(sh.L, &a, blocks, s);
}
