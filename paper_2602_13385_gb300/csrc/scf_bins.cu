// Radial bins (scf_bins.h): the stable counting sort of the particles by bin,
// the interpolation tables, and the two small contractions between bins and
// radial orders.
#include <cmath>
#include <type_traits>
#include <vector>

#include "scf_bins.h"

static __constant__ ScfBinConst c_leg;

cudaError_t scf_upload_const_bins(const ScfBinConst* t) { return cudaMemcpyToSymbol(c_leg, t, sizeof(*t)); }

namespace {

template <typename T> struct V4of;
template <> struct V4of<double> { using type = ScfD4; };
template <> struct V4of<float> { using type = float4; };

// Bin of a particle: theta = acos(xi) = 2 atan(1 / sqrt(t)), t = s^(1/alpha), s = r / b.
// In single precision (it only selects the polynomial piece; where rounding moves a
// particle across an edge, |tau| ends a little above 1), but a double-precision handle's
// units are the caller's: the position is divided by b in double, and the square is
// formed from components scaled by a power of two where it would leave the float range
// (at large alpha s = 1e25 is still bins away from the outermost one).
__device__ __forceinline__ float radius_of(float x, float y, float z, float binv) {
  return sqrtf(x * x + y * y + z * z) * binv;  // as the moments and the field form it
}
__device__ __forceinline__ float radius_of(double x, double y, double z, double binv) {
  float u = (float)(x * binv), v = (float)(y * binv), w = (float)(z * binv);
  const float top = fmaxf(fabsf(u), fmaxf(fabsf(v), fabsf(w)));
  const float up = top > 1e18f ? 0x1p-64f : top < 1e-18f ? 0x1p64f : 1.f;
  const float down = top > 1e18f ? 0x1p64f : top < 1e-18f ? 0x1p-64f : 1.f;
  u *= up;
  v *= up;
  w *= up;
  return sqrtf(u * u + v * v + w * w) * down;
}
template <typename T>
__device__ __forceinline__ int bin_of(T x, T y, T z, T binv, float inv_alpha, int K) {
  const float s = radius_of(x, y, z, binv);
  const float t = inv_alpha == 1.f ? s : powf(s, inv_alpha);
  const float th = 2.f * atan2f(1.f, sqrtf(t));
  return min(max((int)(th * ((float)K * 0.318309886f)), 0), K - 1);
}

// Pass 1 of the sort: half kick and drift (step mode), the particle's bin, its
// place among the block's particles of that bin, and the block's counts.  Warp w
// owns the w-th run of 32 J particles; places by match_any within 32 particles and
// per-warp counts, so the order within a bin is the caller's order and the moment
// sums are the same on every run.  All loads of a thread's J particles are in
// flight together; bound by the state's traffic (5 records a particle in step mode).
template <typename T, int J>
__global__ void __launch_bounds__(kBinSortThreads) k_bin_count(BinArgs a) {
  using V4 = typename V4of<T>::type;
  extern __shared__ __align__(16) unsigned smem_u[];
  unsigned short* cnt = reinterpret_cast<unsigned short*>(smem_u);  // [warps][K]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, blk = blockIdx.x, K = a.K;
  for (int i = tid; i < kBinWarps * K / 2; i += kBinSortThreads) smem_u[i] = 0;
  __shared__ T s_b;
  if (tid == 0) s_b = (T)(1.0 / a.b_prog[a.blk_prog[blk]]);
  const float ia = a.inv_alphaf;
  const int64_t k0 = a.blk_begin[blk] + warp * (32 * J) + lane, k1 = a.blk_end[blk];
  V4* pos = reinterpret_cast<V4*>(a.pos);
  V4 p[J];
  const bool step = a.mode == SCF_MODE_STEP;
#pragma unroll
  for (int j = 0; j < J; ++j)
    if (k0 + 32 * j < k1) p[j] = pos[k0 + 32 * j];
  if (step) {
    V4 v[J], g[J];
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (k0 + 32 * j < k1) {
        v[j] = reinterpret_cast<const V4*>(a.vel)[k0 + 32 * j];
        g[j] = reinterpret_cast<const V4*>(a.acc)[k0 + 32 * j];
      }
    const T h = sizeof(T) == 8 ? (T)(0.5 * a.dt) : (T)a.half_dtf, dt = sizeof(T) == 8 ? (T)a.dt : (T)a.dtf;
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (k0 + 32 * j < k1) {
        v[j].x += h * g[j].x;
        v[j].y += h * g[j].y;
        v[j].z += h * g[j].z;
        p[j].x += dt * v[j].x;
        p[j].y += dt * v[j].y;
        p[j].z += dt * v[j].z;
        reinterpret_cast<V4*>(a.vel_out ? a.vel_out : a.vel)[k0 + 32 * j] = v[j];
        pos[k0 + 32 * j] = p[j];
        if (a.pos_copy) reinterpret_cast<V4*>(a.pos_copy)[k0 + 32 * j] = p[j];
      }
  }
  __syncthreads();
  const T binv = s_b;
  unsigned short* c = cnt + warp * K;
  int bin[J], place[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const bool on = k0 + 32 * j < k1;
    bin[j] = K;
    if (on) {
      const bool fin = scf_finite3(p[j].x, p[j].y, p[j].z);
      bin[j] = fin ? bin_of<T>(p[j].x, p[j].y, p[j].z, binv, ia, K) : 0;
      if (a.count_status && !(fin && isfinite(p[j].w))) atomicOr(a.status, 1u);
    }
  }
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const unsigned same = __match_any_sync(0xffffffffu, bin[j]);
    const int rank = __popc(same & ((1u << lane) - 1u));
    int base = 0;
    if (bin[j] < K) base = c[bin[j]];
    __syncwarp();
    if (bin[j] < K && rank == 0) c[bin[j]] = (unsigned short)(base + __popc(same));
    __syncwarp();
    place[j] = base + rank;
  }
  __syncthreads();
  for (int i = tid; i < K; i += kBinSortThreads) {
    unsigned run = 0;
#pragma unroll
    for (int w = 0; w < kBinWarps; ++w) {
      const unsigned t = cnt[w * K + i];
      cnt[w * K + i] = (unsigned short)run;
      run += t;
    }
    a.hist[(size_t)blk * K + i] = run;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < J; ++j)
    if (bin[j] < K) a.code[k0 + 32 * j] = ((unsigned)bin[j] << 16) | (unsigned)(c[bin[j]] + place[j]);
}

// Pass 2: per bin, the counts of a progenitor's blocks become offsets within the
// bin (8 bins, one 32-byte sector of a row, by 128 block slices: a few loads a
// thread, all in flight); the progenitor's last block to finish then scans the
// totals into the first particle, the first moment task and the first field
// block of every bin.
constexpr int kScanX = 8, kScanY = 128;
__global__ void __launch_bounds__(kScanX * kScanY) k_bin_scan(BinArgs a) {
  __shared__ unsigned s[kScanY][kScanX + 1];
  __shared__ unsigned s_w[3][32];
  __shared__ bool s_last;
  const int p = blockIdx.y, K = a.K, tid = threadIdx.x, x = tid & 31, y = tid >> 5;  // lane, warp
  const int b0 = a.prog_blk_off[p], nb = a.prog_blk_off[p + 1] - b0;
  {
    const int i = blockIdx.x * kScanX + tid % kScanX, sl = tid / kScanX;
    const int per = (nb + kScanY - 1) / kScanY, r0 = min(nb, sl * per), r1 = min(nb, r0 + per);
    unsigned sum = 0;
    if (i < K)
#pragma unroll 8
      for (int r = r0; r < r1; ++r) sum += a.hist[(size_t)(b0 + r) * K + i];
    s[sl][tid % kScanX] = sum;
    __syncthreads();
    if (y < kScanX) {  // warp y scans bin y over the slices, four a lane
      unsigned v[4], t = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[j] = s[4 * x + j][y];
        t += v[j];
      }
      unsigned c = t;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned o = __shfl_up_sync(0xffffffffu, c, d);
        if (x >= d) c += o;
      }
      if (x == 31 && blockIdx.x * kScanX + y < K) a.total[(size_t)p * K + blockIdx.x * kScanX + y] = c;
      c -= t;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        s[4 * x + j][y] = c;
        c += v[j];
      }
    }
    __syncthreads();
    if (i < K) {
      unsigned run = s[sl][tid % kScanX];
#pragma unroll 8
      for (int r = r0; r < r1; ++r) {
        unsigned* h = &a.hist[(size_t)(b0 + r) * K + i];
        const unsigned c = *h;
        *h = run;
        run += c;
      }
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    const unsigned t = atomicAdd(&a.ticket[p], 1u);
    s_last = t == gridDim.x - 1;
    if (s_last) a.ticket[p] = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const unsigned* tot = a.total + (size_t)p * K;
  const int pt = (K + 1023) / 1024, i0 = min(K, tid * pt), i1 = min(K, i0 + pt);
  unsigned n[3] = {0, 0, 0};  // particles, moment tasks, field blocks
  for (int k = i0; k < i1; ++k) {
    const unsigned t = __ldcg(&tot[k]);
    n[0] += t;
    n[1] += (t + a.task - 1) / a.task;
    n[2] += (t + kBinFieldTask - 1) / kBinFieldTask;
  }
  unsigned c[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    c[q] = n[q];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned o = __shfl_up_sync(0xffffffffu, c[q], d);
      if (x >= d) c[q] += o;
    }
    if (x == 31) s_w[q][y] = c[q];
  }
  __syncthreads();
  if (y < 3) {  // warp q scans the warps' totals
    const unsigned v = s_w[y][x];
    unsigned t = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned o = __shfl_up_sync(0xffffffffu, t, d);
      if (x >= d) t += o;
    }
    s_w[y][x] = t - v;
  }
  __syncthreads();
  unsigned* out[3] = {a.bin_start, a.task_start, a.field_start};
  unsigned run[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    out[q] += (size_t)p * (K + 1);
    run[q] = s_w[q][y] + c[q] - n[q];
  }
  for (int k = i0; k < i1; ++k) {
    const unsigned t = __ldcg(&tot[k]);
#pragma unroll
    for (int q = 0; q < 3; ++q) out[q][k] = run[q];
    run[0] += t;
    run[1] += (t + a.task - 1) / a.task;
    run[2] += (t + kBinFieldTask - 1) / kBinFieldTask;
  }
  if (tid == 1023) {  // the last thread's run ends at K
#pragma unroll
    for (int q = 0; q < 3; ++q) out[q][K] = run[q];
    a.binv[p] = 1.0 / a.b_prog[p];
  }
}

// Pass 3: every particle to its place.  The bins' offsets are staged in shared
// memory and a particle leaves as whole 32-byte sectors: the scattered accesses
// (one L1 pass a sector) bound this pass.
template <typename T, int J>
__global__ void __launch_bounds__(kBinSortThreads) k_bin_scatter(BinArgs a) {
  using V4 = typename V4of<T>::type;
  extern __shared__ __align__(16) unsigned smem_u[];
  const int blk = blockIdx.x, p = a.blk_prog[blk], K = a.K;
  const int64_t k0 = a.blk_begin[blk] + threadIdx.x, k1 = a.blk_end[blk], o = a.prog_off[p];
  const V4* pos = reinterpret_cast<const V4*>(a.pos_copy ? a.pos_copy : a.pos);
  const unsigned* start = a.bin_start + (size_t)p * (K + 1);
  const unsigned* hist = a.hist + (size_t)blk * K;
  unsigned code[J];
  V4 x[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int64_t k = k0 + j * kBinSortThreads;
    if (k < k1) {
      code[j] = a.code[k];
      x[j] = pos[k];
      if (a.mask != nullptr && a.mask[k] == 0) x[j].w = 0;
    }
  }
  for (int i = threadIdx.x; i < K; i += kBinSortThreads) smem_u[i] = start[i] + hist[i];
  __syncthreads();
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int64_t k = k0 + j * kBinSortThreads;
    if (k < k1) {
      const int bin = (int)(code[j] >> 16);
      const int64_t dst = o + smem_u[bin] + (code[j] & 0xffffu);
      if constexpr (sizeof(T) == 4) {
        const unsigned long long key = (unsigned long long)(unsigned)k | (unsigned long long)(unsigned)bin << 32;
        asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(reinterpret_cast<ScfBinRec*>(a.spos) + dst),
                     "l"((unsigned long long)__float_as_uint(x[j].x) | (unsigned long long)__float_as_uint(x[j].y) << 32),
                     "l"((unsigned long long)__float_as_uint(x[j].z) | (unsigned long long)__float_as_uint(x[j].w) << 32),
                     "l"(key), "l"(0ull)
                     : "memory");
      } else {
        asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(reinterpret_cast<ScfD4*>(a.spos) + dst),
                     "d"(x[j].x), "d"(x[j].y), "d"(x[j].z), "d"(x[j].w)
                     : "memory");
        a.skey[dst] = make_int2((int)k, bin);
      }
    }
  }
}

// hi + lo += v, the rounding error of hi + v kept in lo (Knuth's TwoSum).
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float v) {
  const float t = __fadd_rn(hi, v), b = __fsub_rn(t, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, b)), __fsub_rn(v, b)));
  hi = t;
}
// acc += a b for (high, low) pairs; acc.y collects the low parts unnormalised.
__device__ __forceinline__ void pair_fma(float2& acc, float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, __fmaf_rn(a.x, b.x, -p)));
  two_sum_add(acc.x, acc.y, p);
  acc.y = __fadd_rn(acc.y, e);
}

// Partial coefficient rows from the moments: block (g, p, z) takes the bins g,
// g + groups, ... of progenitor p in order.  A bin's moment rows (one per task)
// are added in order, four values and four rows in flight a thread, then the
// block's two threads of a column add t M to every other of its radial orders (z
// splits them further).  Double precision: T (nmax + 1) FP64 FMAs a column and
// occupied bin, bound by that pipe.  Single precision: the rows by an error-free
// two-sum and the products and their sums as (high, low) float pairs (an FP64 FMA
// takes 64 single-precision slots here, a pair term 12), folded into double at the end.
template <typename T, int NT, int NH>
__global__ void __maxnreg__(64) k_transform(TransformArgs a) {
  extern __shared__ double s_m[];  // [NT][colpad], pairs of floats in single precision
  using V = typename std::conditional<sizeof(T) == 8, ScfD4, float4>::type;
  using M = typename std::conditional<sizeof(T) == 8, double, float2>::type;
  M* sm = reinterpret_cast<M*>(s_m);
  const int p = blockIdx.y, colpad = a.colpad, EV = NT * colpad / 4;
  const int nq = gridDim.z * (blockDim.x / colpad);
  const int col = threadIdx.x % colpad, q = blockIdx.z * (blockDim.x / colpad) + threadIdx.x / colpad;
  const int lmax = a.lmax, NN = a.nmax + 1;
  int l = 0;
  while ((l + 1) * (l + 1) <= col) ++l;
  const bool live = l <= lmax;
  const unsigned* ts = a.task_start + (size_t)p * (a.K + 1);
  const V* rows = reinterpret_cast<const V*>(a.rows) + (size_t)a.row_off[p] * EV;
  M acc[NH];
#pragma unroll
  for (int i = 0; i < NH; ++i) acc[i] = M{};
  for (int bin = blockIdx.x; bin < a.K; bin += a.groups) {
    const int r0 = (int)ts[bin], r1 = (int)ts[bin + 1];
    if (r0 == r1) continue;  // the same for the whole block
    __syncthreads();
    for (int ev = threadIdx.x; ev < EV; ev += blockDim.x) {
      T hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
      for (int k = r0; k < r1; k += 4) {
        V v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (k + j < r1) v[j] = rows[(size_t)(k + j) * EV + ev];
          else v[j].x = v[j].y = v[j].z = v[j].w = 0;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const T w[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            if constexpr (sizeof(T) == 8) hi[c] += w[c];
            else two_sum_add(hi[c], lo[c], w[c]);
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if constexpr (sizeof(T) == 8) sm[4 * ev + c] = hi[c];
        else sm[4 * ev + c] = make_float2(hi[c], lo[c]);
      }
    }
    __syncthreads();
    if (live) {
      M m[NT];
#pragma unroll
      for (int d = 0; d < NT; ++d) {
        m[d] = sm[d * colpad + col];
        if constexpr (sizeof(T) == 4) {  // renormalised, as the products need
          const float t = __fadd_rn(m[d].x, m[d].y);
          m[d].y = __fsub_rn(m[d].y, __fsub_rn(t, m[d].x));
          m[d].x = t;
        }
      }
      const size_t t0 = ((size_t)bin * (lmax + 1) + l) * NN * NT;
#pragma unroll
      for (int i = 0; i < NH; ++i) {
        const int n = nq * i + q;
        if (n < NN) {
#pragma unroll
          for (int d = 0; d < NT / 2; ++d) {
            if constexpr (sizeof(T) == 8) {
              const double2 v = __ldg(reinterpret_cast<const double2*>(a.t + t0) + n * (NT / 2) + d);
              acc[i] += v.x * m[2 * d];
              acc[i] += v.y * m[2 * d + 1];
            } else {
              const float4 v = __ldg(reinterpret_cast<const float4*>(a.t2 + t0) + n * (NT / 2) + d);
              pair_fma(acc[i], make_float2(v.x, v.y), m[2 * d]);
              pair_fma(acc[i], make_float2(v.z, v.w), m[2 * d + 1]);
            }
          }
        }
      }
    }
  }
  double* out = a.partials + ((size_t)p * a.groups + blockIdx.x) * 2 * a.nc;
  if (live) {
    const int m = col - l * l;  // cosine m = 0..l, then sine m - l = 1..l
    const int lm = m <= l ? scf_lm(l, m) : scf_lm(l, m - l);
    const int idx = m <= l ? lm : a.nc + lm;
#pragma unroll
    for (int i = 0; i < NH; ++i) {
      const int n = nq * i + q;
      if (n < NN) {
        if constexpr (sizeof(T) == 8) out[n * a.nlm + idx] = acc[i];
        else out[n * a.nlm + idx] = ((double)acc[i].x + (double)acc[i].y) * c_leg.sig[lm];
        if (m == 0) out[a.nc + n * a.nlm + idx] = 0.0;
      }
    }
  }
}

// Field rows: block (bin, p), thread ((l, m), n mod slices); the slices' sums
// are added in order through shared memory.
template <typename T> constexpr int kRowSlices = sizeof(T) == 8 ? 2 : 4;
template <typename T, int NT>
__global__ void __launch_bounds__(384) k_field_rows(FieldRowArgs a) {
  using V2 = typename std::conditional<sizeof(T) == 8, double2, float2>::type;
  constexpr int NQ = kRowSlices<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V2* part = reinterpret_cast<V2*>(smem_raw);  // [slices][NT][(l, m)] (cosine, sine)
  const int p = blockIdx.y, bin = blockIdx.x;
  if (a.total[(size_t)p * a.K + bin] == 0) return;
  const int L = a.L, NN = a.nmax + 1, nl = (L + 1) * (L + 2) / 2;
  const int lm = threadIdx.x % nl, q = threadIdx.x / nl;
  if (q < NQ) {
    int l = 0;
    while ((l + 1) * (l + 2) / 2 <= lm) ++l;
    V2 c[NT];
#pragma unroll
    for (int d = 0; d < NT; ++d) c[d].x = c[d].y = 0;
    if (l <= a.lmax) {
      const V2* F = reinterpret_cast<const V2*>(a.F) + (size_t)p * a.nc + lm;
      const V2* t = reinterpret_cast<const V2*>(reinterpret_cast<const T*>(a.t) + ((size_t)bin * (a.lmax + 1) + l) * NN * NT);
#pragma unroll 6
      for (int n = q; n < NN; n += NQ) {
        const V2 f = F[(size_t)n * a.nlm];
#pragma unroll
        for (int d = 0; d < NT / 2; ++d) {
          const V2 v = __ldg(&t[n * (NT / 2) + d]);
          c[2 * d].x += f.x * v.x;
          c[2 * d].y += f.y * v.x;
          c[2 * d + 1].x += f.x * v.y;
          c[2 * d + 1].y += f.y * v.y;
        }
      }
    }
#pragma unroll
    for (int d = 0; d < NT; ++d) part[(q * NT + d) * nl + lm] = c[d];
  }
  __syncthreads();
  T* row = reinterpret_cast<T*>(a.P) + ((size_t)p * a.K + bin) * scf_bin_row(L, NT);
  for (int e = threadIdx.x; e < NT * nl; e += blockDim.x) {
    V2 v = part[e];
#pragma unroll
    for (int k = 1; k < NQ; ++k) {
      const V2 w = part[k * NT * nl + e];
      v.x += w.x;
      v.y += w.y;
    }
    const int d = e / nl, i = e - d * nl;
    int l = 0;
    while ((l + 1) * (l + 2) / 2 <= i) ++l;
    const int m = i - l * (l + 1) / 2;
    const T sig = (T)c_leg.sig[i];
    v.x *= sig;
    v.y *= sig;
    if (m == 0) row[l * NT + d] = v.x;
    else *reinterpret_cast<V2*>(row + scf_bin_off(L, NT, l, m) + 2 * d) = v;
  }
}

// Double-double arithmetic (Dekker 1971, Knuth's TwoSum, FMA-based products)
// for the tables: their rounding is shared by every particle of a bin, so they
// are formed to full double precision.
struct DD {
  double h, l;
};
__device__ __forceinline__ DD dd_fast(double a, double b) {
  const double s = __dadd_rn(a, b);
  return {s, __dsub_rn(b, __dsub_rn(s, a))};
}
__device__ __forceinline__ DD dd_add(DD a, DD b) {
  const double s = __dadd_rn(a.h, b.h), bb = __dsub_rn(s, a.h);
  const double e = __dadd_rn(__dsub_rn(a.h, __dsub_rn(s, bb)), __dsub_rn(b.h, bb));
  return dd_fast(s, __dadd_rn(e, __dadd_rn(a.l, b.l)));
}
__device__ __forceinline__ DD dd_mul(DD a, DD b) {
  const double p = __dmul_rn(a.h, b.h);
  const double e = __fma_rn(a.h, b.h, -p);
  return dd_fast(p, __fma_rn(a.h, b.l, __fma_rn(a.l, b.h, e)));
}
__device__ __forceinline__ DD dd_muld(DD a, double b) {
  const double p = __dmul_rn(a.h, b);
  return dd_fast(p, __fma_rn(a.l, b, __fma_rn(a.h, b, -p)));
}
__device__ __forceinline__ DD dd_divd(DD a, double b) {
  const double q = a.h / b;
  const double r = __fma_rn(-q, b, a.h);
  return dd_fast(q, (r + a.l) / b);
}
// s += a b, the low parts collected unnormalised.
__device__ __forceinline__ void dd_acc(DD& s, DD a, DD b) {
  const double p = __dmul_rn(a.h, b.h);
  const double e = __fma_rn(a.l, b.h, __fma_rn(a.h, b.l, __fma_rn(a.h, b.h, -p)));
  const double t = __dadd_rn(s.h, p), bb = __dsub_rn(t, s.h);
  const double r = __dadd_rn(__dsub_rn(s.h, __dsub_rn(t, bb)), __dsub_rn(p, bb));
  s.l = __dadd_rn(s.l, __dadd_rn(r, e));
  s.h = t;
}

// Bin frames: q_c and inv = 2 / (q range), rounded to the element type so that
// the tables are exact for the tau that the kernels form.
__global__ void k_bin_frame(BinTableArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.K) return;
  const double s0 = sinpi(0.5 * i / a.K), s1 = sinpi(0.5 * (i + 1) / a.K);
  const double q0 = s0 * s0, q1 = s1 * s1;
  const double qc = 0.5 * (q0 + q1), inv = 2.0 / (q1 - q0);
  if (a.f32) reinterpret_cast<float2*>(a.frame)[i] = make_float2((float)qc, (float)inv);
  else reinterpret_cast<double2*>(a.frame)[i] = make_double2(qc, inv);
}

// Interpolation polynomials of degree l in a bin: one group of GW lanes per
// (bin, l).  Lane j < T - 1 runs the Gegenbauer recurrence of dC_n/dtau
// (2 lambda dxi/dtau C_{n-1}^(lambda+1)) at node j, lane T - 1 that of C_n at tau = 0;
// the derivative's node values become monomial coefficients and are integrated.
// Bound by the FP64 pipe: the recurrences carry n! C_n, without a division a step
// (1 / n! is folded into the last product), and the nodes are symmetric, so even
// coefficients take the sums of node pairs and odd ones the differences ((20,10),
// K = 1664: 1251 us with a division a step and full products, 631 with these).
template <int GW, int T>
__global__ void __launch_bounds__(32) k_bin_table(BinTableArgs a) {
  extern __shared__ DD s_f[];  // [32 / GW][nmax + 1][GW]
  constexpr int ND = T - 1, H = ND / 2;
  static_assert(ND % 2 == 1 && T <= GW, "");
  const int lane = threadIdx.x, g = lane / GW, j = lane % GW;
  const int NN = a.nmax + 1;
  const int item = blockIdx.x * (32 / GW) + g;
  const bool on = item < a.K * (a.lmax + 1);
  const int bin = on ? item / (a.lmax + 1) : 0, l = on ? item % (a.lmax + 1) : 0;
  DD* f = s_f + g * NN * GW;
  double qc, inv;
  if (a.f32) {
    const float2 v = reinterpret_cast<const float2*>(a.frame)[bin];
    qc = v.x;
    inv = v.y;
  } else {
    const double2 v = reinterpret_cast<const double2*>(a.frame)[bin];
    qc = v.x;
    inv = v.y;
  }
  const double lam = (2.0 * l + 1.0) * a.alpha + 0.5;
  const DD hw = dd_divd({2.0, 0.0}, inv);  // dxi/dtau
  if (j <= ND) {
    const bool value = j == ND;
    DD xi = dd_add({1.0, 0.0}, {-2.0 * qc, 0.0});
    if (!value) xi = dd_add(xi, dd_mul(hw, {a.nodes[j], a.nodes[ND + j]}));
    const double al = value ? lam : lam + 1.0;
    DD c1 = {0.0, 0.0}, c0 = value ? DD{1.0, 0.0} : dd_mul({2.0 * lam, 0.0}, hw);
    // value lane: f[n] = n! C_n; derivative lanes: f[n] = (n - 1)! dC_n/dtau
    const int shift = value ? 0 : 1;
    if (!value) f[j] = {0.0, 0.0};
    if (shift < NN) f[shift * GW + j] = c0;
    for (int n = 1; n + shift < NN; ++n) {
      const double v = n + 2.0 * al - 2.0, w = -(n - 1.0) * v;
      const DD c = dd_add(dd_muld(dd_mul(xi, c0), 2.0 * (n + al - 1.0)), dd_mul(c1, {w, __fma_rn(-(n - 1.0), v, -w)}));
      c1 = c0;
      c0 = c;
      f[(n + shift) * GW + j] = c;
    }
  }
  __syncwarp();
  if (!on) return;
  for (int n = j; n < NN; n += GW) {
    const size_t at = ((size_t)item * NN + n) * T;
    const double igs = a.inv_gscale[l * NN + n];
    const double2* scale = reinterpret_cast<const double2*>(a.scale) + n * T;
    auto put = [&](int d, DD e) {
      const double2 w = __ldg(scale + d);
      const double v = dd_mul(e, {w.x, w.y}).h;
      if (a.f32) {
        const float hi = (float)v;
        a.tf[at + d] = (float)(v * igs);
        a.t2[at + d] = make_float2(hi, (float)(v - (double)hi));
      } else {
        a.t[at + d] = v;
      }
    };
    const DD* fn = f + n * GW;
    DD sum[H + 1], dif[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const DD u = fn[k], w = fn[ND - 1 - k];
      sum[k] = dd_add(u, w);
      dif[k] = dd_add(u, {-w.h, -w.l});
    }
    sum[H] = fn[H];
    put(0, fn[ND]);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      DD e = {0.0, 0.0};
#pragma unroll
      for (int k = 0; k < (d % 2 == 0 ? H + 1 : H); ++k)
        dd_acc(e, {__ldg(a.vinv + d * ND + k), __ldg(a.vinv + ND * ND + d * ND + k)}, d % 2 == 0 ? sum[k] : dif[k]);
      put(d + 1, e);
    }
  }
}

}  // namespace

void scf_bin_nodes(int T, double* nodes, double* vinv) {
  using LD = long double;
  const int N = T - 1;
  const LD pi = 3.14159265358979323846264338327950288L;
  std::vector<LD> x(N);
  for (int j = 0; j < N; ++j) {  // symmetric to the last bit
    x[j] = 2 * j + 1 == N ? 0.0L : 2 * j + 1 < N ? std::cos((2 * j + 1) * pi / (2 * N)) : -x[N - 1 - j];
    nodes[j] = (double)x[j];
    nodes[N + j] = (double)(x[j] - (LD)nodes[j]);
  }
  // column j of the inverse Vandermonde matrix: the monomial coefficients of the Lagrange polynomial of node j
  for (int j = 0; j < N; ++j) {
    std::vector<LD> c(N, 0.0L);
    c[0] = 1.0L;
    int deg = 0;
    for (int k = 0; k < N; ++k) {
      if (k == j) continue;
      const LD w = 1.0L / (x[j] - x[k]);
      for (int d = ++deg; d >= 0; --d) c[d] = w * ((d > 0 ? c[d - 1] : 0.0L) - x[k] * (d < deg ? c[d] : 0.0L));
    }
    for (int d = 0; d < N; ++d) {
      vinv[d * N + j] = (double)c[d];
      vinv[N * N + d * N + j] = (double)(c[d] - (LD)vinv[d * N + j]);
    }
  }
}

void scf_bin_scale(int T, int nmax, double* scale) {
  using LD = long double;
  LD fact = 1.0L, last = 1.0L;  // n!, (n - 1)!
  for (int n = 0; n <= nmax; ++n) {
    if (n > 0) {
      last = fact;
      fact *= n;
    }
    for (int d = 0; d < T; ++d) {
      const LD v = 1.0L / (d == 0 ? fact : last * d);
      scale[2 * (n * T + d)] = (double)v;
      scale[2 * (n * T + d) + 1] = (double)(v - (LD)(double)v);
    }
  }
}

cudaError_t scf_bin_table_launch(const BinTableArgs& a, cudaStream_t s) {
  k_bin_frame<<<(a.K + 127) / 128, 128, 0, s>>>(a);
  const int items = a.K * (a.lmax + 1);
  const size_t sm = 32 * sizeof(DD) * (size_t)(a.nmax + 1);
  if (a.T == 6) k_bin_table<8, 6><<<(items + 3) / 4, 32, sm, s>>>(a);
  else if (a.T == 8) k_bin_table<8, 8><<<(items + 3) / 4, 32, sm, s>>>(a);
  else k_bin_table<16, 10><<<(items + 1) / 2, 32, sm, s>>>(a);
  return cudaGetLastError();
}

// What every handle may launch with, set once a handle to the same value: the limit
// belongs to the kernel, and a launch must not find it lowered for another handle.
template <typename T, int J>
static cudaError_t sort_prepare() {
  return cudaFuncSetAttribute(k_bin_count<T, J>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(sizeof(unsigned short) * kBinWarps * kBinMaxK));
}

template <typename T, int J>
static cudaError_t sort_t(const BinArgs& a, cudaStream_t s) {
  k_bin_count<T, J><<<a.n_blocks, kBinSortThreads, sizeof(unsigned short) * kBinWarps * a.K, s>>>(a);
  k_bin_scan<<<dim3((a.K + kScanX - 1) / kScanX, a.n_prog), kScanX * kScanY, 0, s>>>(a);
  k_bin_scatter<T, J><<<a.n_blocks, kBinSortThreads, sizeof(unsigned) * a.K, s>>>(a);
  return cudaGetLastError();
}

cudaError_t scf_bin_sort_prepare(int f32, const ScfBinShape& sh) {
  const int J = sh.chunk / kBinSortThreads;
  if (f32) return J == 1 ? sort_prepare<float, 1>() : J == 2 ? sort_prepare<float, 2>() : sort_prepare<float, 4>();
  return J == 1 ? sort_prepare<double, 1>() : J == 2 ? sort_prepare<double, 2>() : sort_prepare<double, 4>();
}

cudaError_t scf_bin_sort_launch(const BinArgs& a, cudaStream_t s) {
  const int J = a.chunk / kBinSortThreads;
  if (a.f32) return J == 1 ? sort_t<float, 1>(a, s) : J == 2 ? sort_t<float, 2>(a, s) : sort_t<float, 4>(a, s);
  return J == 1 ? sort_t<double, 1>(a, s) : J == 2 ? sort_t<double, 2>(a, s) : sort_t<double, 4>(a, s);
}

template <typename T, int NT>
static cudaError_t transform_t(const TransformArgs& a, cudaStream_t s) {
  // radial orders of a thread: (nmax + 1) over 4 (double) or 8 (single) slices,
  // so that all blocks are resident at once
  const int z = sizeof(T) == 8 ? 2 : 4;
  const dim3 grid(a.groups, a.n_prog, z);
  const int threads = 2 * a.colpad, per = (a.nmax + 2 * z) / (2 * z);
  constexpr int kMost = sizeof(T) == 8 ? (SCF_NMAX_CAP + 4) / 4 : (SCF_NMAX_CAP + 8) / 8;
  const size_t sm = sizeof(double) * NT * a.colpad;
  if (per <= 3) k_transform<T, NT, 3><<<grid, threads, sm, s>>>(a);
  else if (per <= 6) k_transform<T, NT, 6><<<grid, threads, sm, s>>>(a);
  else if constexpr (kMost > 6) k_transform<T, NT, kMost><<<grid, threads, sm, s>>>(a);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t scf_transform_launch(const TransformArgs& a, cudaStream_t s) {
  if (a.f32) return a.T == 6 ? transform_t<float, 6>(a, s) : transform_t<float, 8>(a, s);
  return a.T == 8 ? transform_t<double, 8>(a, s) : transform_t<double, 10>(a, s);
}

template <typename T, int NT>
static cudaError_t rows_t(const FieldRowArgs& a, cudaStream_t s) {
  const int nl = (a.L + 1) * (a.L + 2) / 2, threads = (kRowSlices<T> * nl + 31) / 32 * 32;
  k_field_rows<T, NT><<<dim3(a.K, a.n_prog), threads, 2 * sizeof(T) * kRowSlices<T> * NT * nl, s>>>(a);
  return cudaGetLastError();
}

cudaError_t scf_field_rows_launch(const FieldRowArgs& a, cudaStream_t s) {
  if (a.f32) return a.T == 6 ? rows_t<float, 6>(a, s) : rows_t<float, 8>(a, s);
  return a.T == 8 ? rows_t<double, 8>(a, s) : rows_t<double, 10>(a, s);
}
