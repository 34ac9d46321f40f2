// Radial bins (internal header): the coefficient and field passes over particles
// sorted by radius.
//
// The radial functions of degree l are a prefactor times the polynomials
// C_n(xi), n = 0..nmax.  The range of xi is cut into K bins, uniform in
// theta = acos(xi); in a bin every C_n is replaced by its own polynomial of
// degree T - 1 in the bin's coordinate tau = (q_c - q) inv (xi = 1 - 2 q),
//   C_n^(lambda_l)(xi) = sum_{d < T} t[bin][l][n][d] tau^d,
// interpolated so that value and derivative agree to rounding (the bin's width
// in theta is chosen from the fastest oscillation, nmax + lambda_lmax, and T).
// Largest error of dC_n/dxi over all bins, l and n, relative to its amplitude there
// (the envelope of its oscillation), coarser / finer bins: (20,10), alpha = 1, 2.5e-9
// / 8e-9 for the single-precision pairs of (K, T) and 3.3e-17 / 1.9e-16 for the
// double-precision ones; over (6..40, 3..12) and alpha from 0.1 to 4 at most 3.3e-8
// and 5e-16, at nmax = 40 and alpha = 0.1.  So
//   coefficients  Sh_nlm = sum_bins sum_d t[bin][l][n][d] M[bin][d][lm],
//                 M = the moments sum_k tau_k^d (m_k s^l q^(2l+1) Pb_lm W_m),
//   field         sum_n F_nlm C_n = sum_d P[bin][lm][d] tau^d,
//                 P[bin][lm][d] = sum_n F_nlm t[bin][l][n][d],
// with T terms a particle where the direct sums have nmax + 1, no radial
// recurrence, and the derivative from the same T numbers.  Both directions use
// the same polynomials, so the field stays the exact gradient of the energy
// that the coefficients define.
#pragma once

#include "scf_internal.h"

constexpr int kBinSortThreads = 512;
constexpr int kBinWarps = kBinSortThreads / 32;
constexpr int kBinMaxK = 7168;         // bins that the sort's per-warp counts have room for (224 KB)
constexpr int kBinFieldThreads = 128;  // field block, single precision
constexpr int kBinFieldTask = 256;     // and its particles, all of one bin, at most

// Legendre constants of the binned kernels.  With Pb_lm = sig_lm Ph_lm the
// recurrence along l at fixed m is Ph_lm = c Ph_{l-1,m} - gam_lm Ph_{l-2,m},
// Ph_mm = 1; sig is applied to the coefficient sums and to the field rows, and
// the derivative's lk_lm becomes kap_lm = lk_lm sig_{l,m+1} / sig_lm.
// (The double-precision moments keep the normalised recurrence of the direct
// kernel, ScfConst's la and lb: its rounded constants leak a few 1e-16 of the
// monopole into the even degrees, and so the two paths agree in that too.)
struct ScfBinConst {
  double gam[SCF_NLM_CAP], kap[SCF_NLM_CAP], sig[SCF_NLM_CAP];
  double la[SCF_NLM_CAP], lb[SCF_NLM_CAP], ldiag[SCF_LMAX_CAP + 1];
  float gamf[SCF_NLM_CAP], kapf[SCF_NLM_CAP];
  float gamlo[SCF_NLM_CAP];  // gam - gamf, for the moments at m = 0
};

// Degrees the kernels are compiled for; a smaller lmax runs the next one with
// zero rows.  Columns of a moment row: l*l + m (cosine), l*l + l + m (sine, m >= 1).
__host__ __device__ constexpr int scf_bin_cols(int L) { return (L + 1) * (L + 1); }
__host__ __device__ constexpr int scf_bin_colpad(int L) { return (scf_bin_cols(L) + 31) / 32 * 32; }
// Elements of a field row: m = 0 first (T values a degree, cosine only, padded
// to 4), then for m >= 1, l >= m, T (cosine, sine) pairs.
__host__ __device__ constexpr int scf_bin_row0(int L, int T) { return ((L + 1) * T + 3) / 4 * 4; }
__host__ __device__ constexpr int scf_bin_row(int L, int T) { return scf_bin_row0(L, T) + L * (L + 1) * T; }
// Offset of (l, m), m >= 1, in a field row.
__host__ __device__ constexpr int scf_bin_off(int L, int T, int l, int m) {
  return scf_bin_row0(L, T) + 2 * T * ((m - 1) * L - (m - 1) * (m - 2) / 2 + (l - m));
}

// A sorted particle in single precision: one 32-byte sector, written at once
// (position and masked mass; particle, bin).  In double precision the position
// record fills a sector by itself and (particle, bin) is an array of its own.
struct __align__(32) ScfBinRec {
  float4 p;
  int4 key;
};

// Shape of a handle's bins.
struct ScfBinShape {
  int K, T, L;     // bins, terms, compiled degree
  int groups;      // bin groups of the coefficient transform (rows for kernel 2) per progenitor
  int chunk;       // particles of a sorting block: 512, 1024 or 2048
  int task;        // particles of one moment task (one block) at most
};

struct BinArgs {
  // particles (caller's arrays; modes as in K1Args)
  void* pos;
  void* vel;
  const void* acc;
  void* vel_out;           // step mode: where the half-kicked velocities go (null: vel)
  void* pos_copy;          // step mode, optional: a copy of the drifted positions, read by the scatter
  const uint8_t* mask;
  int mode;
  double dt;
  int f32;
  float dtf, half_dtf, inv_alphaf;  // no conversions from double in the single-precision threads
  const double* b_prog;
  unsigned* status;
  // sorting blocks: chunks of one progenitor
  const int* blk_prog;
  const int64_t* blk_begin;
  const int64_t* blk_end;
  const int* prog_blk_off; // [n_prog + 1]
  const int64_t* prog_off; // [n_prog + 1] particle offsets
  int n_blocks, n_prog;
  int K, chunk, task;
  unsigned* code;          // [N] bin << 16 | place within (block, bin), caller's order
  unsigned* hist;          // [n_blocks][K] counts, then offsets within the bin
  unsigned* total;         // [n_prog][K]
  unsigned* ticket;        // [n_prog] finished scan blocks (0 between passes)
  unsigned* bin_start;     // [n_prog][K + 1] first particle of a bin, from the progenitor's first
  unsigned* task_start;    // [n_prog][K + 1] first moment task of a bin
  unsigned* field_start;   // [n_prog][K + 1] first field block of a bin
  double* binv;            // [n_prog] 1 / b
  void* spos;              // [N] sorted particles: ScfBinRec, or ScfD4 with
  int2* skey;              // [N] (particle, bin) (masked mass in w)
  int count_status;        // flag non-finite particles (the coefficient pass)
};
// The shared memory that a handle's sort and moment kernels may take (once, before the first launch).
cudaError_t scf_bin_sort_prepare(int f32, const ScfBinShape& sh);
cudaError_t scf_moments_prepare(int f32, const ScfBinShape& sh);
cudaError_t scf_moments_dual_prepare(const ScfBinShape& sh);
cudaError_t scf_bin_sort_launch(const BinArgs& a, cudaStream_t s);

struct MomentArgs {
  const void* spos;
  const unsigned* bin_start;
  const unsigned* task_start;
  const int64_t* prog_off;
  const int* blk_prog;     // moment blocks: progenitor and task
  const int* blk_task;
  const int64_t* row_off;  // [n_prog] first moment row of a progenitor
  const void* frame;       // [K] (q_c, inv) pairs of the element type
  void* rows;              // moment rows [task][T][colpad]
  const double* binv;
  double alpha, inv_alpha;
  float alphaf, inv_alphaf;
  int K;
};
// Adjoint: the directional derivative of the moments of unit masses along weight * vbar.
struct MomentDualArgs {
  MomentArgs m;
  const int2* skey;
  AdjArgs adj;
};
cudaError_t scf_moments_dual_launch(const ScfBinShape& sh, const MomentDualArgs& a, int blocks, cudaStream_t s);
cudaError_t scf_moments_launch(int f32, const ScfBinShape& sh, const MomentArgs& a, int blocks, cudaStream_t s);

// Moment rows -> partial coefficient rows [prog][groups][2 NC] (doubles).
struct TransformArgs {
  const void* rows;
  const int64_t* row_off;
  const unsigned* task_start;
  const double* t;         // [K][lmax + 1][nmax + 1][T]
  const float2* t2;        // single precision: the same as (high, low) floats
  double* partials;
  int K, T, colpad, groups, nmax, lmax, nlm, nc, n_prog, f32;
};
cudaError_t scf_transform_launch(const TransformArgs& a, cudaStream_t s);

// Force coefficients F -> field rows P of every occupied bin.
struct FieldRowArgs {
  const void* F;           // [n_prog][NC] pairs, element type of the precision (single: times gscale)
  const void* t;           // [K][lmax + 1][nmax + 1][T], element type (single: over gscale)
  const unsigned* total;   // [n_prog][K]
  void* P;                 // [n_prog][K][row]
  int K, T, L, nmax, lmax, nlm, nc, n_prog, f32;
};
cudaError_t scf_field_rows_launch(const FieldRowArgs& a, cudaStream_t s);

// Kernel 3 over sorted particles.
struct BinFieldArgs {
  const void* spos;
  const int2* skey;
  void* vel;
  const void* vel_in;      // step mode: velocities to kick (null: vel)
  void* acc;
  const void* P;           // [n_prog][K][row]
  const void* frame;       // [K] (q_c, inv)
  const double* com;
  const double* aR;
  const float* tid;
  // blocks: progenitor, and its first field task (single precision) or first
  // and last + 1 sorted particle (double precision)
  const int* blk_prog;
  const int* blk_task;
  const int64_t* blk_begin;
  const int64_t* blk_end;
  const unsigned* bin_start;
  const unsigned* field_start;
  const int64_t* prog_off;
  const double* binv;
  int K, mode, n_prog;
  double dt, alpha, inv_alpha;
  ScfHostParams host;
  unsigned* status;
  AdjArgs adj;             // modes ADJ_J and ADJ_DUAL (double precision)
};
constexpr int kBinField64Threads = 32;
// xbar += derivative of the field along weight * vbar (and the tidal partials, one row a block).
cudaError_t scf_bin_field_dual_launch(const ScfBinShape& sh, const BinFieldArgs& a, int blocks, cudaStream_t s);
cudaError_t scf_bin_field_launch(int f32, const ScfBinShape& sh, const BinFieldArgs& a, int blocks, cudaStream_t s);

// Interpolation polynomials of the family in `tab` (alpha): frame and t tables.
struct BinTableArgs {
  int K, T, nmax, lmax, f32;
  double alpha;
  const double* vinv;      // device [2][(T-1)][(T-1)]: hi and lo parts of the node-to-monomial matrix
  const double* nodes;     // device [2][T-1]: hi and lo parts of the Chebyshev nodes
  const double* scale;     // device [nmax + 1][T] (hi, lo): 1 / n! at d = 0, 1 / ((n - 1)! d) (16-byte aligned)
  const double* inv_gscale;  // device [lmax + 1][nmax + 1]
  void* frame;             // [K] pairs of the element type
  double* t;               // [K][lmax + 1][nmax + 1][T]
  float* tf;               // single precision: t / gscale
  float2* t2;              // single precision: t as (high, low) floats
};
cudaError_t scf_bin_table_launch(const BinTableArgs& a, cudaStream_t s);
// Host side of it: nodes and node-to-monomial matrix, hi and lo parts; scale.
void scf_bin_nodes(int T, double* nodes, double* vinv);
void scf_bin_scale(int T, int nmax, double* scale);

cudaError_t scf_upload_const_bins(const ScfBinConst* t);
cudaError_t scf_upload_const_bin_moments(const ScfBinConst* t);
cudaError_t scf_upload_const_bin_field(const ScfBinConst* t);
cudaError_t scf_upload_const_bin_adjoint(const ScfBinConst* t);
