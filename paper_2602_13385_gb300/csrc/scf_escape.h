// Internal interface of the escape-physics kernels (scf_escape.cu): the
// boundedness test, the energy-based Lagrange radius with its coefficient-set
// mask, and the tidal scales at the cluster centre (Sec. 2.2).  Not part of
// the public ABI.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "scf_device.cuh"

// Most pair-sum slots (doubles per particle) of the workspace, and of ordered pairs.
constexpr int kBoundMaxSlots = 64;
constexpr int kBoundMaxSegments = 16;

// How a handle's pair sums run.
struct BoundPlan {
  bool ordered = true;         // every ordered pair; else rounds of chunks
  int slots = 1;               // of BoundArgs::part
  int groups = 1, rounds = 1;  // of a launch over rounds, of a block: groups (1 + rounds) slots
  int64_t chunks = 0, max_chunks = 0;  // of all progenitors, of the largest
};

struct BoundArgs {
  const void* pos;             // [N][4] float (mixed) or double
  const void* vel;             // [N][4]
  const int64_t* prog_off;     // [n_prog + 1] particle offsets
  int n_prog;
  int64_t n_total, max_n;      // particles of all progenitors, of the largest
  int n_sm;
  int f32;                     // particle arrays are float4
  int slots;                   // slots of part
  int round0, rounds;          // of a pair launch (set by scf_bound_launch)
  double G, kin, frac;
  double* part;                // [slots][N] partial sums of m_j / r_ij
  unsigned long long* key;     // [N] bits of r^2
  double* E_out;               // [N] energies, or null
  uint8_t* bound;              // [N] 1 = bound
  uint8_t* mask;               // [N] 1 = r <= r_x, or null
  double* stats;               // [n_prog][4] = (n_bound, M_bound, r_x, n_in_set)
};

struct TidalArgs {
  const double* com;           // [n_prog][6] centre (R, V), or null (R = 0)
  const double* M_c;           // cluster masses with stride M_stride, or null (r_t = 0)
  int M_stride;
  int n_prog;
  double G, eta;
  ScfHostParams host;
  double* out;                 // [n_prog][16]
};

// With one slot every sample can run ordered pairs (ordered = true, slots = 1).
BoundPlan scf_bound_plan(const int64_t* offsets, int n_prog, int f32, int n_sm);
cudaError_t scf_bound_launch(const BoundArgs& a, const BoundPlan& pl, cudaStream_t s);
cudaError_t scf_tidal_launch(const TidalArgs& a, cudaStream_t s);
// The selection alone (bound flags and radius keys from a previous
// scf_bound_launch; mask may be null).
cudaError_t scf_select_launch(const BoundArgs& a, cudaStream_t s);
// b_prog[p] = r_x / scf_half_mass_divisor(alpha) from the stats of a selection at
// frac = 0.5: r_x / (1 + sqrt 2) at alpha = 1, r_x (2^(1/(alpha+1)) - 1)^alpha otherwise.
double scf_half_mass_divisor(double alpha);
cudaError_t scf_retune_b_launch(const double* stats, double* b_prog, int n_prog, double alpha, cudaStream_t s);
