// Tidal part of the adjoint shared by its field kernels (scf_adjoint.cu, scf_bins_adjoint.cu).
#pragma once

#include "scf_device.cuh"
#include "scf_internal.h"

// Particle at R + p with direction d: g += T(R + p) d, and its terms of the
// block partials (SCF_ADJ_Q).
__device__ __forceinline__ void scf_adj_tide(const ScfHostParams& host, double Px, double Py, double Pz, double dx,
                                             double dy, double dz, double& gx, double& gy, double& gz, double* acc) {
  Dual hx, hy, hz;
  scf_host_accel_t<Dual>(host, Dual(Px, dx), Dual(Py, dy), Dual(Pz, dz), hx, hy, hz);
  gx += hx.d;
  gy += hy.d;
  gz += hz.d;
  acc[0] += dx;
  acc[1] += dy;
  acc[2] += dz;
  acc[3] += hx.d;
  acc[4] += hy.d;
  acc[5] += hz.d;
#pragma unroll
  for (int c = 0; c < SCF_HOST_CAP; ++c) {
    if (c >= host.n) break;
    double ux, uy, uz;  // a_c / GM_c
    scf_host_comp_accel<double>(host.kind[c], 1.0, host.a[c], host.b[c], Px, Py, Pz, ux, uy, uz);
    Dual sx, sy, sz;    // derivative in the scale length a_c
    scf_host_comp_accel<Dual>(host.kind[c], Dual(host.GM[c]), Dual(host.a[c], 1.0), Dual(host.b[c]), Dual(Px), Dual(Py),
                              Dual(Pz), sx, sy, sz);
    acc[6 + 2 * c] += dx * ux + dy * uy + dz * uz;
    acc[7 + 2 * c] += dx * sx.d + dy * sy.d + dz * sz.d;
  }
}
