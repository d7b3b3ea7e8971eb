// Fixed-point Taylor launches of FP64 orbitals (k_fixed.cu): argument block and host entry points.
#pragma once

#include <cuda_runtime.h>

namespace tdks {

struct FxArgs {
  const double2* psi_in;    // [norb_tot][npts]
  double2* psi_out;         // may alias psi_in
  double2* backup;          // nullable: copy of the input orbitals
  const double* V64;        // potential of the step, [npts] or [ncell][npts]
  int2* V;                  // its digits (written by the preparing launch)
  long long vstride;        // offset of a cell's potential (0: one for all)
  int nx, ny, nz, npts, pstride;
  int ncta, zl, zlen, nseg; // CTAs per orbital, planes per CTA, planes per column segment, segments
  int norb, nk, ncell;
  const double *kpts, *kw;
  double Ap[3], Ap_obs[3];
  const double *Ap_cell, *Ap_obs_cell;   // nullable: [ncell][3]
  double dt, dV;
  int w2[4], w1[4];         // integer weights at distance 1..4: 5040 D2 and 840 D1
  int2 lap[3];              // digits of -dt 2^15 / (2 * 5040 h^2)
  double der_fac[3];        // dt 2^11 / (840 h)
  double obs_fac[3];        // 2^11 / (840 h)
  double diag;              // centre weight of -1/2 D2, all axes
  double lap_bound;         // |dt| sum 3.251 / h^2
  // projectors: digit tables of the sphere entries
  int natom, nsph;
  const int* sph_sidx;      // [nsph] index in the whole padded orbital
  const double* sph_d;      // [nsph][3]
  const int4* beta;         // [nsph][2]: digits of beta_p 2^Kb, p = 0..3
  const int2* sph_dfx;      // [nsph][3]: digits of the displacement, 2^Kd
  const int2* ent_rng;      // [ncta][natom] entries in a CTA's planes
  const int2* sp_rng;       // [ncta] unique sphere points in a CTA's planes
  const int *sp_pt, *sp_off, *pt_ent, *ent_atom;
  const double* ecfac;      // [natom][4]: E_p dV 2^(sN + 4 - Kb)
  const double* jfac;       // [natom][4]: 2 E_p dV^2 2^(2 (sN + 4 - Kb) + 57 - Kd)
  int sN, Kb;
  int4 *ph, *pho;           // [nk][nsph] phase factors (step, observables); per cell with phstride
  long long phstride;
  double* rho;              // nullable: rho += 2 w_k |u_out|^2
  int write_out;
  double* obs;              // nullable: per orbital {norm, J_loc[3], J_nl[3], 0}
  int* need;                // [norb_tot] 1: out of the fixed-point range, nothing written
  int* vbad;                // [ncell] 1: a potential value beyond the digits (cleared by the FP64 kernel launched after)
};

// How a grid is split for `norb_tot` orbitals; false: one CTA of a cluster of 8 cannot hold its slab.
bool fx_split(int nx, int ny, int nz, int pstride, int natom, int norb_tot, int* ncta, int* zl, int* zlen, int* nseg);
cudaError_t launch_cell_fx(const FxArgs& a, bool periodic, bool obs_at_start, cudaStream_t s);

}  // namespace tdks
