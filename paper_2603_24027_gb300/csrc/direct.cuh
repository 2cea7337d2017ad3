// direct.cuh -- arguments of the direct half-steps (kernels_direct.cu).
#pragma once

#include "bdct.cuh"
#include "fdtd_internal.cuh"

namespace fdtd {

// Direct half-steps of small grids (kernels_direct.cu): one pair of x cells per
// thread, plain loads; tape values, objective seeds and both detectors' sums
// ride in the launches.
struct DirectBox {
  int lo[3], hi[3];    // cells [lo, hi)
};
struct DirectArgs {
  Geo g;
  float* F;            // fields, updated in place
  float* L;            // adjoint fields, updated in place
  const float* cb;
  float* psiA;         // auxiliaries read (the forward updates them in place)
  float* psiB;         // adjoint auxiliaries written
  PsiLayout pl;
  double* gacc;
  int dlo[3], dhi[3];
  Src src;
  Det det, det2;
  double* obj;         // this step's slots of the two objectives
  double* obj2;
  float jn;
  int xq;              // exact reversal (0 = off), 2^xq, 2^-xq
  float xs, xi;
  int seeded;          // reverse: add the objective seeds (E phase: lam_H of this step; H
                       // phase: lam_E of the next reverse step), seeds[0..1] in device memory
  const double* seeds;
  int tmode;           // 1: record (forward) or restore (reverse) the phase's faces
  int tdtype;          // tape element type
  Faces fc;
  BdctLayout bl;       // block codec: its sample layout and basis table (device)
  const float* beta;
  void* tape;          // forward: the sample; reverse: the tape
  long long stride;    // elements of a sample
  float* scale_slot;   // forward: the sample's scales
  const float* scales;
  Interp ip;
  unsigned* err;
  int dep;             // launch as a programmatic dependent (0: sampled timing, which needs
                       // each launch's own time)
  // set by launch_direct
  DirectBox sbox, dbox, dbox2;   // source and detector planes
  int trows, drows;              // grid rows of tape blocks, of detector blocks (forward E)
  int dpairs, dpairs2;           // pairs that meet the detector planes
  unsigned mrow, mint;           // reciprocals of the pairs in a row, in an interior row
};
bool direct_fits(const Geo& g);
cudaError_t launch_direct(int which, const DirectArgs& a, cudaStream_t s);

}  // namespace fdtd
