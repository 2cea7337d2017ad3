// tape_common.cuh -- addressing shared by the tape kernels: the cells of the
// recorded faces and the detector seeding of the reverse step.
#pragma once

#include "fdtd_internal.cuh"

namespace fdtd {

// Cell at (u, v) of the plane normal to `axis` at `index`; (u, v) are the
// two other axes in increasing order.
__device__ __forceinline__ long long cell_on_plane(const Geo& g, int axis, int index, int u,
                                                   int v) {
  const int x = axis == 0 ? index : u;
  const int y = axis == 1 ? index : (axis == 0 ? u : v);
  const int z = axis == 2 ? index : v;
  return (long long)z * g.plane + (long long)y * g.px + x;
}

// Value r of face fd ([comp][v][u]): its field component and cell.
__device__ __forceinline__ long long face_value_cell(const Geo& g, const FaceDesc& fd, int r,
                                                    int* comp) {
  const int row = r / fd.nu, u = r - row * fd.nu;
  const int t = row >= fd.nv, v = row - t * fd.nv;
  *comp = t ? fd.comp1 : fd.comp0;
  return cell_on_plane(g, fd.axis, fd.layer, g.P + u, g.P + v);
}

// An objective seed: *l += s v, rounded once.
__device__ __forceinline__ void add_seed(float* l, float s, float v) { *l = __fmaf_rn(s, v, *l); }

// The seeds of detector d at its cell q.
__device__ __forceinline__ void seed_cell(const float* __restrict__ F, float* __restrict__ L,
                                          const Geo& g, const Det& d, float s, long long q) {
  if (d.kind == 1) {
    for (int c = 0; c < 3; ++c) add_seed(&L[c * g.nc + q], s, 2.0f * F[c * g.nc + q]);
  } else {
    const int bb = (d.axis + 1) % 3, c = (d.axis + 2) % 3;
    const float Eb = F[bb * g.nc + q], Ec = F[c * g.nc + q];
    const float Hb = F[(3 + bb) * g.nc + q], Hc = F[(3 + c) * g.nc + q];
    add_seed(&L[bb * g.nc + q], s, Hc);
    add_seed(&L[c * g.nc + q], -s, Hb);
    add_seed(&L[(3 + c) * g.nc + q], s, Eb);
    add_seed(&L[(3 + bb) * g.nc + q], -s, Ec);
  }
}

// Detector blocks of the restore launch: block b (of det_blocks per
// detector) adds the objective seeds on the detector planes: seeds[0] *
// dl_n/d(E^{n+1}, Ht^{n+1/2}) for the detector, seeds[1] * dm_n/d(...) for the
// second one (E2_PLANE: 2 s E; POYNTING_PLANE: the cross-product terms).
__device__ __forceinline__ void seed_detectors(float* __restrict__ F, float* __restrict__ L,
                                               const Geo& g, const Det& det, const Det& det2,
                                               const double* __restrict__ seeds, int b,
                                               int det_blocks) {
  const int which = b >= det_blocks;
  const Det& d = which ? det2 : det;
  if (!d.kind) return;
  const int du = d.u1 - d.u0, dv = d.v1 - d.v0;
  const int r = (b - which * det_blocks) * blockDim.x + threadIdx.x;
  if (r >= du * dv) return;
  const int v = r / du, e = r - v * du;
  int x, y, z;
  const int u = d.u0 + e, w = d.v0 + v;
  x = d.axis == 0 ? d.index : u;
  y = d.axis == 1 ? d.index : (d.axis == 0 ? u : w);
  z = d.axis == 2 ? d.index : w;
  const long long q = (long long)z * g.plane + (long long)y * g.px + x;
  // a cell on both planes belongs to the first detector's thread, which adds
  // both seeds
  int uu, vv;
  const Det& o = which ? det : det2;
  const bool both =
      o.kind && on_plane(o.axis, o.index, o.u0, o.u1, o.v0, o.v1, x, y, z, &uu, &vv);
  if (which && both) return;
  seed_cell(F, L, g, d, (float)seeds[which], q);
  if (both) seed_cell(F, L, g, det2, (float)seeds[1], q);
}

}  // namespace fdtd
