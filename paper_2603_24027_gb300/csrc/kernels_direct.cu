// kernels_direct.cu -- half-steps of grids whose state stays in the L2 cache.
//
// The staged kernels (kernels_lag2.cu) march a CTA over a chunk of z planes,
// one plane per shared-memory stage: on a small grid that is a serial chain
// of plane latencies on a handful of CTAs (48^3: 72 CTAs of nine planes each).
// Here every pair of x cells is one thread that loads all it needs straight
// from global memory, in one round: the field neighbours, the CPML
// auxiliaries and profiles, cb and the adjoint are independent loads, so a
// launch costs about one L2 latency however many planes the grid has, and
// every SM gets work.  What bounds a launch is that latency plus the launch
// itself, so the number of launches on the chain counts:
//   * a forward step is two launches (H, E), a reverse step two (E phase, H
//     phase); the tape's unscaled record, its restore, the objective seeds and
//     the second detector's sum ride in them as extra blocks or as extra work
//     of the cells concerned (below);
//   * in the reverse phases the primal and the adjoint updates are separate
//     blocks of one launch (twice the threads, half the registers).
//
// The forward's H half-step runs its planes up and its E half-step down, so
// that each starts on the planes the other has just left in L2: on grids whose
// state does not fit, part of every half-step still reads from L2 (us per step, both
// up -> up and down: 60.3 -> 55.4 on 200 x 200 x 100, 76.5 -> 70.8 on 233 x 181 x 117,
// 8.92 -> 8.84 on 100 x 100 x 50).  The reverse phases gain too little (118 -> 116 on
// 200 x 200 x 100, where the staged ones take 104) and lose as much on small grids.
//
// Measured (GB300, us per forward / reverse step, split staged -> direct; the
// CUDA graph's launches included): 48^3 with the FP32 tape of every step 26.7 /
// 30.6 -> 4.9 / 6.7; 100 x 100 x 50 26.3 / 37.2 -> 8.8 / 14.9; 150 x 110 x 70 with
// two detectors 30.6 / 39.0 -> 14.5 / 27.2, where it moves 93 (forward) and 188
// (reverse) bytes per cell and step through L2, at 7 to 8 TB/s.
//
// Tape values in the half-steps: E^n of the high faces is recorded beside the
// H half-step (which leaves E alone) and Ht^{n+1/2} of the low faces beside
// the E half-step.  In reverse, E^n of the high faces is restored beside the
// E phase of step n (nothing reads those cells before its H phase), and
// Ht^{n-1/2} of the low faces beside the H phase of step n, for step n - 1.
// The objective seeds of step n - 1: lam_E gets its part where the H phase of
// step n stores the cell, lam_H where the E phase of step n - 1 loads it (no
// other cell reads lam_H before that).  A seed needs the primal fields of its
// own cell, which the primal blocks of the same launch may already have
// replaced; so on a pair of cells with a detector cell the adjoint thread runs
// the primal update itself, before it uses the values, and the primal blocks
// leave that pair out.
//
// Every cell sees the sequence of rounded operations of the staged kernels: the
// fields, the tape, the adjoint and the gradient are bit-identical to theirs.
#include "direct.cuh"
#include "lag_common.cuh"
#include "tape_common.cuh"

namespace fdtd {

using namespace lag2;

namespace direct {

// 128 threads: 2.8 CTAs per SM already at 48^3 (256: 16.5 against 13.8 us per
// forward step on 100 x 100 x 50).  Eight CTAs per SM, 64 registers: the pass is
// bound by the loads in flight, and more warps pay more than registers (94
// registers in the E half-step: 77.7 against 64.0 us per forward step on 200 x
// 200 x 100; ten CTAs, 48 registers: spills, 78 us).  In the reverse phases the
// auxiliaries are loaded in their branches: loaded ahead, as in the forward,
// they take 142 registers (5 % less at 48^3, 58 % more at 200 x 200 x 100).
constexpr int NT = 128;

#ifdef FDTD_BOUNDS_CHECK
__device__ __forceinline__ bool store_ok(const DirectArgs& a, const float* p) {
  const long long n6 = 6 * a.g.nc;
  if (in_buf(p, a.F, n6) || in_buf(p, a.L, n6) || in_buf(p, a.psiA, a.pl.total) ||
      in_buf(p, a.psiB, a.pl.total))
    return true;
  atomicOr(a.err, ERR_BOUNDS);
  return false;
}
#endif

template <bool EX>
__device__ __forceinline__ float inc(float d, const DirectArgs& a) {
  return EX ? grid_inc(d, 1, a.xs, a.xi) : d;
}

// Loads at an unsigned 32-bit byte offset from a base that is the same for the
// whole launch: the base stays in a uniform register, and an access costs one
// 32-bit addition instead of a 64-bit one (the path takes grids whose component
// arrays are far below 4 GB).
__device__ __forceinline__ float2 at2(const float* base, unsigned o) {
  return *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(base) + o);
}
__device__ __forceinline__ float at1(const float* base, unsigned o) {
  return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + o);
}
// Store a pair there; cell 0 is written where f0, cell 1 where f1.
__device__ __forceinline__ void put2(const DirectArgs& a, float* base, unsigned o, float u, float v,
                                     bool f0, bool f1) {
  float* p = reinterpret_cast<float*>(reinterpret_cast<char*>(base) + o);
#ifdef FDTD_BOUNDS_CHECK
  f0 = f0 && store_ok(a, p);
  f1 = f1 && store_ok(a, p + 1);
#endif
  if (f0 && f1) {
    *reinterpret_cast<float2*>(p) = make_float2(u, v);
  } else {
    if (f0) p[0] = u;
    if (f1) p[1] = v;
  }
}

// Byte offset of cell (x, y, z) within one component of axis AX's auxiliary
// array, and that component's base.
template <int AX>
__device__ __forceinline__ unsigned psi_off(const PsiLayout& L, int x, int y, int z) {
  const PsiAxis& A = L.ax[AX];
  const int xx = AX == 0 ? psi_map(A, x) : x;
  const int yy = AX == 1 ? psi_map(A, y) : y;
  const int zz = AX == 2 ? psi_map(A, z) : z;
  return 4u * ((unsigned)(zz * A.d1 + yy) * (unsigned)A.d0 + (unsigned)xx);
}
template <int AX, class T>
__device__ __forceinline__ T* psi_base(const PsiLayout& L, T* set, int c) {
  return set + L.ax[AX].off + c * L.ax[AX].cs;
}

// Programmatic dependent launch: the next half-step's CTAs may start once every
// CTA of this one has triggered or left, and then wait until this launch has
// completed with all its writes, so that the launch latency overlaps.  Triggered
// after the loads in the forward and before the stores in the reverse (us per
// forward / reverse step, plain launches -> these: 48^3 5.2 / 6.8 -> 4.9 / 6.7, 100 x
// 100 x 50 10.0 / 15.6 -> 8.9 / 14.8, 150 x 110 x 70 16.1 / 27.7 -> 14.5 / 27.2; a
// trigger at the start costs 48^3 8.2 in the reverse: the waiting CTAs take the
// running ones' place).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ float2 zero2() { return make_float2(0.f, 0.f); }

// b, a, 1/kappa of one position (side PR_BE or PR_BH).
struct Co {
  float b, a, k;
};
__device__ __forceinline__ Co coef(const Geo& g, int ax, int side, int pos) {
  return Co{prof(g, ax, side, pos), prof(g, ax, side + 1, pos), prof(g, ax, side + 2, pos)};
}

// Source and detector planes as boxes of cells (empty without one).
__device__ __forceinline__ bool in_box(const DirectBox& b, int x, int y, int z) {
  return z >= b.lo[2] && z < b.hi[2] && y >= b.lo[1] && y < b.hi[1] && x >= b.lo[0] && x < b.hi[0];
}
// Does the pair (x, x + 1) meet the box?
__device__ __forceinline__ bool pair_in_box(const DirectBox& b, int x, int y, int z) {
  return z >= b.lo[2] && z < b.hi[2] && y >= b.lo[1] && y < b.hi[1] && x + 1 >= b.lo[0] &&
         x < b.hi[0];
}
__device__ __forceinline__ bool pair_on_det(const DirectArgs& a, int x, int y, int z) {
  return pair_in_box(a.dbox, x, y, z) || pair_in_box(a.dbox2, x, y, z);
}

// Source term w J of cell (x, y, z) of the source's box.
__device__ __forceinline__ float src_term(const DirectArgs& a, int x, int y, int z) {
  return __fmul_rn(src_wt(a.src, x, y, z), a.jn);
}
__device__ __forceinline__ void add_source(const DirectArgs& a, int x, int y, int z, float& c0,
                                           float& c1, float& c2) {
  const float wj = src_term(a, x, y, z);
  if (a.src.comp == 0) c0 = __fsub_rn(c0, wj);
  else if (a.src.comp == 1) c1 = __fsub_rn(c1, wj);
  else c2 = __fsub_rn(c2, wj);
}

// i / h for i h < 2^32, with m = ceil(2^32 / h) mod 2^32 (0: h = 1).
__device__ __forceinline__ int quot(int i, unsigned m) {
  return m ? (int)__umulhi((unsigned)i, m) : i;
}

// ---------------------------------------------------------------- tape ---
// Value r of the faces of one side (side 1: the high faces, E; 0: the low
// faces, Ht), counted over those three faces; -1 past the last.
__device__ __forceinline__ int side_face(const Faces& fc, int side, int r, int* rr) {
  int f = side;
#pragma unroll
  for (int t = 0; t < 3; ++t, f += 2) {
    const int n = fc.start[f + 1] - fc.start[f];
    if (r < n) {
      *rr = r;
      return f;
    }
    r -= n;
  }
  return -1;
}

// Record (unscaled formats): one thread per value.
__device__ __forceinline__ void record_side(const DirectArgs& a, int side, int r) {
  int rr;
  const int f = side_face(a.fc, side, r, &rr);
  if (f < 0) return;
  const FaceDesc& fd = a.fc.f[f];
  if (rr == 0) a.scale_slot[f] = 1.0f;
  int comp;
  const long long q = face_value_cell(a.g, fd, rr, &comp);
  const float x = a.F[comp * a.g.nc + q];
  const long long o = fd.off + rr;
#ifdef FDTD_BOUNDS_CHECK
  if (o < 0 || o >= a.stride) {   // one sample's values
    atomicOr(a.err, ERR_BOUNDS);
    return;
  }
#endif
  switch (a.tdtype) {
    case 0: reinterpret_cast<Code<0>::T*>(a.tape)[o] = Code<0>::enc(x); break;
    case 1: reinterpret_cast<Code<1>::T*>(a.tape)[o] = Code<1>::enc(x); break;
    case 2: reinterpret_cast<Code<2>::T*>(a.tape)[o] = Code<2>::enc(x); break;
    case 3: reinterpret_cast<Code<3>::T*>(a.tape)[o] = Code<3>::enc(x); break;
    case 4: reinterpret_cast<Code<4>::T*>(a.tape)[o] = Code<4>::enc(x); break;
    case 5: reinterpret_cast<Code<5>::T*>(a.tape)[o] = Code<5>::enc(x); break;
    case 6: reinterpret_cast<Code<6>::T*>(a.tape)[o] = Code<6>::enc(x); break;
    case 7: reinterpret_cast<Code<7>::T*>(a.tape)[o] = Code<7>::enc(x); break;
    case 8: reinterpret_cast<Code<8>::T*>(a.tape)[o] = Code<8>::enc(x); break;
  }
}

template <int DT>
__device__ __forceinline__ float restored(const DirectArgs& a, int f, long long o) {
  typedef typename Code<DT>::T T;
  const T* tp = reinterpret_cast<const T*>(a.tape) + o;
  const int fld = f & 1;
  float val = 0.f;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int s = a.ip.slot[fld][m];
    if (s >= 0) {
      float x = Code<DT>::dec(tp[(long long)s * a.stride]);
      if (DT >= 2) x = __fmul_rn(x, __ldg(a.scales + s * 6 + f));
      val = __fmaf_rn(a.ip.w[fld][m], x, val);
    }
  }
  return val;
}

// Restore the faces of one side: one thread per value.
__device__ __forceinline__ void restore_side(const DirectArgs& a, int side, int r) {
  int rr;
  const int f = side_face(a.fc, side, r, &rr);
  if (f < 0) return;
  const FaceDesc& fd = a.fc.f[f];
  const long long o = fd.off + rr;
  float val = 0.f;
  switch (a.tdtype) {
    case 0: val = restored<0>(a, f, o); break;
    case 1: val = restored<1>(a, f, o); break;
    case 2: val = restored<2>(a, f, o); break;
    case 3: val = restored<3>(a, f, o); break;
    case 4: val = restored<4>(a, f, o); break;
    case 5: val = restored<5>(a, f, o); break;
    case 6: val = restored<6>(a, f, o); break;
    case 7: val = restored<7>(a, f, o); break;
    case 8: val = restored<8>(a, f, o); break;
    case kTapeBdct:
      val = bdct_restored(a.bl, fd, f, rr, reinterpret_cast<const unsigned char*>(a.tape), a.stride,
                          a.ip, a.beta);
      break;
  }
  int comp;
  const long long q = face_value_cell(a.g, fd, rr, &comp);
#ifdef FDTD_BOUNDS_CHECK
  if (!store_ok(a, a.F + comp * a.g.nc + q)) return;
#endif
  a.F[comp * a.g.nc + q] = val;
}

// The pair of cells of thread i of plane z: pairs of a plane are consecutive
// in memory (rows padded to an even pitch), so a warp's accesses are too.
struct Pair {
  int x, y, z;
  unsigned q;      // byte offset of the pair in a component array
  bool v0, v1;
};
__device__ __forceinline__ Pair pair_of(const DirectArgs& a, int z) {
  Pair p;
  p.z = z;
  const int i = (int)blockIdx.x * NT + (int)threadIdx.x;
  const int h = a.g.px >> 1;
  p.y = quot(i, a.mrow);
  p.x = 2 * (i - p.y * h);
  p.q = 4u * (unsigned)a.g.plane * (unsigned)z + 8u * (unsigned)i;
  p.v0 = p.y < a.g.ny && p.x < a.g.nx;
  p.v1 = p.v0 && p.x + 1 < a.g.nx;
  return p;
}
// Tape blocks come first: the value this thread handles.
__device__ __forceinline__ int tape_value() {
  return ((int)blockIdx.y * (int)gridDim.x + (int)blockIdx.x) * NT + (int)threadIdx.x;
}

// ============================================================ forward H ===
template <bool EX>
__global__ void __launch_bounds__(NT, 8) k_dir_fwd_h(const __grid_constant__ DirectArgs a) {
  pdl_wait();
  if ((int)blockIdx.y < a.trows) {   // E^n of the high faces
    record_side(a, 1, tape_value());
    return;
  }
  const Geo& g = a.g;
  const Pair p = pair_of(a, (int)blockIdx.y - a.trows);
  if (!p.v0) return;
  const int x = p.x, y = p.y, z = p.z;
  const unsigned q = p.q, rp = 4u * (unsigned)g.px, pl = 4u * (unsigned)g.plane;
  const long long nc = g.nc;
  const bool sx0 = in_slab(x, g.nx, g.P), sx1 = p.v1 && in_slab(x + 1, g.nx, g.P);
  const bool sx = sx0 || sx1, sy = in_slab(y, g.ny, g.P), sz = in_slab(z, g.nz, g.P);
  const bool yn = y + 1 < g.ny, zn = z + 1 < g.nz, xn = x + 2 < g.nx;
  const float* E = a.F;
  float* H = a.F + 3 * nc;
  float* psi = a.psiA;
  // every load of the pair, independent of each other
  const float2 ex = at2(E, q), ey = at2(E + nc, q), ez = at2(E + 2 * nc, q);
  const float2 ezy = yn ? at2(E + 2 * nc, q + rp) : zero2(), exy = yn ? at2(E, q + rp) : zero2();
  const float2 exz = zn ? at2(E, q + pl) : zero2(), eyz = zn ? at2(E + nc, q + pl) : zero2();
  const float ezx = xn ? at1(E + 2 * nc, q + 8) : 0.f, eyx = xn ? at1(E + nc, q + 8) : 0.f;
  const float2 h0 = at2(H, q), h1 = at2(H + nc, q), h2 = at2(H + 2 * nc, q);
  unsigned ix = 0, iy = 0, iz = 0;
  float2 px0 = zero2(), px1 = zero2(), py0 = zero2(), py1 = zero2(), pz0 = zero2(), pz1 = zero2();
  Co cx0 = {}, cx1 = {}, cy = {}, cz = {};
  if (sx) {
    ix = psi_off<0>(a.pl, x, y, z);
    px0 = at2(psi_base<0>(a.pl, psi, 0), ix);
    px1 = at2(psi_base<0>(a.pl, psi, 1), ix);
    if (sx0) cx0 = coef(g, 0, PR_BH, x);
    if (sx1) cx1 = coef(g, 0, PR_BH, x + 1);
  }
  if (sy) {
    iy = psi_off<1>(a.pl, x, y, z);
    py0 = at2(psi_base<1>(a.pl, psi, 0), iy);
    py1 = at2(psi_base<1>(a.pl, psi, 1), iy);
    cy = coef(g, 1, PR_BH, y);
  }
  if (sz) {
    iz = psi_off<2>(a.pl, x, y, z);
    pz0 = at2(psi_base<2>(a.pl, psi, 0), iz);
    pz1 = at2(psi_base<2>(a.pl, psi, 1), iz);
    cz = coef(g, 2, PR_BH, z);
  }
  pdl_trigger();
  float t0[2] = {ezy.x - ez.x, ezy.y - ez.y};   // dEz/dy
  float t1[2] = {eyz.x - ey.x, eyz.y - ey.y};   // dEy/dz
  float t2[2] = {exz.x - ex.x, exz.y - ex.y};   // dEx/dz
  float t3[2] = {ez.y - ez.x, ezx - ez.y};      // dEz/dx
  float t4[2] = {ey.y - ey.x, eyx - ey.y};      // dEy/dx
  float t5[2] = {exy.x - ex.x, exy.y - ex.y};   // dEx/dy
  if (sx) {
    float s3[2] = {0.f, 0.f}, s4[2] = {0.f, 0.f};
    if (sx0) {
      t3[0] = cpml(t3[0], px0.x, cx0.b, cx0.a, cx0.k, &s3[0]);
      t4[0] = cpml(t4[0], px1.x, cx0.b, cx0.a, cx0.k, &s4[0]);
    }
    if (sx1) {
      t3[1] = cpml(t3[1], px0.y, cx1.b, cx1.a, cx1.k, &s3[1]);
      t4[1] = cpml(t4[1], px1.y, cx1.b, cx1.a, cx1.k, &s4[1]);
    }
    put2(a, psi_base<0>(a.pl, psi, 0), ix, s3[0], s3[1], sx0, sx1);
    put2(a, psi_base<0>(a.pl, psi, 1), ix, s4[0], s4[1], sx0, sx1);
  }
  if (sy) {
    float s0[2], s5[2];
    t0[0] = cpml(t0[0], py0.x, cy.b, cy.a, cy.k, &s0[0]);
    t0[1] = cpml(t0[1], py0.y, cy.b, cy.a, cy.k, &s0[1]);
    t5[0] = cpml(t5[0], py1.x, cy.b, cy.a, cy.k, &s5[0]);
    t5[1] = cpml(t5[1], py1.y, cy.b, cy.a, cy.k, &s5[1]);
    put2(a, psi_base<1>(a.pl, psi, 0), iy, s0[0], s0[1], true, p.v1);
    put2(a, psi_base<1>(a.pl, psi, 1), iy, s5[0], s5[1], true, p.v1);
  }
  if (sz) {
    float s1[2], s2[2];
    t1[0] = cpml(t1[0], pz0.x, cz.b, cz.a, cz.k, &s1[0]);
    t1[1] = cpml(t1[1], pz0.y, cz.b, cz.a, cz.k, &s1[1]);
    t2[0] = cpml(t2[0], pz1.x, cz.b, cz.a, cz.k, &s2[0]);
    t2[1] = cpml(t2[1], pz1.y, cz.b, cz.a, cz.k, &s2[1]);
    put2(a, psi_base<2>(a.pl, psi, 0), iz, s1[0], s1[1], true, p.v1);
    put2(a, psi_base<2>(a.pl, psi, 1), iz, s2[0], s2[1], true, p.v1);
  }
  const float ho0[2] = {h0.x, h0.y}, ho1[2] = {h1.x, h1.y}, ho2[2] = {h2.x, h2.y};
  float hx[2], hy[2], hz[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const float cx = t0[c] - t1[c], cyy = t2[c] - t3[c], czz = t4[c] - t5[c];
    hx[c] = __fsub_rn(ho0[c], inc<EX>(__fmul_rn(g.S, cx), a));
    hy[c] = __fsub_rn(ho1[c], inc<EX>(__fmul_rn(g.S, cyy), a));
    hz[c] = __fsub_rn(ho2[c], inc<EX>(__fmul_rn(g.S, czz), a));
  }
  put2(a, H, q, hx[0], hx[1], true, p.v1);
  put2(a, H + nc, q, hy[0], hy[1], true, p.v1);
  put2(a, H + 2 * nc, q, hz[0], hz[1], true, p.v1);
}

// l_n of one cell.
__device__ __forceinline__ double det_value(const Det& d, const float e[3], const float h[3]) {
  if (d.kind == 1) return (double)e[0] * e[0] + (double)e[1] * e[1] + (double)e[2] * e[2];
  const int ax = d.axis;
  const float Eb = ax == 0 ? e[1] : (ax == 1 ? e[2] : e[0]);
  const float Ec = ax == 0 ? e[2] : (ax == 1 ? e[0] : e[1]);
  const float Hb = ax == 0 ? h[1] : (ax == 1 ? h[2] : h[0]);
  const float Hc = ax == 0 ? h[2] : (ax == 1 ? h[0] : h[1]);
  return (double)Eb * Hc - (double)Ec * Hb;
}

__device__ __forceinline__ void block_add(double v, double* red, double* out) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < NT / 32; ++w) t += red[w];
    if (t != 0.0) atomicAdd(out, t);
  }
}

// ============================================================ forward E ===
// E^{n+1} of a pair in en, Ht^{n+1/2} there in hh.
template <bool EX>
__device__ __forceinline__ void update_e(const DirectArgs& a, int x, int y, int z, unsigned q,
                                         bool v1, float en[2][3], float hh[2][3]) {
  const Geo& g = a.g;
  const unsigned rp = 4u * (unsigned)g.px, pl = 4u * (unsigned)g.plane;
  const long long nc = g.nc;
  const bool sx0 = in_slab(x, g.nx, g.P), sx1 = v1 && in_slab(x + 1, g.nx, g.P);
  const bool sx = sx0 || sx1, sy = in_slab(y, g.ny, g.P), sz = in_slab(z, g.nz, g.P);
  float* E = a.F;
  const float* H = a.F + 3 * nc;
  float* psi = a.psiA;
  const float2 hx = at2(H, q), hy = at2(H + nc, q), hz = at2(H + 2 * nc, q);
  const float2 hzy = y > 0 ? at2(H + 2 * nc, q - rp) : zero2();
  const float2 hxy = y > 0 ? at2(H, q - rp) : zero2();
  const float2 hxz = z > 0 ? at2(H, q - pl) : zero2(), hyz = z > 0 ? at2(H + nc, q - pl) : zero2();
  const float hzx = x > 0 ? at1(H + 2 * nc, q - 4) : 0.f, hyx = x > 0 ? at1(H + nc, q - 4) : 0.f;
  const float2 e0 = at2(E, q), e1 = at2(E + nc, q), e2 = at2(E + 2 * nc, q);
  const float2 cb2 = at2(a.cb, q);
    unsigned ix = 0, iy = 0, iz = 0;
  float2 px0 = zero2(), px1 = zero2(), py0 = zero2(), py1 = zero2(), pz0 = zero2(), pz1 = zero2();
  Co cx0 = {}, cx1 = {}, cy = {}, cz = {};
  if (sx) {
    ix = psi_off<0>(a.pl, x, y, z);
    px0 = at2(psi_base<0>(a.pl, psi, 2), ix);
    px1 = at2(psi_base<0>(a.pl, psi, 3), ix);
    if (sx0) cx0 = coef(g, 0, PR_BE, x);
    if (sx1) cx1 = coef(g, 0, PR_BE, x + 1);
  }
  if (sy) {
    iy = psi_off<1>(a.pl, x, y, z);
    py0 = at2(psi_base<1>(a.pl, psi, 2), iy);
    py1 = at2(psi_base<1>(a.pl, psi, 3), iy);
    cy = coef(g, 1, PR_BE, y);
  }
  if (sz) {
    iz = psi_off<2>(a.pl, x, y, z);
    pz0 = at2(psi_base<2>(a.pl, psi, 2), iz);
    pz1 = at2(psi_base<2>(a.pl, psi, 3), iz);
    cz = coef(g, 2, PR_BE, z);
  }
  pdl_trigger();
  float t6[2] = {hz.x - hzy.x, hz.y - hzy.y};    // dHz/dy
  float t7[2] = {hy.x - hyz.x, hy.y - hyz.y};    // dHy/dz
  float t8[2] = {hx.x - hxz.x, hx.y - hxz.y};    // dHx/dz
  float t9[2] = {hz.x - hzx, hz.y - hz.x};       // dHz/dx
  float t10[2] = {hy.x - hyx, hy.y - hy.x};      // dHy/dx
  float t11[2] = {hx.x - hxy.x, hx.y - hxy.y};   // dHx/dy
  if (sx) {
    float s9[2] = {0.f, 0.f}, s10[2] = {0.f, 0.f};
    if (sx0) {
      t9[0] = cpml(t9[0], px0.x, cx0.b, cx0.a, cx0.k, &s9[0]);
      t10[0] = cpml(t10[0], px1.x, cx0.b, cx0.a, cx0.k, &s10[0]);
    }
    if (sx1) {
      t9[1] = cpml(t9[1], px0.y, cx1.b, cx1.a, cx1.k, &s9[1]);
      t10[1] = cpml(t10[1], px1.y, cx1.b, cx1.a, cx1.k, &s10[1]);
    }
    put2(a, psi_base<0>(a.pl, psi, 2), ix, s9[0], s9[1], sx0, sx1);
    put2(a, psi_base<0>(a.pl, psi, 3), ix, s10[0], s10[1], sx0, sx1);
  }
  if (sy) {
    float s6[2], s11[2];
    t6[0] = cpml(t6[0], py0.x, cy.b, cy.a, cy.k, &s6[0]);
    t6[1] = cpml(t6[1], py0.y, cy.b, cy.a, cy.k, &s6[1]);
    t11[0] = cpml(t11[0], py1.x, cy.b, cy.a, cy.k, &s11[0]);
    t11[1] = cpml(t11[1], py1.y, cy.b, cy.a, cy.k, &s11[1]);
    put2(a, psi_base<1>(a.pl, psi, 2), iy, s6[0], s6[1], true, v1);
    put2(a, psi_base<1>(a.pl, psi, 3), iy, s11[0], s11[1], true, v1);
  }
  if (sz) {
    float s7[2], s8[2];
    t7[0] = cpml(t7[0], pz0.x, cz.b, cz.a, cz.k, &s7[0]);
    t7[1] = cpml(t7[1], pz0.y, cz.b, cz.a, cz.k, &s7[1]);
    t8[0] = cpml(t8[0], pz1.x, cz.b, cz.a, cz.k, &s8[0]);
    t8[1] = cpml(t8[1], pz1.y, cz.b, cz.a, cz.k, &s8[1]);
    put2(a, psi_base<2>(a.pl, psi, 2), iz, s7[0], s7[1], true, v1);
    put2(a, psi_base<2>(a.pl, psi, 3), iz, s8[0], s8[1], true, v1);
  }
  const float eo0[2] = {e0.x, e0.y}, eo1[2] = {e1.x, e1.y}, eo2[2] = {e2.x, e2.y};
  const float cbv[2] = {cb2.x, cb2.y};
  const bool src = pair_in_box(a.sbox, x, y, z);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    float c0 = t6[c] - t7[c], c1 = t8[c] - t9[c], c2 = t10[c] - t11[c];
    if (src && in_box(a.sbox, x + c, y, z)) add_source(a, x + c, y, z, c0, c1, c2);
    en[c][0] = __fadd_rn(eo0[c], inc<EX>(__fmul_rn(cbv[c], c0), a));
    en[c][1] = __fadd_rn(eo1[c], inc<EX>(__fmul_rn(cbv[c], c1), a));
    en[c][2] = __fadd_rn(eo2[c], inc<EX>(__fmul_rn(cbv[c], c2), a));
  }
  put2(a, E, q, en[0][0], en[1][0], true, v1);
  put2(a, E + nc, q, en[0][1], en[1][1], true, v1);
  put2(a, E + 2 * nc, q, en[0][2], en[1][2], true, v1);
  hh[0][0] = hx.x; hh[0][1] = hy.x; hh[0][2] = hz.x;
  hh[1][0] = hx.y; hh[1][1] = hy.y; hh[1][2] = hz.y;
}

// Pairs that meet a detector plane have blocks of their own, which list just
// those pairs (a plane normal to x has one cell in every row: summed where its
// rows are updated, nearly every block of the grid would pay for an FP64
// reduction and an atomic for a single cell).
template <bool EX>
__global__ void __launch_bounds__(NT, 8) k_dir_fwd_e(const __grid_constant__ DirectArgs a) {
  pdl_wait();
  const int row = (int)blockIdx.y;
  if (row < a.trows) {   // Ht^{n+1/2} of the low faces
    record_side(a, 0, tape_value());
    return;
  }
  float en[2][3], hh[2][3];
  const int zb = row - a.trows - a.drows;
  if (zb >= 0) {
    const Pair p = pair_of(a, a.g.nz - 1 - zb);   // down: see the head of this file
    if (!p.v0 || pair_on_det(a, p.x, p.y, p.z)) return;
    update_e<EX>(a, p.x, p.y, p.z, p.q, p.v1, en, hh);
    return;
  }
  __shared__ double red[2][NT / 32];
  int i = ((row - a.trows) * (int)gridDim.x + (int)blockIdx.x) * NT + (int)threadIdx.x;
  const DirectBox* b = &a.dbox;
  bool ok = i < a.dpairs;
  if (!ok) {
    i -= a.dpairs;
    b = &a.dbox2;
    ok = i < a.dpairs2;
  }
  double l1 = 0.0, l2 = 0.0;
  if (ok) {
    const int x0 = b->lo[0] >> 1, w = ((b->hi[0] + 1) >> 1) - x0, hgt = b->hi[1] - b->lo[1];
    const int r = i / w, x = 2 * (i - r * w + x0);
    const int zi = r / hgt, y = r - zi * hgt + b->lo[1], z = zi + b->lo[2];
    // a pair on both planes belongs to the first
    if (b == &a.dbox || !pair_in_box(a.dbox, x, y, z)) {
      const unsigned q =
          4u * ((unsigned)a.g.plane * (unsigned)z + (unsigned)(y * a.g.px + x));
      update_e<EX>(a, x, y, z, q, x + 1 < a.g.nx, en, hh);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (in_box(a.dbox, x + c, y, z)) l1 += det_value(a.det, en[c], hh[c]);
        if (in_box(a.dbox2, x + c, y, z)) l2 += det_value(a.det2, en[c], hh[c]);
      }
    }
  }
  block_add(l1, red[0], a.obj);
  if (a.dpairs2) block_add(l2, red[1], a.obj2);
}

// ======================================================= reverse E phase ===
// Primal inverse E update of a pair and its dL/dcb (cells w0 / w1 only).
template <bool EX>
__device__ __forceinline__ void primal_e(const DirectArgs& a, int x, int y, int z, unsigned q,
                                         bool w0, bool w1) {
  const Geo& g = a.g;
  const unsigned rp = 4u * (unsigned)g.px, pl = 4u * (unsigned)g.plane;
  const long long nc = g.nc;
  float* E = a.F;
  const float* H = a.F + 3 * nc;
  const float2 hx = at2(H, q), hy = at2(H + nc, q), hz = at2(H + 2 * nc, q);
  const float2 hzy = at2(H + 2 * nc, q - rp), hxy = at2(H, q - rp);
  const float2 hxz = at2(H, q - pl), hyz = at2(H + nc, q - pl);
  // cell 0 is left out where it has no -x neighbour (then it is not interior)
  const float hzx = x > 0 ? at1(H + 2 * nc, q - 4) : 0.f, hyx = x > 0 ? at1(H + nc, q - 4) : 0.f;
  const float2 e0 = at2(E, q), e1 = at2(E + nc, q), e2 = at2(E + 2 * nc, q);
  const float2 cb2 = at2(a.cb, q);
  const bool dyz = y >= a.dlo[1] && y < a.dhi[1] && z >= a.dlo[2] && z < a.dhi[2];
  const bool g0 = dyz && w0 && x >= a.dlo[0] && x < a.dhi[0];
  const bool g1 = dyz && w1 && x + 1 >= a.dlo[0] && x + 1 < a.dhi[0];
  float2 l0 = zero2(), l1 = zero2(), l2 = zero2();
  if (g0 || g1) {
    l0 = at2(a.L, q);
    l1 = at2(a.L + nc, q);
    l2 = at2(a.L + 2 * nc, q);
  }
  const float d6[2] = {hz.x - hzy.x, hz.y - hzy.y}, d7[2] = {hy.x - hyz.x, hy.y - hyz.y};
  const float d8[2] = {hx.x - hxz.x, hx.y - hxz.y}, d9[2] = {hz.x - hzx, hz.y - hz.x};
  const float d10[2] = {hy.x - hyx, hy.y - hy.x}, d11[2] = {hx.x - hxy.x, hx.y - hxy.y};
  const float eo0[2] = {e0.x, e0.y}, eo1[2] = {e1.x, e1.y}, eo2[2] = {e2.x, e2.y};
  const float cbv[2] = {cb2.x, cb2.y};
  const float lx[2] = {l0.x, l0.y}, ly[2] = {l1.x, l1.y}, lz[2] = {l2.x, l2.y};
  float en0[2], en1[2], en2[2];
  const bool src = pair_in_box(a.sbox, x, y, z);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    float c0 = d6[c] - d7[c], c1 = d8[c] - d9[c], c2 = d10[c] - d11[c];
    if (src && in_box(a.sbox, x + c, y, z)) add_source(a, x + c, y, z, c0, c1, c2);
    en0[c] = __fsub_rn(eo0[c], inc<EX>(__fmul_rn(cbv[c], c0), a));
    en1[c] = __fsub_rn(eo1[c], inc<EX>(__fmul_rn(cbv[c], c1), a));
    en2[c] = __fsub_rn(eo2[c], inc<EX>(__fmul_rn(cbv[c], c2), a));
    if (c == 0 ? g0 : g1) {
      const float s = grad_term(lx[c], ly[c], lz[c], c0, c1, c2);
      const int dX = a.dhi[0] - a.dlo[0], dY = a.dhi[1] - a.dlo[1];
      const long long qd =
          ((long long)(z - a.dlo[2]) * dY + (y - a.dlo[1])) * dX + (x + c - a.dlo[0]);
#ifdef FDTD_BOUNDS_CHECK
      if (qd < 0 || qd >= (long long)dX * dY * (a.dhi[2] - a.dlo[2])) {
        atomicOr(a.err, ERR_BOUNDS);
        continue;
      }
#endif
      atomicAdd(a.gacc + qd, (double)s);
    }
  }
  pdl_trigger();
  put2(a, E, q, en0[0], en0[1], w0, w1);
  put2(a, E + nc, q, en1[0], en1[1], w0, w1);
  put2(a, E + 2 * nc, q, en2[0], en2[1], w0, w1);
}

// Thread i of the primal blocks: a pair of the interior box (rows [P, ny - P)
// of the planes [P, nz - P)); w0, w1: its cells inside.
struct PrimalPair {
  int x, y, z;
  unsigned q;
  bool w0, w1;
};
__device__ __forceinline__ bool primal_cells(const Geo& g, int x, int y, int z, bool* w0, bool* w1) {
  const bool in = y >= g.P && y < g.ny - g.P && z >= g.P && z < g.nz - g.P;
  *w0 = in && x >= g.P && x < g.nx - g.P;
  *w1 = in && x + 1 >= g.P && x + 1 < g.nx - g.P;
  return *w0 || *w1;
}
__device__ __forceinline__ PrimalPair primal_pair(const DirectArgs& a, int z) {
  const Geo& g = a.g;
  PrimalPair p;
  const int i = (int)blockIdx.x * NT + (int)threadIdx.x;
  const int h0 = g.P >> 1, h = ((g.nx - g.P + 1) >> 1) - h0;   // pairs of an interior row
  const int yi = quot(i, a.mint);
  p.x = 2 * (i - yi * h + h0);
  p.y = yi + g.P;
  p.z = z;
  primal_cells(g, p.x, p.y, p.z, &p.w0, &p.w1);
  p.q = 4u * ((unsigned)g.plane * (unsigned)z + (unsigned)(p.y * g.px + p.x));
  return p;
}

// lam_H seeds of step n at a cell: e = E^{n+1} there.
__device__ __forceinline__ void seed_h(const Det& d, float s, const float e[3], float lh[3]) {
  if (d.kind != 2) return;
  const int bb = (d.axis + 1) % 3, c = (d.axis + 2) % 3;
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    if (t == c) add_seed(&lh[t], s, bb == 0 ? e[0] : (bb == 1 ? e[1] : e[2]));
    if (t == bb) add_seed(&lh[t], -s, c == 0 ? e[0] : (c == 1 ? e[1] : e[2]));
  }
}

template <bool EX>
__global__ void __launch_bounds__(NT, 8) k_dir_rev_e(const __grid_constant__ DirectArgs a) {
  pdl_wait();
  if ((int)blockIdx.y < a.trows) {   // E^n of the high faces
    restore_side(a, 1, tape_value());
    return;
  }
  const Geo& g = a.g;
  const int zb = (int)blockIdx.y - a.trows;
  if (zb >= g.nz) {   // primal blocks
    const PrimalPair p = primal_pair(a, zb - g.nz + g.P);
    if (!(p.w0 || p.w1) || (a.seeded && pair_on_det(a, p.x, p.y, p.z))) return;
    primal_e<EX>(a, p.x, p.y, p.z, p.q, p.w0, p.w1);
    return;
  }
  const Pair p = pair_of(a, zb);
  if (!p.v0) return;
  const int x = p.x, y = p.y, z = p.z;
  const unsigned q = p.q, rp = 4u * (unsigned)g.px, pl = 4u * (unsigned)g.plane;
  const long long nc = g.nc;
  const float* lE = a.L;
  float* lH = a.L + 3 * nc;
  const float* lpA = a.psiA;
  float* lpB = a.psiB;
  const float2 lh0 = at2(lH, q), lh1 = at2(lH + nc, q), lh2 = at2(lH + 2 * nc, q);
  float lh[2][3] = {{lh0.x, lh1.x, lh2.x}, {lh0.y, lh1.y, lh2.y}};
  if (a.seeded && pair_on_det(a, x, y, z)) {
    const float2 e0 = at2(a.F, q), e1 = at2(a.F + nc, q), e2 = at2(a.F + 2 * nc, q);
    const float e[2][3] = {{e0.x, e1.x, e2.x}, {e0.y, e1.y, e2.y}};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (in_box(a.dbox, x + c, y, z)) seed_h(a.det, (float)a.seeds[0], e[c], lh[c]);
      if (in_box(a.dbox2, x + c, y, z)) seed_h(a.det2, (float)a.seeds[1], e[c], lh[c]);
    }
    bool w0, w1;
    if (primal_cells(g, x, y, z, &w0, &w1)) primal_e<EX>(a, x, y, z, q, w0, w1);
  }
  const bool sx0 = in_slab(x, g.nx, g.P), sx1 = p.v1 && in_slab(x + 1, g.nx, g.P);
  const bool xn = x + 2 < g.nx, yn = y + 1 < g.ny, zn = z + 1 < g.nz;
  const bool sx2 = xn && in_slab(x + 2, g.nx, g.P), sx = sx0 || sx1;
  const bool sy = in_slab(y, g.ny, g.P), sy1 = yn && in_slab(y + 1, g.ny, g.P);
  const bool sz = in_slab(z, g.nz, g.P), sz1 = zn && in_slab(z + 1, g.nz, g.P);
  const float2 cb2 = at2(a.cb, q), cby = yn ? at2(a.cb, q + rp) : zero2();
  const float2 cbz = zn ? at2(a.cb, q + pl) : zero2();
  const float cbx = xn ? at1(a.cb, q + 8) : 0.f;
  const float2 lx = at2(lE, q), ly = at2(lE + nc, q), lz = at2(lE + 2 * nc, q);
  const float2 lxy = yn ? at2(lE, q + rp) : zero2(), lzy = yn ? at2(lE + 2 * nc, q + rp) : zero2();
  const float2 lxz = zn ? at2(lE, q + pl) : zero2(), lyz = zn ? at2(lE + nc, q + pl) : zero2();
  const float lyx = xn ? at1(lE + nc, q + 8) : 0.f, lzx = xn ? at1(lE + 2 * nc, q + 8) : 0.f;
  // own terms (t6: Ex,y,+; t7: Ex,z,-; t8: Ey,z,+; t9: Ey,x,-; t10: Ez,x,+; t11: Ez,y,-)
  // and the same terms of the +y, +z and +x neighbours
  const float cbv[2] = {cb2.x, cb2.y};
  const float lex[2] = {lx.x, lx.y}, ley[2] = {ly.x, ly.y}, lez[2] = {lz.x, lz.y};
  float o6[2], o7[2], o8[2], o9[2], o10[2], o11[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const float wx = __fmul_rn(cbv[c], lex[c]), wy = __fmul_rn(cbv[c], ley[c]), wz = __fmul_rn(cbv[c], lez[c]);
    o6[c] = wx; o11[c] = -wz; o7[c] = -wx; o8[c] = wy; o9[c] = -wy; o10[c] = wz;
  }
  float n6[2] = {0.f, 0.f}, n11[2] = {0.f, 0.f}, n7[2] = {0.f, 0.f}, n8[2] = {0.f, 0.f};
  float n9x = 0.f, n10x = 0.f;
  if (yn) {
    n6[0] = __fmul_rn(cby.x, lxy.x); n6[1] = __fmul_rn(cby.y, lxy.y);
    n11[0] = __fmul_rn(-cby.x, lzy.x); n11[1] = __fmul_rn(-cby.y, lzy.y);
  }
  if (zn) {
    n7[0] = __fmul_rn(-cbz.x, lxz.x); n7[1] = __fmul_rn(-cbz.y, lxz.y);
    n8[0] = __fmul_rn(cbz.x, lyz.x); n8[1] = __fmul_rn(cbz.y, lyz.y);
  }
  if (xn) {
    n9x = __fmul_rn(-cbx, lyx);
    n10x = __fmul_rn(cbx, lzx);
  }
  float dummy;
  if (sy || sy1) {
    if (sy) {
      const unsigned iy = psi_off<1>(a.pl, x, y, z);
      const Co ky = coef(g, 1, PR_BE, y);
      const float2 py0 = at2(psi_base<1>(a.pl, lpA, 2), iy), py1 = at2(psi_base<1>(a.pl, lpA, 3), iy);
      float s6[2], s11[2];
      o6[0] = adj(o6[0], py0.x, ky.b, ky.a, ky.k, &s6[0]);
      o6[1] = adj(o6[1], py0.y, ky.b, ky.a, ky.k, &s6[1]);
      o11[0] = adj(o11[0], py1.x, ky.b, ky.a, ky.k, &s11[0]);
      o11[1] = adj(o11[1], py1.y, ky.b, ky.a, ky.k, &s11[1]);
      put2(a, psi_base<1>(a.pl, lpB, 2), iy, s6[0], s6[1], true, p.v1);
      put2(a, psi_base<1>(a.pl, lpB, 3), iy, s11[0], s11[1], true, p.v1);
    }
    if (sy1) {
      const unsigned iy = psi_off<1>(a.pl, x, y + 1, z);
      const Co kyn = coef(g, 1, PR_BE, y + 1);
      const float2 qy0 = at2(psi_base<1>(a.pl, lpA, 2), iy), qy1 = at2(psi_base<1>(a.pl, lpA, 3), iy);
      n6[0] = adj(n6[0], qy0.x, kyn.b, kyn.a, kyn.k, &dummy);
      n6[1] = adj(n6[1], qy0.y, kyn.b, kyn.a, kyn.k, &dummy);
      n11[0] = adj(n11[0], qy1.x, kyn.b, kyn.a, kyn.k, &dummy);
      n11[1] = adj(n11[1], qy1.y, kyn.b, kyn.a, kyn.k, &dummy);
    }
  }
  if (sz || sz1) {
    if (sz) {
      const unsigned iz = psi_off<2>(a.pl, x, y, z);
      const Co kz = coef(g, 2, PR_BE, z);
      const float2 pz0 = at2(psi_base<2>(a.pl, lpA, 2), iz), pz1 = at2(psi_base<2>(a.pl, lpA, 3), iz);
      float s7[2], s8[2];
      o7[0] = adj(o7[0], pz0.x, kz.b, kz.a, kz.k, &s7[0]);
      o7[1] = adj(o7[1], pz0.y, kz.b, kz.a, kz.k, &s7[1]);
      o8[0] = adj(o8[0], pz1.x, kz.b, kz.a, kz.k, &s8[0]);
      o8[1] = adj(o8[1], pz1.y, kz.b, kz.a, kz.k, &s8[1]);
      put2(a, psi_base<2>(a.pl, lpB, 2), iz, s7[0], s7[1], true, p.v1);
      put2(a, psi_base<2>(a.pl, lpB, 3), iz, s8[0], s8[1], true, p.v1);
    }
    if (sz1) {
      const unsigned iz = psi_off<2>(a.pl, x, y, z + 1);
      const Co kzn = coef(g, 2, PR_BE, z + 1);
      const float2 qz0 = at2(psi_base<2>(a.pl, lpA, 2), iz), qz1 = at2(psi_base<2>(a.pl, lpA, 3), iz);
      n7[0] = adj(n7[0], qz0.x, kzn.b, kzn.a, kzn.k, &dummy);
      n7[1] = adj(n7[1], qz0.y, kzn.b, kzn.a, kzn.k, &dummy);
      n8[0] = adj(n8[0], qz1.x, kzn.b, kzn.a, kzn.k, &dummy);
      n8[1] = adj(n8[1], qz1.y, kzn.b, kzn.a, kzn.k, &dummy);
    }
  }
  if (sx || sx2) {
    if (sx) {
      const unsigned ix = psi_off<0>(a.pl, x, y, z);
      const float2 px0 = at2(psi_base<0>(a.pl, lpA, 2), ix), px1 = at2(psi_base<0>(a.pl, lpA, 3), ix);
      float s9[2] = {0.f, 0.f}, s10[2] = {0.f, 0.f};
      if (sx0) {
        const Co kx0 = coef(g, 0, PR_BE, x);
        o9[0] = adj(o9[0], px0.x, kx0.b, kx0.a, kx0.k, &s9[0]);
        o10[0] = adj(o10[0], px1.x, kx0.b, kx0.a, kx0.k, &s10[0]);
      }
      if (sx1) {
        const Co kx1 = coef(g, 0, PR_BE, x + 1);
        o9[1] = adj(o9[1], px0.y, kx1.b, kx1.a, kx1.k, &s9[1]);
        o10[1] = adj(o10[1], px1.y, kx1.b, kx1.a, kx1.k, &s10[1]);
      }
      put2(a, psi_base<0>(a.pl, lpB, 2), ix, s9[0], s9[1], sx0, sx1);
      put2(a, psi_base<0>(a.pl, lpB, 3), ix, s10[0], s10[1], sx0, sx1);
    }
    if (sx2) {
      const unsigned ix = psi_off<0>(a.pl, x + 2, y, z);
      const Co kxn = coef(g, 0, PR_BE, x + 2);
      const float qx0 = at1(psi_base<0>(a.pl, lpA, 2), ix), qx1 = at1(psi_base<0>(a.pl, lpA, 3), ix);
      n9x = adj(n9x, qx0, kxn.b, kxn.a, kxn.k, &dummy);
      n10x = adj(n10x, qx1, kxn.b, kxn.a, kxn.k, &dummy);
    }
  }
  // cell 0's +x terms are cell 1's own terms
  const float n9[2] = {p.v1 ? o9[1] : 0.f, n9x}, n10[2] = {p.v1 ? o10[1] : 0.f, n10x};
  float rx[2], ry[2], rz[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    rx[c] = lh[c][0] + ((o8[c] - n8[c]) + (o11[c] - n11[c]));
    ry[c] = lh[c][1] + ((o7[c] - n7[c]) + (o10[c] - n10[c]));
    rz[c] = lh[c][2] + ((o6[c] - n6[c]) + (o9[c] - n9[c]));
  }
  pdl_trigger();
  put2(a, lH, q, rx[0], rx[1], true, p.v1);
  put2(a, lH + nc, q, ry[0], ry[1], true, p.v1);
  put2(a, lH + 2 * nc, q, rz[0], rz[1], true, p.v1);
}

// ======================================================= reverse H phase ===
// Primal inverse H update of a pair; the new values of its cells in hn.
template <bool EX>
__device__ __forceinline__ void primal_h(const DirectArgs& a, int x, unsigned q, bool w0, bool w1,
                                         float hn[2][3]) {
  const Geo& g = a.g;
  const unsigned rp = 4u * (unsigned)g.px, pl = 4u * (unsigned)g.plane;
  const long long nc = g.nc;
  const float* E = a.F;
  float* H = a.F + 3 * nc;
  const float2 ex = at2(E, q), ey = at2(E + nc, q), ez = at2(E + 2 * nc, q);
  const float2 ezy = at2(E + 2 * nc, q + rp), exy = at2(E, q + rp);
  const float2 exz = at2(E, q + pl), eyz = at2(E + nc, q + pl);
  const bool xn = x + 2 < g.nx;
  const float ezx = xn ? at1(E + 2 * nc, q + 8) : 0.f, eyx = xn ? at1(E + nc, q + 8) : 0.f;
  const float2 h0 = at2(H, q), h1 = at2(H + nc, q), h2 = at2(H + 2 * nc, q);
  const float d0[2] = {ezy.x - ez.x, ezy.y - ez.y}, d1[2] = {eyz.x - ey.x, eyz.y - ey.y};
  const float d2[2] = {exz.x - ex.x, exz.y - ex.y}, d3[2] = {ez.y - ez.x, ezx - ez.y};
  const float d4[2] = {ey.y - ey.x, eyx - ey.y}, d5[2] = {exy.x - ex.x, exy.y - ex.y};
  const float o0[2] = {h0.x, h0.y}, o1[2] = {h1.x, h1.y}, o2[2] = {h2.x, h2.y};
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const bool w = c == 0 ? w0 : w1;
    hn[c][0] = w ? __fadd_rn(o0[c], inc<EX>(__fmul_rn(g.S, d0[c] - d1[c]), a)) : o0[c];
    hn[c][1] = w ? __fadd_rn(o1[c], inc<EX>(__fmul_rn(g.S, d2[c] - d3[c]), a)) : o1[c];
    hn[c][2] = w ? __fadd_rn(o2[c], inc<EX>(__fmul_rn(g.S, d4[c] - d5[c]), a)) : o2[c];
  }
  pdl_trigger();
  put2(a, H, q, hn[0][0], hn[1][0], w0, w1);
  put2(a, H + nc, q, hn[0][1], hn[1][1], w0, w1);
  put2(a, H + 2 * nc, q, hn[0][2], hn[1][2], w0, w1);
}

// lam_E seeds of step n - 1 at a cell: e = E^n, h = Ht^{n-1/2} there.
__device__ __forceinline__ void seed_e(const Det& d, float s, const float e[3], const float h[3],
                                       float le[3]) {
  if (d.kind == 1) {
#pragma unroll
    for (int t = 0; t < 3; ++t) add_seed(&le[t], s, 2.0f * e[t]);
    return;
  }
  const int bb = (d.axis + 1) % 3, c = (d.axis + 2) % 3;
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    if (t == bb) add_seed(&le[t], s, c == 0 ? h[0] : (c == 1 ? h[1] : h[2]));
    if (t == c) add_seed(&le[t], -s, bb == 0 ? h[0] : (bb == 1 ? h[1] : h[2]));
  }
}

template <bool EX>
__global__ void __launch_bounds__(NT, 8) k_dir_rev_h(const __grid_constant__ DirectArgs a) {
  pdl_wait();
  if ((int)blockIdx.y < a.trows) {   // Ht^{n-1/2} of the low faces
    restore_side(a, 0, tape_value());
    return;
  }
  const Geo& g = a.g;
  const int zb = (int)blockIdx.y - a.trows;
  if (zb >= g.nz) {   // primal blocks
    const PrimalPair p = primal_pair(a, zb - g.nz + g.P);
    if (!(p.w0 || p.w1) || (a.seeded && pair_on_det(a, p.x, p.y, p.z))) return;
    float hn[2][3];
    primal_h<EX>(a, p.x, p.q, p.w0, p.w1, hn);
    return;
  }
  const Pair p = pair_of(a, zb);
  if (!p.v0) return;
  const int x = p.x, y = p.y, z = p.z;
  const unsigned q = p.q, rp = 4u * (unsigned)g.px, pl = 4u * (unsigned)g.plane;
  const long long nc = g.nc;
  float* lE = a.L;
  const float* lH = a.L + 3 * nc;
  const float* lpA = a.psiA;
  float* lpB = a.psiB;
  const float S_ = g.S;
  const bool xp = x > 0, yp = y > 0, zp = z > 0;
  const bool sx0 = in_slab(x, g.nx, g.P), sx1 = p.v1 && in_slab(x + 1, g.nx, g.P), sx = sx0 || sx1;
  const bool sxm = xp && in_slab(x - 1, g.nx, g.P);
  const bool sy = in_slab(y, g.ny, g.P), sym = yp && in_slab(y - 1, g.ny, g.P);
  const bool sz = in_slab(z, g.nz, g.P), szm = zp && in_slab(z - 1, g.nz, g.P);
  const float2 lx = at2(lH, q), ly = at2(lH + nc, q), lz = at2(lH + 2 * nc, q);
  const float2 lxy = yp ? at2(lH, q - rp) : zero2(), lzy = yp ? at2(lH + 2 * nc, q - rp) : zero2();
  const float2 lxz = zp ? at2(lH, q - pl) : zero2(), lyz = zp ? at2(lH + nc, q - pl) : zero2();
  const float lyx = xp ? at1(lH + nc, q - 4) : 0.f, lzx = xp ? at1(lH + 2 * nc, q - 4) : 0.f;
  const float2 le0 = at2(lE, q), le1 = at2(lE + nc, q), le2 = at2(lE + 2 * nc, q);
  // own terms (t0: Hx,y,+; t1: Hx,z,-; t2: Hy,z,+; t3: Hy,x,-; t4: Hz,x,+; t5: Hz,y,-), v =
  // -S s lam_H, and the same terms of the -y, -z and -x neighbours
  const float lhx[2] = {lx.x, lx.y}, lhy[2] = {ly.x, ly.y}, lhz[2] = {lz.x, lz.y};
  float o0[2], o1[2], o2[2], o3[2], o4[2], o5[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    o0[c] = __fmul_rn(-S_, lhx[c]);
    o5[c] = __fmul_rn(S_, lhz[c]);
    o1[c] = __fmul_rn(S_, lhx[c]);
    o2[c] = __fmul_rn(-S_, lhy[c]);
    o3[c] = __fmul_rn(S_, lhy[c]);
    o4[c] = __fmul_rn(-S_, lhz[c]);
  }
  float m0[2] = {__fmul_rn(-S_, lxy.x), __fmul_rn(-S_, lxy.y)}, m5[2] = {__fmul_rn(S_, lzy.x), __fmul_rn(S_, lzy.y)};
  float m1[2] = {__fmul_rn(S_, lxz.x), __fmul_rn(S_, lxz.y)}, m2[2] = {__fmul_rn(-S_, lyz.x), __fmul_rn(-S_, lyz.y)};
  float m3x = __fmul_rn(S_, lyx), m4x = __fmul_rn(-S_, lzx);
  float dummy;
  if (sy || sym) {
    if (sy) {
      const unsigned iy = psi_off<1>(a.pl, x, y, z);
      const Co ky = coef(g, 1, PR_BH, y);
      const float2 py0 = at2(psi_base<1>(a.pl, lpA, 0), iy), py1 = at2(psi_base<1>(a.pl, lpA, 1), iy);
      float s4[2], s5[2];
      o0[0] = adj(o0[0], py0.x, ky.b, ky.a, ky.k, &s4[0]);
      o0[1] = adj(o0[1], py0.y, ky.b, ky.a, ky.k, &s4[1]);
      o5[0] = adj(o5[0], py1.x, ky.b, ky.a, ky.k, &s5[0]);
      o5[1] = adj(o5[1], py1.y, ky.b, ky.a, ky.k, &s5[1]);
      put2(a, psi_base<1>(a.pl, lpB, 0), iy, s4[0], s4[1], true, p.v1);
      put2(a, psi_base<1>(a.pl, lpB, 1), iy, s5[0], s5[1], true, p.v1);
    }
    if (sym) {
      const unsigned iy = psi_off<1>(a.pl, x, y - 1, z);
      const Co kyn = coef(g, 1, PR_BH, y - 1);
      const float2 qy0 = at2(psi_base<1>(a.pl, lpA, 0), iy), qy1 = at2(psi_base<1>(a.pl, lpA, 1), iy);
      m0[0] = adj(m0[0], qy0.x, kyn.b, kyn.a, kyn.k, &dummy);
      m0[1] = adj(m0[1], qy0.y, kyn.b, kyn.a, kyn.k, &dummy);
      m5[0] = adj(m5[0], qy1.x, kyn.b, kyn.a, kyn.k, &dummy);
      m5[1] = adj(m5[1], qy1.y, kyn.b, kyn.a, kyn.k, &dummy);
    }
  }
  if (sx || sxm) {
    if (sx) {
      const unsigned ix = psi_off<0>(a.pl, x, y, z);
      const float2 px0 = at2(psi_base<0>(a.pl, lpA, 0), ix), px1 = at2(psi_base<0>(a.pl, lpA, 1), ix);
      float s0[2] = {0.f, 0.f}, s1[2] = {0.f, 0.f};
      if (sx0) {
        const Co kx0 = coef(g, 0, PR_BH, x);
        o3[0] = adj(o3[0], px0.x, kx0.b, kx0.a, kx0.k, &s0[0]);
        o4[0] = adj(o4[0], px1.x, kx0.b, kx0.a, kx0.k, &s1[0]);
      }
      if (sx1) {
        const Co kx1 = coef(g, 0, PR_BH, x + 1);
        o3[1] = adj(o3[1], px0.y, kx1.b, kx1.a, kx1.k, &s0[1]);
        o4[1] = adj(o4[1], px1.y, kx1.b, kx1.a, kx1.k, &s1[1]);
      }
      put2(a, psi_base<0>(a.pl, lpB, 0), ix, s0[0], s0[1], sx0, sx1);
      put2(a, psi_base<0>(a.pl, lpB, 1), ix, s1[0], s1[1], sx0, sx1);
    }
    if (sxm) {
      const unsigned ix = psi_off<0>(a.pl, x - 1, y, z);
      const Co kxn = coef(g, 0, PR_BH, x - 1);
      const float qx0 = at1(psi_base<0>(a.pl, lpA, 0), ix), qx1 = at1(psi_base<0>(a.pl, lpA, 1), ix);
      m3x = adj(m3x, qx0, kxn.b, kxn.a, kxn.k, &dummy);
      m4x = adj(m4x, qx1, kxn.b, kxn.a, kxn.k, &dummy);
    }
  }
  if (sz || szm) {
    if (sz) {
      const unsigned iz = psi_off<2>(a.pl, x, y, z);
      const Co kz = coef(g, 2, PR_BH, z);
      const float2 pz0 = at2(psi_base<2>(a.pl, lpA, 0), iz), pz1 = at2(psi_base<2>(a.pl, lpA, 1), iz);
      float s8[2], s9[2];
      o1[0] = adj(o1[0], pz0.x, kz.b, kz.a, kz.k, &s8[0]);
      o1[1] = adj(o1[1], pz0.y, kz.b, kz.a, kz.k, &s8[1]);
      o2[0] = adj(o2[0], pz1.x, kz.b, kz.a, kz.k, &s9[0]);
      o2[1] = adj(o2[1], pz1.y, kz.b, kz.a, kz.k, &s9[1]);
      put2(a, psi_base<2>(a.pl, lpB, 0), iz, s8[0], s8[1], true, p.v1);
      put2(a, psi_base<2>(a.pl, lpB, 1), iz, s9[0], s9[1], true, p.v1);
    }
    if (szm) {
      const unsigned iz = psi_off<2>(a.pl, x, y, z - 1);
      const Co kzn = coef(g, 2, PR_BH, z - 1);
      const float2 qz0 = at2(psi_base<2>(a.pl, lpA, 0), iz), qz1 = at2(psi_base<2>(a.pl, lpA, 1), iz);
      m1[0] = adj(m1[0], qz0.x, kzn.b, kzn.a, kzn.k, &dummy);
      m1[1] = adj(m1[1], qz0.y, kzn.b, kzn.a, kzn.k, &dummy);
      m2[0] = adj(m2[0], qz1.x, kzn.b, kzn.a, kzn.k, &dummy);
      m2[1] = adj(m2[1], qz1.y, kzn.b, kzn.a, kzn.k, &dummy);
    }
  }
  // cell 1's -x terms are cell 0's own terms
  const float m3[2] = {m3x, o3[0]}, m4[2] = {m4x, o4[0]};
  const float eo[2][3] = {{le0.x, le1.x, le2.x}, {le0.y, le1.y, le2.y}};
  float le[2][3];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    le[c][0] = eo[c][0] + ((m2[c] - o2[c]) + (m5[c] - o5[c]));
    le[c][1] = eo[c][1] + ((m1[c] - o1[c]) + (m4[c] - o4[c]));
    le[c][2] = eo[c][2] + ((m0[c] - o0[c]) + (m3[c] - o3[c]));
  }
  if (a.seeded && pair_on_det(a, x, y, z)) {
    bool w0, w1;
    float hn[2][3];
    primal_cells(g, x, y, z, &w0, &w1);
    primal_h<EX>(a, x, q, w0, w1, hn);
    const float2 e0 = at2(a.F, q), e1 = at2(a.F + nc, q), e2 = at2(a.F + 2 * nc, q);
    const float e[2][3] = {{e0.x, e1.x, e2.x}, {e0.y, e1.y, e2.y}};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (in_box(a.dbox, x + c, y, z)) seed_e(a.det, (float)a.seeds[0], e[c], hn[c], le[c]);
      if (in_box(a.dbox2, x + c, y, z)) seed_e(a.det2, (float)a.seeds[1], e[c], hn[c], le[c]);
    }
  }
  pdl_trigger();
  put2(a, lE, q, le[0][0], le[1][0], true, p.v1);
  put2(a, lE + nc, q, le[0][1], le[1][1], true, p.v1);
  put2(a, lE + 2 * nc, q, le[0][2], le[1][2], true, p.v1);
}

}  // namespace direct

using namespace direct;

template <class KT>
static cudaError_t launch_dep(KT kernel, dim3 grid, cudaStream_t s, const DirectArgs& a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(NT);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.dep ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

// which: 0 forward H, 1 forward E, 2 reverse E phase, 3 reverse H phase.
// a.tmode != 0 adds the tape blocks of the side the phase handles (0, 2: the
// high faces' E; 1, 3: the low faces' Ht).
static DirectBox box_of(int kind, int axis, int index, int u0, int u1, int v0, int v1) {
  DirectBox b = {{0, 0, 0}, {0, 0, 0}};
  if (!kind) return b;
  const int ua = axis == 0 ? 1 : 0, va = axis == 2 ? 1 : 2;
  b.lo[axis] = index; b.hi[axis] = index + 1;
  b.lo[ua] = u0; b.hi[ua] = u1;
  b.lo[va] = v0; b.hi[va] = v1;
  return b;
}

// What the kernels' index arithmetic takes: byte offsets below 2^32 within a
// component array, plane and row counts within the grid's dimensions, and
// exact quotients by multiplication (see quot).
bool direct_fits(const Geo& g) {
  const long long h = g.px / 2, i = g.plane / 2 + NT;
  return 4 * g.nc < (1LL << 32) && i * h < (1LL << 32) && g.nz <= 16000 && g.nx > 2 * g.P &&
         g.ny > 2 * g.P && g.nz > 2 * g.P;
}

cudaError_t launch_direct(int which, const DirectArgs& a_, cudaStream_t s) {
  DirectArgs a = a_;
  const Geo& g = a.g;
  if (!direct_fits(g)) return cudaErrorInvalidValue;
  const int side = (which == 0 || which == 2) ? 1 : 0;
  int nv = 0;
  for (int f = side; f < 6; f += 2) nv += a.fc.start[f + 1] - a.fc.start[f];
  a.sbox = box_of(a.src.kind, a.src.axis, a.src.index, a.src.u0, a.src.u1, a.src.v0, a.src.v1);
  a.dbox = box_of(a.det.kind, a.det.axis, a.det.index, a.det.u0, a.det.u1, a.det.v0, a.det.v1);
  a.dbox2 = box_of(a.det2.kind, a.det2.axis, a.det2.index, a.det2.u0, a.det2.u1, a.det2.v0,
                   a.det2.v1);
  auto magic = [](int h) { return (unsigned)(((1ULL << 32) + h - 1) / h); };
  a.mrow = magic(g.px >> 1);
  a.mint = magic(((g.nx - g.P + 1) >> 1) - (g.P >> 1));
  const int nbp = (int)((g.plane / 2 + NT - 1) / NT);   // blocks per plane
  a.trows = a.tmode ? (nv + nbp * NT - 1) / (nbp * NT) : 0;
  auto pairs = [](const DirectBox& b) {
    return (((b.hi[0] + 1) >> 1) - (b.lo[0] >> 1)) * (b.hi[1] - b.lo[1]) * (b.hi[2] - b.lo[2]);
  };
  a.dpairs = pairs(a.dbox);
  a.dpairs2 = pairs(a.dbox2);
  a.drows = which == 1 ? (a.dpairs + a.dpairs2 + nbp * NT - 1) / (nbp * NT) : 0;
  const dim3 grid(nbp, a.trows + a.drows + g.nz + (which >= 2 ? g.nz - 2 * g.P : 0));
  const bool ex = a.xq != 0;
  switch (which) {
    case 0:
      return ex ? launch_dep(k_dir_fwd_h<true>, grid, s, a) : launch_dep(k_dir_fwd_h<false>, grid, s, a);
    case 1:
      return ex ? launch_dep(k_dir_fwd_e<true>, grid, s, a) : launch_dep(k_dir_fwd_e<false>, grid, s, a);
    case 2:
      return ex ? launch_dep(k_dir_rev_e<true>, grid, s, a) : launch_dep(k_dir_rev_e<false>, grid, s, a);
    case 3:
      return ex ? launch_dep(k_dir_rev_h<true>, grid, s, a) : launch_dep(k_dir_rev_h<false>, grid, s, a);
  }
  return cudaErrorInvalidValue;
}

}  // namespace fdtd
