// kernels_fwd_fused.cu -- one forward time step of a unit in one pass, CPML included.
//
// A forward step n of the leapfrog (the simulation whose gradient Sec. 2
// computes):
//     Ht^{n+1/2} = Ht^{n-1/2} - S curl E^n              (forward differences)
//     E^{n+1}    = E^n + cb (curl Ht^{n+1/2} - J)       (backward differences)
// The split half-steps (kernels_lag2.cu) read E and Ht in both launches, 76 B
// per cell.  Here a CTA runs both half-steps of its unit in one pass: it reads
// E^n, Ht^{n-1/2} and cb once and writes E^{n+1} and Ht^{n+1/2} once (52 B) into
// the other buffer of a ping-pong pair, so no CTA reads a value another CTA of
// the launch has already replaced; the auxiliaries go from one set to another in
// the same way.
//
// E^{n+1} of a cell needs Ht^{n+1/2} at -x, -y and -z.  Across z it comes one
// iteration later (the E update lags one plane); across x and y the CTA computes
// Ht^{n+1/2} itself on a one-cell halo of its tile (a fifth warp: a row of 16
// pairs at y0-1 and a column of 8 cells at x0-1), from the same staged inputs,
// the halo's own CPML terms among them.  Every cell sees the same sequence of
// explicitly rounded operations as in the split kernels, so the fields are
// bit-identical to theirs.  The exchange between the half-steps happens in the
// staged Ht box: a pair's Ht^{n-1/2} is read by its own thread only, which then
// puts Ht^{n+1/2} of the plane before in its place.
//
// Units come in five kinds by the CPML axes they can meet, each with a kernel that
// stages and tests only those (PX, PY, PZ): the CPML-free box, the tiles of the
// box below and above it (z), the tile columns beside it (x and z), the tile
// rows beside it (y and z), the corners (all).  The source and the detector may
// lie in any unit.
//
// What bounds it: DRAM for the z units (162 us for 1.0 GB on 600 x 600 x 300), the
// instructions and latency of two barriers per plane for the columns (177 us) and
// corners.  Two stages, so that four (corners) or five CTAs fit an SM.  Against the
// split half-steps over the same units (526 us per step): 474 us, and step n of
// these units reads nothing the two-step pass writes, so that it runs beside the
// pass: 1031 -> 962 us per forward step on 600 x 600 x 300, 373 -> 347 on 411 x 389 x
// 203 (before the pass itself changed).
#include <cudaTypedefs.h>

#include "lag_common.cuh"

namespace fdtd {

using namespace lag2;

namespace fwdf {

constexpr int TW = 32, TY = 8;

// Shared memory (byte offsets): S stages of an E box (TW+8) x (TY+2) and an Ht
// box (TW+4) x (TY+1) at (x0-4, y0-1) (3 components each) of plane p, the cb box
// TW x TY of plane p-1; per CPML axis the auxiliaries of the H half-step at plane p
// ((TW+4) x (TY+1) at (x0-4, y0-1)) and of the E half-step at plane p-1 (TW x TY).
// The stages' mbarriers and, with x / y CPML terms, the profiles of the tile's
// cells and halo follow.
template <int S, bool PX, bool PY, bool PZ>
struct FL {
  static constexpr int WW = TW + 8, WR = TY + 2, WP = WW * WR;
  static constexpr int HW = TW + 4, HR = TY + 1, HP = HW * HR;
  static constexpr int OP = TW * TY;
  static constexpr int E = 0;
  static constexpr int H = E + r128(3 * WP * 4);
  static constexpr int CB = H + r128(3 * HP * 4);
  static constexpr int HX = CB + r128(OP * 4);
  static constexpr int HY = HX + (PX ? r128(2 * HP * 4) : 0);
  static constexpr int HZ = HY + (PY ? r128(2 * HP * 4) : 0);
  static constexpr int EX = HZ + (PZ ? r128(2 * HP * 4) : 0);
  static constexpr int EY = EX + (PX ? r128(2 * OP * 4) : 0);
  static constexpr int EZ = EY + (PY ? r128(2 * OP * 4) : 0);
  static constexpr int STAGE = EZ + (PZ ? r128(2 * OP * 4) : 0);
  static constexpr int BARS = S * STAGE;
  static constexpr int SP = r128(BARS + 8 * S), SPXN = TW + 4, SPYN = TY + 4;
  static constexpr int RED = SP + ((PX ? 6 * SPXN : 0) + (PY ? 6 * SPYN : 0)) * 4;
  static int smem() { return RED + 8 * 8; }
};

template <int S, bool EX, bool PX, bool PY, bool PZ>
__global__ void __launch_bounds__(TW / 2 * (TY + 2), (PX && PY ? 4 : 5))
k_fwd_fused(const __grid_constant__ FwdMaps m, const __grid_constant__ StepArgs a) {
  typedef FL<S, PX, PY, PZ> Y;
  extern __shared__ __align__(128) unsigned char dsm[];
  const Geo& g = a.g;
  const RevUnits& U = a.U;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * (TW / 2) + tx;
  // the unit: columns / rows beside the box are its left, then its right ones
  const int bx = blockIdx.x, by = blockIdx.y, bz = blockIdx.z;
  const int tix = PX ? (bx < U.ix0 ? bx : U.ix1 + (bx - U.ix0)) : bx + U.ix0;
  const int tiy = PY ? (by < U.iy0 ? by : U.iy1 + (by - U.iy0)) : by + U.iy0;
  const int cz = PX || PY ? bz : (PZ ? zonly_chunk(U, bz) : bz + U.iz0);
  const int x0 = tix * TW, y0 = tiy * TY;
  const int k0 = cz * a.zchunk, k1 = min(g.nz, k0 + a.zchunk);
  // task: the tile's pair (main), a pair of the -y halo row, or the -x halo
  // column (pair x0-2, x0-1)
  const bool mainT = ty < TY;
  const bool rowT = ty == TY;
  const bool colT = ty == TY + 1 && tx < TY;
  const bool task = mainT || rowT || colT;
  const int x = colT ? x0 - 2 : x0 + 2 * tx;
  const int y = mainT ? y0 + ty : (rowT ? y0 - 1 : y0 + tx);
  const bool iny = !PY || (y >= 0 && y < g.ny);
  const bool v0 = mainT && iny && (!PX || x < g.nx), v1 = mainT && iny && (!PX || x + 1 < g.nx);
  const bool outside = (PX && x < 0) || (PY && y < 0);   // halo beyond the grid: Ht = 0
  bool sx0 = false, sx1 = false, sy = false;
  if (PX) {
    sx0 = task && iny && x >= 0 && x < g.nx && in_slab(x, g.nx, g.P);
    sx1 = task && iny && x + 1 >= 0 && x + 1 < g.nx && in_slab(x + 1, g.nx, g.P);
  }
  if (PY) sy = task && iny && in_slab(y, g.ny, g.P);
  // the x / y profiles the tile's cells and halo read, [6][TW+4] from x0-4 and
  // [6][TY+4] from y0-2
  float* SPX = reinterpret_cast<float*>(dsm + Y::SP);
  float* SPY = SPX + (PX ? 6 * Y::SPXN : 0);
  constexpr int NTH = TW / 2 * (TY + 2);
  if (PX)
    for (int i = tid; i < 6 * Y::SPXN; i += NTH) {
      const int w = i / Y::SPXN, xi = x0 - 4 + i % Y::SPXN;
      SPX[i] = (xi >= 0 && xi < g.nx) ? prof(g, 0, w, xi) : 0.f;
    }
  if (PY)
    for (int i = tid; i < 6 * Y::SPYN; i += NTH) {
      const int w = i / Y::SPYN, yi = y0 - 2 + i % Y::SPYN;
      SPY[i] = (yi >= 0 && yi < g.ny) ? prof(g, 1, w, yi) : 0.f;
    }
  auto spx = [&](int w, int xx) { return SPX[w * Y::SPXN + xx - x0 + 4]; };
  auto spy = [&](int w) { return SPY[w * Y::SPYN + y - y0 + 2]; };
  // plane k0-1 starts Ht'(k0-1); plane p in [k0, k1) finishes Ht'(p-1),
  // updates E(p-1) (from k0+1 on) and starts Ht'(p); plane k1 finishes
  // Ht'(k1-1) and updates E(k1-1)
  const int p0_ = k0 - 1, p1_ = k1;
  uint64_t* bars = ring_init<S>(dsm, Y::STAGE);   // at Y::BARS (also syncs the profiles)
  int qx0 = x0, qy0 = y0;
  bool txh = false, txe = false, tyh = false, tye = false;
  if (PX || PY) psi_box_starts<TW, TY>(a.pl, x0, y0, &qx0, &qy0);
  if (PX) {
    txh = tile_in_slab(max(x0 - 2, 0), min(x0 + TW - 1, g.nx - 1), g.nx, g.P);
    txe = tile_in_slab(x0, min(x0 + TW - 1, g.nx - 1), g.nx, g.P);
  }
  if (PY) {
    tyh = tile_in_slab(max(y0 - 1, 0), min(y0 + TY - 1, g.ny - 1), g.ny, g.P);
    tye = tile_in_slab(y0, min(y0 + TY - 1, g.ny - 1), g.ny, g.P);
  }
  auto boxes = [&](int p, auto&& f) {
    if (p >= 0) {
      f(Y::E, &m.F40, x0 - 4, y0 - 1, p, 0, 3 * Y::WP * 4);   // plane nz: zeros
      if (p < k1) {
        f(Y::H, &m.F36, x0 - 4, y0 - 1, p, 3, 3 * Y::HP * 4);
        if (PX && txh) f(Y::HX, &m.Qx36, qx0 - 4, y0 - 1, p, 0, 2 * Y::HP * 4);
        if (PY && tyh) f(Y::HY, &m.Qy36, x0 - 4, qy0 - 1, p, 0, 2 * Y::HP * 4);
        if (PZ && in_slab(p, g.nz, g.P))
          f(Y::HZ, &m.Qz36, x0 - 4, y0 - 1, psi_map(a.pl.ax[2], p), 0, 2 * Y::HP * 4);
      }
    }
    const int pm = p - 1;
    if (pm >= k0) {
      f(Y::CB, &m.cb32, x0, y0, pm, 0, Y::OP * 4);
      if (PX && txe) f(Y::EX, &m.Qxo, qx0, y0, pm, 2, 2 * Y::OP * 4);
      if (PY && tye) f(Y::EY, &m.Qyo, x0, qy0, pm, 2, 2 * Y::OP * 4);
      if (PZ && in_slab(pm, g.nz, g.P))
        f(Y::EZ, &m.Qzo, x0, y0, psi_map(a.pl.ax[2], pm), 2, 2 * Y::OP * 4);
    }
  };
  auto issue = [&](int p, unsigned char* st, uint64_t* bar) {
    stage_plane(boxes, p, st, bar, false);
  };
  if (tid == 0)
    for (int i = 0; i < S && p0_ + i <= p1_; ++i) issue(p0_ + i, dsm + i * Y::STAGE, bars + i);
  const int wb = (y - y0 + 1) * Y::WW + (x - x0 + 4);   // the pair in the E box
  const int hb = (y - y0 + 1) * Y::HW + (x - x0 + 4);   // the pair in the Ht and psi_H boxes
  const int ob = (y - y0) * TW + (x - x0);               // the pair in the own boxes (main)
  const float S_ = g.S;
  const long long nc = g.nc;
  const unsigned oxy = 4u * (unsigned)(y * g.px + x);    // the pair within a plane (bytes)
  const unsigned opx = PX ? 4u * (unsigned)(y * a.pl.ax[0].d0 + psi_map(a.pl.ax[0], x)) : 0u;
  const unsigned opy = PY ? 4u * (unsigned)(psi_map(a.pl.ax[1], y) * a.pl.ax[1].d0 + x) : 0u;
  // component c of axis ax's auxiliaries, plane (or row) z, of the set written
  auto psi_plane = [&](int ax, int c, int z) {
    const PsiAxis& A = a.pl.ax[ax];
    return a.psiB + A.off + c * A.cs + (ax == 2 ? psi_map(A, z) : z) * A.ps;
  };
  // do the source and the detector planes meet the unit's cells?
  const bool src = a.src.kind && (a.src.axis == 0 ? a.src.index >= x0 && a.src.index < x0 + TW
                                  : a.src.axis == 1 ? a.src.index >= y0 && a.src.index < y0 + TY
                                                    : a.src.index >= k0 && a.src.index < k1);
  const bool det = a.det.kind && (a.det.axis == 0 ? a.det.index >= x0 && a.det.index < x0 + TW
                                  : a.det.axis == 1 ? a.det.index >= y0 && a.det.index < y0 + TY
                                                    : a.det.index >= k0 && a.det.index < k1);
  // Ht'(p-1) in progress at the pair: E(p-1), the x / y difference terms, Ht(p-1), its
  // z auxiliaries
  float c_ex[2] = {0.f, 0.f}, c_ey[2] = {0.f, 0.f}, c_ez[2] = {0.f, 0.f};
  float c_t0[2] = {0.f, 0.f}, c_t3[2] = {0.f, 0.f}, c_t4[2] = {0.f, 0.f}, c_t5[2] = {0.f, 0.f};
  float c_hx[2] = {0.f, 0.f}, c_hy[2] = {0.f, 0.f}, c_hz[2] = {0.f, 0.f};
  float c_pz0[2] = {0.f, 0.f}, c_pz1[2] = {0.f, 0.f};
  float c_fx[2] = {0.f, 0.f}, c_fy[2] = {0.f, 0.f};   // Ht'x, Ht'y of plane p-2
  double lsum = 0.0;
  int stg = 0;
  uint32_t par = 0;
  bool ok = true;
  for (int p = p0_; p <= p1_; ++p) {
    unsigned char* st = dsm + stg * Y::STAGE;
    const bool head = p < k0, tail = p == k1;
    // z profiles of plane p - 1, on their way while plane p arrives
    const bool sz = PZ && p >= 1 && !head && in_slab(p - 1, g.nz, g.P);
    float bzh = 0.f, azh = 0.f, kzh = 0.f, bze = 0.f, aze = 0.f, kze = 0.f;
    if (sz) {
      bzh = prof(g, 2, PR_BH, p - 1); azh = prof(g, 2, PR_AH, p - 1); kzh = prof(g, 2, PR_KH, p - 1);
      bze = prof(g, 2, PR_BE, p - 1); aze = prof(g, 2, PR_AE, p - 1); kze = prof(g, 2, PR_KE, p - 1);
    }
    if (!mbar_wait(bars + stg, par, kWaitCycles)) ok = false;
    const float* Eb = reinterpret_cast<const float*>(st + Y::E) + wb;
    float* Hb = reinterpret_cast<float*>(st + Y::H) + hb;
    float fx[2] = {0.f, 0.f}, fy[2] = {0.f, 0.f}, fz[2] = {0.f, 0.f};   // Ht'(p-1) at the pair
    // ---- finish Ht'(p-1) with dEy/dz and dEx/dz ----
    if (task && !head) {
      if (p >= 1 && !outside) {
        const float2 ex2 = ld2(Eb, 0), ey2 = ld2(Eb, Y::WP);
        const float ex[2] = {ex2.x, ex2.y}, ey[2] = {ey2.x, ey2.y};
        float t1[2], t2[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          t1[c] = ey[c] - c_ey[c];
          t2[c] = ex[c] - c_ex[c];
        }
        if (sz) {
          float s1[2], s2[2];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            t1[c] = cpml(t1[c], c_pz0[c], bzh, azh, kzh, &s1[c]);
            t2[c] = cpml(t2[c], c_pz1[c], bzh, azh, kzh, &s2[c]);
          }
          if (p - 1 >= k0) {
            put2(a, psi_plane(2, 0, p - 1), oxy, s1[0], s1[1], v0, v1);
            put2(a, psi_plane(2, 1, p - 1), oxy, s2[0], s2[1], v0, v1);
          }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float cx = c_t0[c] - t1[c], cy = t2[c] - c_t3[c], czz = c_t4[c] - c_t5[c];
          fx[c] = __fsub_rn(c_hx[c], inc_of<EX>(__fmul_rn(S_, cx), a));
          fy[c] = __fsub_rn(c_hy[c], inc_of<EX>(__fmul_rn(S_, cy), a));
          fz[c] = __fsub_rn(c_hz[c], inc_of<EX>(__fmul_rn(S_, czz), a));
        }
        if (p - 1 >= k0) {
          float* O = a.Fn + 3 * nc + (p - 1) * g.plane;
          put2(a, O, oxy, fx[0], fx[1], v0, v1);
          put2(a, O + nc, oxy, fy[0], fy[1], v0, v1);
          put2(a, O + 2 * nc, oxy, fz[0], fz[1], v0, v1);
        }
      }
    }
    if (task) {   // Ht(p) leaves its box, Ht'(p-1) takes its place
      if (!tail) {
        const float2 h0 = ld2(Hb, 0), h1 = ld2(Hb, Y::HP), h2 = ld2(Hb, 2 * Y::HP);
        c_hx[0] = h0.x; c_hx[1] = h0.y;
        c_hy[0] = h1.x; c_hy[1] = h1.y;
        c_hz[0] = h2.x; c_hz[1] = h2.y;
      }
      if (!head) {
        *reinterpret_cast<float2*>(Hb) = make_float2(fx[0], fx[1]);
        *reinterpret_cast<float2*>(Hb + Y::HP) = make_float2(fy[0], fy[1]);
        *reinterpret_cast<float2*>(Hb + 2 * Y::HP) = make_float2(fz[0], fz[1]);
      }
    }
    // Ht'(p-1) of the tile and its halo is in the stage; a wait that gave up ends
    // the CTA here
    if (!__syncthreads_and(ok)) { ring_abort<S>(bars, stg, par, p, p1_, a.err); return; }
    // ---- E'(p-1), one plane behind ----
    if (mainT && p - 1 >= k0) {
      const float2 hzy = ld2(Hb, 2 * Y::HP - Y::HW), hxy = ld2(Hb, -Y::HW);   // -y
      const float hzx = Hb[2 * Y::HP - 1], hyx = Hb[Y::HP - 1];                 // -x of cell 0
      float t6[2] = {fz[0] - hzy.x, fz[1] - hzy.y};        // dHz/dy
      float t7[2] = {fy[0] - c_fy[0], fy[1] - c_fy[1]};    // dHy/dz
      float t8[2] = {fx[0] - c_fx[0], fx[1] - c_fx[1]};    // dHx/dz
      float t9[2] = {fz[0] - hzx, fz[1] - fz[0]};          // dHz/dx
      float t10[2] = {fy[0] - hyx, fy[1] - fy[0]};         // dHy/dx
      float t11[2] = {fx[0] - hxy.x, fx[1] - hxy.y};       // dHx/dy
      if (PX && (sx0 || sx1)) {
        const float* P = reinterpret_cast<const float*>(st + Y::EX) + ob;
        const float2 p0 = ld2(P, 0), p1 = ld2(P, Y::OP);
        float s9[2] = {0.f, 0.f}, s10[2] = {0.f, 0.f};
        if (sx0) {
          const float b = spx(PR_BE, x), aa = spx(PR_AE, x), kk = spx(PR_KE, x);
          t9[0] = cpml(t9[0], p0.x, b, aa, kk, &s9[0]);
          t10[0] = cpml(t10[0], p1.x, b, aa, kk, &s10[0]);
        }
        if (sx1) {
          const float b = spx(PR_BE, x + 1), aa = spx(PR_AE, x + 1), kk = spx(PR_KE, x + 1);
          t9[1] = cpml(t9[1], p0.y, b, aa, kk, &s9[1]);
          t10[1] = cpml(t10[1], p1.y, b, aa, kk, &s10[1]);
        }
        put2(a, psi_plane(0, 2, p - 1), opx, s9[0], s9[1], sx0, sx1);
        put2(a, psi_plane(0, 3, p - 1), opx, s10[0], s10[1], sx0, sx1);
      }
      if (PY && sy) {
        const float* P = reinterpret_cast<const float*>(st + Y::EY) + ob;
        const float b = spy(PR_BE), aa = spy(PR_AE), kk = spy(PR_KE);
        const float2 p0 = ld2(P, 0), p1 = ld2(P, Y::OP);
        float s6[2], s11[2];
        t6[0] = cpml(t6[0], p0.x, b, aa, kk, &s6[0]);
        t6[1] = cpml(t6[1], p0.y, b, aa, kk, &s6[1]);
        t11[0] = cpml(t11[0], p1.x, b, aa, kk, &s11[0]);
        t11[1] = cpml(t11[1], p1.y, b, aa, kk, &s11[1]);
        put2(a, psi_plane(1, 2, p - 1), opy, s6[0], s6[1], v0, v1);
        put2(a, psi_plane(1, 3, p - 1), opy, s11[0], s11[1], v0, v1);
      }
      if (sz) {
        const float* P = reinterpret_cast<const float*>(st + Y::EZ) + ob;
        const float2 p0 = ld2(P, 0), p1 = ld2(P, Y::OP);
        float s7[2], s8[2];
        t7[0] = cpml(t7[0], p0.x, bze, aze, kze, &s7[0]);
        t7[1] = cpml(t7[1], p0.y, bze, aze, kze, &s7[1]);
        t8[0] = cpml(t8[0], p1.x, bze, aze, kze, &s8[0]);
        t8[1] = cpml(t8[1], p1.y, bze, aze, kze, &s8[1]);
        put2(a, psi_plane(2, 2, p - 1), oxy, s7[0], s7[1], v0, v1);
        put2(a, psi_plane(2, 3, p - 1), oxy, s8[0], s8[1], v0, v1);
      }
      const float2 cb2 = ld2(reinterpret_cast<const float*>(st + Y::CB), ob);
      const float cbv[2] = {cb2.x, cb2.y};
      float ex[2], ey[2], ez[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float c0 = t6[c] - t7[c], c1 = t8[c] - t9[c], c2 = t10[c] - t11[c];
        if (src) {
          const float w = (c == 0 ? v0 : v1) ? src_wt(a.src, x + c, y, p - 1) : 0.f;
          if (w != 0.f) {
            const float wj = __fmul_rn(w, a.jn);
            if (a.src.comp == 0) c0 = __fsub_rn(c0, wj);
            else if (a.src.comp == 1) c1 = __fsub_rn(c1, wj);
            else c2 = __fsub_rn(c2, wj);
          }
        }
        ex[c] = __fadd_rn(c_ex[c], inc_of<EX>(__fmul_rn(cbv[c], c0), a));
        ey[c] = __fadd_rn(c_ey[c], inc_of<EX>(__fmul_rn(cbv[c], c1), a));
        ez[c] = __fadd_rn(c_ez[c], inc_of<EX>(__fmul_rn(cbv[c], c2), a));
      }
      float* O = a.Fn + (p - 1) * g.plane;
      put2(a, O, oxy, ex[0], ex[1], v0, v1);
      put2(a, O + nc, oxy, ey[0], ey[1], v0, v1);
      put2(a, O + 2 * nc, oxy, ez[0], ez[1], v0, v1);
      if (det) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          int u, v;
          if ((c == 0 ? v0 : v1) && on_plane(a.det.axis, a.det.index, a.det.u0, a.det.u1, a.det.v0,
                                             a.det.v1, x + c, y, p - 1, &u, &v)) {
            if (a.det.kind == 1) {
              lsum += (double)ex[c] * ex[c] + (double)ey[c] * ey[c] + (double)ez[c] * ez[c];
            } else {
              const int ax_ = a.det.axis;
              const float Eb_ = ax_ == 0 ? ey[c] : (ax_ == 1 ? ez[c] : ex[c]);
              const float Ec_ = ax_ == 0 ? ez[c] : (ax_ == 1 ? ex[c] : ey[c]);
              const float Hb_ = ax_ == 0 ? fy[c] : (ax_ == 1 ? fz[c] : fx[c]);
              const float Hc_ = ax_ == 0 ? fz[c] : (ax_ == 1 ? fx[c] : fy[c]);
              lsum += (double)Eb_ * Hc_ - (double)Ec_ * Hb_;
            }
          }
        }
      }
    }
    if (!head) {   // Ht'(p-1) at the pair: the -z neighbour of E'(p)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        c_fx[c] = fx[c];
        c_fy[c] = fy[c];
      }
    }
    // ---- start Ht'(p): its x and y differences ----
    if (task && !tail && p >= 0) {
      const float2 ex2 = ld2(Eb, 0), ey2 = ld2(Eb, Y::WP), ez2 = ld2(Eb, 2 * Y::WP);
      const float2 ezy = ld2(Eb, 2 * Y::WP + Y::WW), exy = ld2(Eb, Y::WW);   // +y
      const float ezx = Eb[2 * Y::WP + 2], eyx = Eb[Y::WP + 2];                // +x of cell 1
      c_t0[0] = ezy.x - ez2.x; c_t0[1] = ezy.y - ez2.y;   // dEz/dy
      c_t3[0] = ez2.y - ez2.x; c_t3[1] = ezx - ez2.y;     // dEz/dx
      c_t4[0] = ey2.y - ey2.x; c_t4[1] = eyx - ey2.y;     // dEy/dx
      c_t5[0] = exy.x - ex2.x; c_t5[1] = exy.y - ex2.y;   // dEx/dy
      c_ex[0] = ex2.x; c_ex[1] = ex2.y;
      c_ey[0] = ey2.x; c_ey[1] = ey2.y;
      c_ez[0] = ez2.x; c_ez[1] = ez2.y;
      if (PX && (sx0 || sx1)) {
        const float* P = reinterpret_cast<const float*>(st + Y::HX) + hb;
        const float2 p0 = ld2(P, 0), p1 = ld2(P, Y::HP);
        float s3[2] = {0.f, 0.f}, s4[2] = {0.f, 0.f};
        if (sx0) {
          const float b = spx(PR_BH, x), aa = spx(PR_AH, x), kk = spx(PR_KH, x);
          c_t3[0] = cpml(c_t3[0], p0.x, b, aa, kk, &s3[0]);
          c_t4[0] = cpml(c_t4[0], p1.x, b, aa, kk, &s4[0]);
        }
        if (sx1) {
          const float b = spx(PR_BH, x + 1), aa = spx(PR_AH, x + 1), kk = spx(PR_KH, x + 1);
          c_t3[1] = cpml(c_t3[1], p0.y, b, aa, kk, &s3[1]);
          c_t4[1] = cpml(c_t4[1], p1.y, b, aa, kk, &s4[1]);
        }
        if (mainT && !head) {
          put2(a, psi_plane(0, 0, p), opx, s3[0], s3[1], sx0, sx1);
          put2(a, psi_plane(0, 1, p), opx, s4[0], s4[1], sx0, sx1);
        }
      }
      if (PY && sy) {
        const float* P = reinterpret_cast<const float*>(st + Y::HY) + hb;
        const float b = spy(PR_BH), aa = spy(PR_AH), kk = spy(PR_KH);
        const float2 p0 = ld2(P, 0), p1 = ld2(P, Y::HP);
        float s0[2], s5[2];
        c_t0[0] = cpml(c_t0[0], p0.x, b, aa, kk, &s0[0]);
        c_t0[1] = cpml(c_t0[1], p0.y, b, aa, kk, &s0[1]);
        c_t5[0] = cpml(c_t5[0], p1.x, b, aa, kk, &s5[0]);
        c_t5[1] = cpml(c_t5[1], p1.y, b, aa, kk, &s5[1]);
        if (!head) {
          put2(a, psi_plane(1, 0, p), opy, s0[0], s0[1], v0, v1);
          put2(a, psi_plane(1, 1, p), opy, s5[0], s5[1], v0, v1);
        }
      }
      if (PZ && in_slab(p, g.nz, g.P)) {
        const float* P = reinterpret_cast<const float*>(st + Y::HZ) + hb;
        const float2 p0 = ld2(P, 0), p1 = ld2(P, Y::HP);
        c_pz0[0] = p0.x; c_pz0[1] = p0.y;
        c_pz1[0] = p1.x; c_pz1[1] = p1.y;
      }
    }
    __syncthreads();   // the stage is free again
    if (tid == 0 && p + S <= p1_) issue(p + S, st, bars + stg);
    if (++stg == S) { stg = 0; par ^= 1u; }
  }
  if (det) {
    double* red = reinterpret_cast<double*>(dsm + Y::RED);
    double v = lsum;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((tid & 31) == 0) red[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int wv = 0; wv < NTH / 32; ++wv) t += red[wv];
      if (t != 0.0) atomicAdd(a.obj, t);
    }
  }
}

template <int S, bool EX, bool PX, bool PY, bool PZ>
static cudaError_t launch_ff(const FwdMaps& m, const StepArgs& a, dim3 grid, cudaStream_t s) {
  auto kernel = k_fwd_fused<S, EX, PX, PY, PZ>;
  const int smem = FL<S, PX, PY, PZ>::smem();
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e) return e;
  kernel<<<grid, dim3(TW / 2, TY + 2), smem, s>>>(m, a);
  return cudaGetLastError();
}

template <bool EX>
static cudaError_t launch_kind(int kind, const FwdMaps& m, const StepArgs& a, dim3 grid,
                               cudaStream_t s) {
  switch (kind) {
    case 0: return launch_ff<2, EX, false, false, false>(m, a, grid, s);
    case 1: return launch_ff<2, EX, false, false, true>(m, a, grid, s);
    case 2: return launch_ff<2, EX, true, false, true>(m, a, grid, s);
    case 3: return launch_ff<2, EX, false, true, true>(m, a, grid, s);
    case 4: return launch_ff<2, EX, true, true, true>(m, a, grid, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace fwdf

cudaError_t launch_fwd_fused(int kind, const FwdMaps& m, const StepArgs& a, const RevUnits& U,
                             cudaStream_t s) {
  if (a.tile_y != fwdf::TY || a.tile_x != fwdf::TW || !a.Fn || !a.psiB)
    return cudaErrorInvalidValue;
  const int nix = U.ix1 - U.ix0, niy = U.iy1 - U.iy0, niz = U.iz1 - U.iz0;
  const int cols = U.ntx - nix, rows = U.nty - niy;
  dim3 grid(0, 0, 0);
  switch (kind) {
    case 0: grid = dim3(nix, niy, niz); break;
    case 1: grid = dim3(nix, niy, U.nzc - niz); break;
    case 2: grid = dim3(cols, niy, U.nzc); break;
    case 3: grid = dim3(nix, rows, U.nzc); break;
    case 4: grid = dim3(cols, rows, U.nzc); break;
    default: return cudaErrorInvalidValue;
  }
  if (grid.x == 0 || grid.y == 0 || grid.z == 0) return cudaSuccess;
  StepArgs b = a;
  b.U = U;
  return a.xq ? fwdf::launch_kind<true>(kind, m, b, grid, s)
              : fwdf::launch_kind<false>(kind, m, b, grid, s);
}

}  // namespace fdtd
