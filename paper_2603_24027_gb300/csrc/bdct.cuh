// bdct.cuh -- block-transform tape codec (tape type 9).
//
// Beyond the paper (Sec. 4 names JPEG-like compression of the boundary tape
// as future work): every face component [v][u] of a tape sample is cut into
// 8 x 8 blocks (cells past the face edge repeat the last row / column), each
// block goes through the orthonormal 2D DCT-II, and the first K coefficients
// in diagonal order (u + v ascending, then v ascending) are kept as int8
// codes round(C / s) with one float32 scale s = max(max|C| / 127, 2^-126) per
// block (1 for an all-zero block).  Everything runs in float32 in a fixed
// order (fmaf over the block's cells row by row, then over the kept
// coefficients in order) so that an independent implementation gives the
// same codes and values bit for bit.
//
// Sample layout: int8 codes [face][comp][block][K] padded to 16 bytes, then
// float32 scales [face][comp][block]; blocks row-major over (bv, bu).
#pragma once

#include "fdtd_internal.cuh"

namespace fdtd {

constexpr int kTapeBdct = 9;
constexpr int kBdctDefaultCoeffs = 10;   // the diagonals u + v <= 3

struct BdctLayout {
  int K;                 // coefficients kept per block
  int nbu[6], nbv[6];    // blocks per face along u and v
  int bstart[7];         // first block of each face (two components each)
  long long code_bytes;  // codes of one sample, padded to 16 bytes
  long long sample_bytes;
};

// Basis table: beta[i * 64 + y * 8 + x] = float(d_u[x] d_v[y]) for the i-th
// coefficient (u, v) in diagonal order, d_u[x] = c_u cos((2x + 1) u pi / 16),
// c_0 = sqrt(1/8), c_u = 1/2; computed in double on the host.
void bdct_basis_host(float* beta);
// (u, v) of the i-th coefficient in diagonal order.
void bdct_order_host(int i, int* u, int* v);
BdctLayout bdct_layout(const Faces& fc, int K);

// Upload the basis table to the device once per device (host-synchronous;
// call outside stream capture).
cudaError_t bdct_ensure_basis();
// The uploaded table of the current device, or NULL before its upload (no
// runtime call a stream capture forbids).
const float* bdct_basis_device();

// Value of cell t (y * 8 + x) of a block from its K codes and scale.
__device__ __forceinline__ float bdct_decode_cell(const signed char* __restrict__ codes, float s,
                                                  int K, int t, const float* __restrict__ beta) {
  float acc = 0.f;
  for (int i = 0; i < K; ++i)
    acc = __fmaf_rn((float)codes[i], __ldg(beta + i * 64 + t), acc);
  return __fmul_rn(acc, s);
}

// Value rr of face f restored from the samples of ip.
__device__ __forceinline__ float bdct_restored(const BdctLayout& bl, const FaceDesc& fd, int f,
                                               int rr, const unsigned char* __restrict__ tape,
                                               long long stride, const Interp& ip,
                                               const float* __restrict__ beta) {
  const int row = rr / fd.nu, u = rr - row * fd.nu;
  const int comp_t = row >= fd.nv, v = row - comp_t * fd.nv;
  const int bu = u >> 3, bv = v >> 3;
  const int b = bl.bstart[f] + comp_t * bl.nbu[f] * bl.nbv[f] + bv * bl.nbu[f] + bu;
  const int t = (v & 7) * 8 + (u & 7);
  const int fld = f & 1;  // 0: Ht on low faces, 1: E on high faces
  float val = 0.f;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int s = ip.slot[fld][m];
    if (s >= 0) {
      const unsigned char* smp = tape + (long long)s * stride;
      const float sc = __ldg(reinterpret_cast<const float*>(smp + bl.code_bytes) + b);
      const float x =
          bdct_decode_cell(reinterpret_cast<const signed char*>(smp) + (long long)b * bl.K, sc,
                           bl.K, t, beta);
      val = __fmaf_rn(ip.w[fld][m], x, val);
    }
  }
  return val;
}

cudaError_t launch_record_bdct(const float* FH, const float* FE, Geo g, const Faces& fc,
                               const BdctLayout& bl, void* tape_sample, cudaStream_t s);
cudaError_t launch_restore_seed_bdct(float* F, float* L, Geo g, const Faces& fc,
                                     const BdctLayout& bl, const void* tape, long long stride,
                                     const Interp& ip, const Det& det, const Det& det2,
                                     const double* seeds, cudaStream_t s);
cudaError_t launch_bdct_encode(const float* in, int nu, int nv, int K, signed char* codes,
                               float* scales, cudaStream_t s);
cudaError_t launch_bdct_decode(const signed char* codes, const float* scales, int nu, int nv,
                               int K, float* out, cudaStream_t s);

}  // namespace fdtd
