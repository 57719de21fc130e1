// z stage of one (kx, ky) column in registers, shared by the y/z kernels that
// hold a whole kx plane on chip (demag_quad.cu, demag_yz3.cu).  The Pz-point
// transform of the nz <= Pz/2 non-zero planes splits into even kz (a
// Pz/2-point FFT of x) and odd kz (a Pz/2-point FFT of x W_Pz^z); the inverse
// restricted to those planes is the even half plus W_Pz^(-z) times the odd
// half.  Entries of the tensor octant: six components innermost.
#pragma once

#include "common.cuh"
#include "regfft.cuh"

namespace mx {

// (a, b, c) <- N (a, b, c) for the symmetric 3x3 tensor N, complex vectors.
__device__ __forceinline__ void tensor_apply(float2& a, float2& b, float2& c, float nxx, float nyy, float nzz,
                                             float nxy, float nxz, float nyz) {
  const float2 mx = a, my = b, mz = c;
  auto row = [&](float u, float v, float w) {  // u mx + v my + w mz
    return __ffma2_rn(make_float2(w, w), mz, __ffma2_rn(make_float2(v, v), my, __fmul2_rn(make_float2(u, u), mx)));
  };
  a = row(nxx, nxy, nxz);
  b = row(nxy, nyy, nyz);
  c = row(nxz, nyz, nzz);
}

// The six components of octant entry kz of a column (tq: its entry at qz = 0,
// qzs floats per step of qz).
struct ZEntry {
  float2 t01, t23, t45;
};
__device__ __forceinline__ ZEntry z_entry(const float* __restrict__ tq, long qzs, int kz) {
  const float2* t = reinterpret_cast<const float2*>(tq + kz * qzs);
  return ZEntry{__ldg(t), __ldg(t + 1), __ldg(t + 2)};
}

// Octant entries the half spectrum of parity PAR needs: kz = 2 q + PAR <= P/2.
template <int P, int PAR> constexpr int z_entries() { return PAR ? (P + 2) / 4 : P / 4 + 1; }

// Tensor multiply of one column's half spectrum, kz parity PAR: y[.][q] holds
// kz = 2 q + PAR; kz and its mirror P - kz share one octant entry (the mirror
// with N_xz and N_yz negated).  entry(kz, q) gives the octant entry of
// kz = 2 q + PAR; sy = -1 where ky > Py/2 (N_xy and N_yz are odd in ky).
template <int P, int PAR, typename F>
__device__ __forceinline__ void z_multiply(float2 (&y)[3][P / 2], F entry, float sy) {
  constexpr int Q = P / 2;
#pragma unroll
  for (int q = 0; q < z_entries<P, PAR>(); ++q) {
    const int kz = 2 * q + PAR;
    const ZEntry t = entry(kz, q);
    const float nxy = sy * t.t23.y, nyz = sy * t.t45.y;
    tensor_apply(y[0][q], y[1][q], y[2][q], t.t01.x, t.t01.y, t.t23.x, nxy, t.t45.x, nyz);
    if (kz != 0 && kz != P / 2) {
      const int qm = Q - q - PAR;  // 2 qm + PAR = P - kz
      tensor_apply(y[0][qm], y[1][qm], y[2][qm], t.t01.x, t.t01.y, t.t23.x, nxy, -t.t45.x, -nyz);
    }
  }
}

// One column, kz parity p (uniform across the warp; a run-time value, so that
// the transforms' code is not duplicated): half-length forward transform of the
// nz planes of each component (times W_P^z first for odd kz), the tensor
// multiply and the inverse half transform (times W_P^-z after it for odd kz);
// y[c][n] is this parity's share of output plane n.  col: the column's element
// in line 0 of the plane; entry(kz, q) gives the octant entry of kz, the q-th
// of its parity.
template <int P, typename F>
__device__ __forceinline__ void z_column(const float2* col, int pitch, int nz, F entry, float sy, int p,
                                         float2 (&y)[3][P / 2]) {
  constexpr int Q = P / 2;
  constexpr int TS = 32 / P;  // W_P^n = c_w32[n TS]
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int n = 0; n < Q; ++n) y[c][n] = n < nz ? col[(c * nz + n) * pitch] : make_float2(0.f, 0.f);
  if (p) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int n = 1; n < Q; ++n) y[c][n] = cmul(y[c][n], c_w32[n * TS]);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) RegFft<Q, false>::run(y[c]);
  if (p)
    z_multiply<P, 1>(y, entry, sy);
  else
    z_multiply<P, 0>(y, entry, sy);
#pragma unroll
  for (int c = 0; c < 3; ++c) RegFft<Q, true>::run(y[c]);
  if (p) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int n = 1; n < Q; ++n) y[c][n] = cmul(y[c][n], cconj(c_w32[n * TS]));
  }
}

}  // namespace mx
