// y and z passes of the demag convolution on grids with few layers (Sec.
// II-B: zero-padded FFT convolution with the tensor spectrum): one block per T
// kx columns holds their planes [c][z][y] in shared memory, in place on the
// small-grid spectrum w1[c][z][y][kx], or (KM) from w1 to w2 on the kx-major
// spectra of the plane path.
//
// Forward y: the Py-point transform of a zero-padded column (inputs y < ny <=
// Py/2) splits into its even outputs, a Py/2-point FFT of x, and its odd
// outputs, a Py/2-point FFT of x W_Py^y; each half is a register line FFT of
// E x S points by S threads.  z stage: a thread takes one ky column's three
// components in registers (zcol.cuh), one kz parity where the block has the
// threads for both, else both in turn.  Inverse y is the mirror image: even +
// W_Py^-y odd.  The zero halves along y and z are never formed, and the block
// meets five barriers (seven with the split z stage), where the block-wide radix passes of yz_fused_kernel
// meet two per pass and transform the padding too.  The tensor octant is in
// plane_octant_index order (six components innermost), so a column's entry is
// three 8-byte loads and neighbouring columns are contiguous.
//
// Bound: the latency of that chain (load, two line FFTs, column, store) at two
// to four blocks per SM, and on large grids instruction issue (58 % of its slots at 640x160x4).
// Measured (one evaluation, kernel alone): 32x32x4 14.1 -> 3.9 us and 201x77x3 73.4
// -> 9 us against yz_fused_kernel; 640x160x4 107 -> 42 us (49 with divisions by
// run-time sizes in the load and store loops), 256x256x4 32 -> 16 us and 256x256x8
// 42 -> 35 us against the four-CTA plane kernel, whose cluster barriers and small
// shares of a plane cost more than they save where a plane fits one block (but for
// grids with at most one kx column to two SMs, quad_first in demag_plane.cu).
#include <math.h>

#include "common.cuh"
#include "fft.cuh"
#include "kernels.cuh"
#include "regfft.cuh"
#include "zcol.cuh"

namespace mx {

// (64 registers per thread, so two 512-thread blocks share an SM, where that spills
// at most a few words: 640x160x4 62 -> 52 us when measured)
template <int E, int S, int P, int T, int NT, bool KM>
__global__ void __launch_bounds__(NT, NT == 512 && E <= 16 && P <= 8 ? 2 : 1) yz3_kernel(const float2* win, float2* wout, Grid g, const float* __restrict__ nhk,
                                                 const float2* __restrict__ twH, const float2* __restrict__ twPy) {
  constexpr int LH = E * S;  // Py / 2
  constexpr int PITCH = LineFft<E, S>::kPitch;
  constexpr int Q = P / 2;
  constexpr int NTASK = 4 * LH * T;  // (column, kz parity) pairs of the z stage
  constexpr bool SPLIT = NTASK <= NT;
  static_assert(SPLIT || (NTASK / 2) % NT == 0 || NTASK / 2 <= NT, "z stage rounds");
  extern __shared__ __align__(16) float2 sm[];
  const int nz = g.nz, ny = g.ny, Hx = g.Hx;
  const int nlines = 3 * nz * T;        // line (c, z, t): even half then odd half, PITCH apart
  float2* twS = sm + 2 * nlines * PITCH;  // W_LH^(s k) at [k S + s]
  float2* twS2 = twS + LH;              // W_Py^y, y < LH
  float2* dummy = twS2 + LH;            // scratch line for idle thread groups
  const int kx0 = blockIdx.x * T;
  const int tid = threadIdx.x;
  // element (cz, y) of kx column t, element e of the block's load and store loops (LH, not
  // ny, values per line and KM with one column: no division by a run-time value)
  static_assert(!KM || T == 1, "kx-major blocks hold one column");
  auto wi = [&](int t, int y, int cz) {
    return KM ? ((long)kx0 * 3 * nz + cz) * ny + y : ((long)cz * ny + y) * Hx + kx0 + t;
  };
  auto et = [&](int e) { return e % T; };
  auto ey = [&](int e) { return (e / T) % LH; };
  auto ecz = [&](int e) { return e / (T * LH); };
  for (int q = tid; q < LH; q += NT) {
    twS[q] = __ldg(&twH[(q % S) * (q / S)]);
    twS2[q] = __ldg(&twPy[q]);
  }
  // z task q: column j of half h (ky = 2 j + h) of kx column t, kz parity par
  const int oyh = (g.Oy + 1) >> 1;
  const long qzs = 12L * oyh;
  struct Task {
    int t, h, j;
    float sy;
    const float* tq;
    bool ok;
  };
  auto task = [&](int q) {
    Task k;
    k.j = q % LH;
    k.h = (q / LH) & 1;
    k.t = (q / (2 * LH)) % T;
    const int ky = 2 * k.j + k.h;
    const bool fy = ky > LH;
    const int qy = fy ? 2 * LH - ky : ky;
    k.sy = fy ? -1.f : 1.f;
    k.ok = kx0 + k.t < Hx;
    k.tq = nhk + plane_octant_index(g, k.ok ? kx0 + k.t : 0, 0, 0, qy);
    return k;
  };
  // the split z stage's tensor entries: constants, so read while the
  // previous kernel may still run
  constexpr bool PRE = SPLIT && P <= 16;
  constexpr int NE = z_entries<P, 0>();
  ZEntry pre[PRE ? NE : 1];
  const int mypar = tid / (2 * LH * T);
  if (PRE && tid < NTASK) {
    const Task k = task(tid);
#pragma unroll
    for (int q = 0; q < NE; ++q) pre[q] = z_entry(k.tq, qzs, min(2 * q + mypar, P / 2));
  }
  pdl_wait_next();  // w1 is the previous kernel's
  __syncthreads();  // the twiddle tables
  {
    const int total = nlines * LH;
    constexpr int KB = 6;  // loads per thread in flight
    for (int e0 = tid; e0 < total; e0 += NT * KB) {
      float2 v[KB];
#pragma unroll
      for (int u = 0; u < KB; ++u) {
        const int e = e0 + u * NT;
        const int t = et(e), y = ey(e), cz = ecz(e);
        v[u] = (e < total && y < ny && kx0 + t < Hx) ? win[wi(t, y, cz)] : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < KB; ++u) {
        const int e = e0 + u * NT;
        if (e >= total) break;
        const int t = et(e), y = ey(e), cz = ecz(e);
        float2* L = sm + 2 * (cz * T + t) * PITCH;
        L[y] = v[u];
        L[PITCH + y] = cmul(v[u], twS2[y]);
      }
    }
  }
  __syncthreads();
  constexpr int LPR = NT / S;  // lines per round, S threads each
  for (int l0 = 0; l0 < 2 * nlines; l0 += LPR) {
    const int l = l0 + tid / S;
    // whole warps leave together; the idle groups of the last one share a scratch line's slots
    if (l0 + (tid & ~31) / S < 2 * nlines)
      line_fft<E, S, false, true, true>(l < 2 * nlines ? sm + l * PITCH : dummy, tid % S, twS);
  }
  __syncthreads();
  const int pitch = 2 * T * PITCH;  // from (c, z) to (c, z + 1)
  if (SPLIT) {
    float2 y[3][Q];
    float2* cp = sm;
    bool ok = false;
    if (tid < NTASK) {
      const Task k = task(tid);
      cp = sm + (2 * k.t + k.h) * PITCH + k.j;
      ok = k.ok;
      z_column<P>(cp, pitch, nz, [&](int kz, int q) { return PRE ? pre[q] : z_entry(k.tq, qzs, kz); }, k.sy, mypar, y);
    }
    __syncthreads();  // both parities have read the columns
    if (ok && mypar == 0) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int n = 0; n < Q; ++n)
          if (n < nz) cp[(c * nz + n) * pitch] = y[c][n];
    }
    __syncthreads();
    if (ok && mypar == 1) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int n = 0; n < Q; ++n)
          if (n < nz) cp[(c * nz + n) * pitch] = cadd(cp[(c * nz + n) * pitch], y[c][n]);
    }
  } else {
    for (int q = tid; q < 2 * LH * T; q += NT) {
      const Task k = task(q);
      float2* cp = sm + (2 * k.t + k.h) * PITCH + k.j;
      float2 a[3][Q], b[3][Q];
      auto entry = [&](int kz, int) { return z_entry(k.tq, qzs, kz); };
      z_column<P>(cp, pitch, nz, entry, k.sy, 0, a);
      z_column<P>(cp, pitch, nz, entry, k.sy, 1, b);
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int n = 0; n < Q; ++n)
          if (n < nz) cp[(c * nz + n) * pitch] = cadd(a[c][n], b[c][n]);
    }
  }
  __syncthreads();
  for (int l0 = 0; l0 < 2 * nlines; l0 += LPR) {
    const int l = l0 + tid / S;
    if (l0 + (tid & ~31) / S < 2 * nlines)
      line_fft<E, S, true, true, true>(l < 2 * nlines ? sm + l * PITCH : dummy, tid % S, twS);
  }
  __syncthreads();
  const int total = nlines * LH;
  for (int e = tid; e < total; e += NT) {
    const int t = et(e), y = ey(e), cz = ecz(e);
    if (y >= ny || kx0 + t >= Hx) continue;
    const float2* L = sm + 2 * (cz * T + t) * PITCH;
    wout[wi(t, y, cz)] = cadd(L[y], cmul(L[PITCH + y], cconj(twS2[y])));
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
// Two blocks per SM.  Beyond that the four-CTA kernel is as fast or faster:
// with one block per SM 512x512x8 takes 134 us against 119, 512x512x4 (117 KB)
// 69 against 72.
constexpr size_t kYz3MaxSmem = 113 * 1024;

template <int E, int S, int P, int T, bool KM>
static mx_status yz3_run(mx_ctx* ctx, cudaStream_t st, bool setup) {
  constexpr int LH = E * S;
  constexpr int WANT = 4 * LH * T;
  constexpr int NT = WANT < 128 ? 128 : (WANT > 512 ? 512 : WANT);
  const size_t sm = sizeof(float2) * ((6 * (size_t)ctx->g.nz * T + 1) * LineFft<E, S>::kPitch + 2 * LH);
  if (setup) {
    if (sm > kYz3MaxSmem) return MX_ERR_UNSUPPORTED;
    MX_CUDA_TRY(cudaFuncSetAttribute(yz3_kernel<E, S, P, T, NT, KM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kYz3MaxSmem));
    return MX_OK;
  }
  launch_pdl(yz3_kernel<E, S, P, T, NT, KM>, dim3((ctx->g.Hx + T - 1) / T), dim3(NT), sm, st, ctx->w1,
             KM ? ctx->w2 : ctx->w1, ctx->g, ctx->nhat, ctx->tw_yh, ctx->tw_y);
  return launch_check("yz3_kernel");
}

template <int E, int S, int P>
static mx_status yz3_t(mx_ctx* ctx, bool km, cudaStream_t st, bool setup) {
  if (km) return yz3_run<E, S, P, 1, true>(ctx, st, setup);
  // one kx column per block, two where that still leaves two blocks per SM
  // (a pair of columns shares its 32-byte sectors)
  return ctx->g.Hx <= 2 * 2 * 152 ? yz3_run<E, S, P, 1, false>(ctx, st, setup)
                                  : yz3_run<E, S, P, 2, false>(ctx, st, setup);
}

template <int E, int S, bool P16, bool P32>
static mx_status yz3_pz(mx_ctx* ctx, bool km, cudaStream_t st, bool setup) {
  switch (ctx->g.Pz) {
    case 4: return yz3_t<E, S, 4>(ctx, km, st, setup);
    case 8: return yz3_t<E, S, 8>(ctx, km, st, setup);
    case 16:
      if constexpr (P16) return yz3_t<E, S, 16>(ctx, km, st, setup);
      return MX_ERR_UNSUPPORTED;
    case 32:
      if constexpr (P32) return yz3_t<E, S, 32>(ctx, km, st, setup);
      return MX_ERR_UNSUPPORTED;
    default: return MX_ERR_UNSUPPORTED;
  }
}

mx_status yz3_pass(mx_ctx* ctx, bool km, cudaStream_t st, bool setup) {
  if (setup) MX_TRY(upload_w32());
  switch (ctx->g.Py / 2) {
    case 512: return yz3_pz<32, 16, false, false>(ctx, km, st, setup);  // (five layers take 143 KB)
    case 256: return yz3_pz<16, 16, true, false>(ctx, km, st, setup);
    case 128: return yz3_pz<16, 8, true, false>(ctx, km, st, setup);
    case 64: return yz3_pz<8, 8, true, true>(ctx, km, st, setup);
    case 32: return yz3_pz<8, 4, true, true>(ctx, km, st, setup);
    case 16: return yz3_pz<4, 4, true, true>(ctx, km, st, setup);
    default: return MX_ERR_UNSUPPORTED;
  }
}

}  // namespace mx
