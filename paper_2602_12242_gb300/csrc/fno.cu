// Fourier-neural-operator demag surrogate of a film (Sec. II-D): lifting
// 3 -> 32 channels, four spectral layers keeping K modes per dimension, a
// 32 -> 128 -> 3 projection; forward, SmoothL1 loss, backward and Adam.
//
//   v_0     = P x + p                               x: normalised m
//   v_{l+1} = act_l(K_l v_l + W_l v_l + w_l)        GELU for l < 3, identity for l = 3
//   K_l v   = irfft2(R_l . rfft2(v) on the kept modes)
//             kept: ky in [0, K) u [H-K, H), kx in [0, K);  Y_o = sum_i X_i R_l[mode][i][o]
//   y       = Q2 gelu(Q1 v_4 + q1) + q2
// H = ny (rows), W = nx (columns).  Activations are FP32 channel planes per row,
// v[b y][channel][x] with rows of Wp = W rounded up to 4 columns (the padding
// is kept at zero), so every pass reads and writes contiguous x.  Only 2K x K of
// the H x (W/2+1) Fourier modes are used, so the transforms are truncated DFTs,
// not FFTs.  Passes of the network:
//   row pass (fno_row)     the inverse row DFT, the pointwise W_l v + w_l and the
//                          activation of a row as one product of length 32 + 2K,
//                          then the row DFT of the result for the next layer
//   column pass (fno_mid)  per (kx, sample): forward column DFT, channel mix,
//                          inverse column DFT, on a cluster of eight CTAs that
//                          take an eighth of the modes and of the rows each
//   projection             per tile of 32 cells; in training with the loss, its
//                          gradient and both weight gradients in one kernel, so
//                          the 128 hidden values per cell never leave the SM
// so a field takes 10 launches.
//
// Backward.  With g = dL/d(K v) and X_g its truncated rfft2, the filter
// gradient is dR[mode][i][o] = c_kx / (H W) * sum_b conj(X[b][i]) X_g[b][o]
// (c_0 = 1, c_kx = 2: the half spectrum stands for its mirror) and the input
// gradient is the same spectral convolution of g with the conjugate-transposed
// filters R'[mode][o][i] = conj(R[mode][i][o]) (so every pass is reused).
// Pointwise weight gradients are sums over cells of outer products.
#include <math.h>

#include <string>
#include <vector>

#include "cluster.cuh"
#include "common.cuh"
#include "kernels.cuh"

namespace mx {

constexpr int kFC = 32;    // channel width
constexpr int kFH = 128;   // projection hidden width
constexpr int kFL = 4;     // spectral layers
constexpr int kFMaxK = 16; // largest K
constexpr int kFMaxN = 1024;

__device__ __forceinline__ float fgelu(float y) { return 0.5f * y * (1.f + erff(y * 0.70710678118654752f)); }
__device__ __forceinline__ float fgelu_grad(float y) {
  return 0.5f * (1.f + erff(y * 0.70710678118654752f)) + y * 0.39894228040143268f * expf(-0.5f * y * y);
}

// Shared-memory pitch of a row of Wp floats: 4 modulo 32, so eight channels at
// one x, read as float4, meet no bank twice.
__host__ __device__ __forceinline__ int fno_pitch(int Wp) { return (Wp + 31) / 32 * 32 + 4; }

__device__ __forceinline__ float4 f4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ldg4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float dot4(float4 a, float4 b, float s) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s))));
}
// acc[i][j] += a[i] b[j] over 4 x 4 values
__device__ __forceinline__ void outer4(float (&acc)[4][4], float4 a, float4 b) {
  const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
}
// the same over 8 x 8 values, each operand two float4
__device__ __forceinline__ void outer8(float (&acc)[8][8], float4 a0, float4 a1, float4 b0, float4 b1) {
  const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
  const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
}

// Sums v[0..N) over the 2^BITS lanes that differ in lane bits FIRST .. and
// leaves each of them N / 2^BITS of the totals: entries q = idx + 2^BITS k, k =
// 0, 1, .., of the lane with those bits = idx, in v[k].
template <int N, int BITS, int FIRST> __device__ __forceinline__ void reduce_scatter(float* v, int lane) {
  if constexpr (BITS > 0) {
    // the lane with the lowest of its bits set keeps the odd entries
    const int bit = 1 << FIRST;
    const bool hi = lane & bit;
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      const float keep = hi ? v[2 * k + 1] : v[2 * k], give = hi ? v[2 * k] : v[2 * k + 1];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
    }
    reduce_scatter<N / 2, BITS - 1, FIRST + 1>(v, lane);
  }
}

// Row DFT of the channel planes vs[c][x] (pitch P) of one row: A[kx][c] =
// sum_x vs[c][x] e^{-2 pi i kx x / W}.  tw[2 kx][x], tw[2 kx + 1][x] (pitch tp):
// cos and -sin, zero in the padding.  Eight lanes share a tile of 8 twiddle rows
// x 8 channels (TWS: the twiddle rows are in shared memory), a share of the cells each (4 FMA per float loaded, which is what
// the load path needs to keep up with the FMA pipe), and reduce it by shuffles.
template <bool TWS>
__device__ __forceinline__ void fno_row_dft(const float* vs, int P, int Wp, int K, const float* tw, int tp,
                                            float2* __restrict__ A) {
  constexpr int LB = 3, SP = 1 << LB, TPW = 32 / SP;  // lanes per tile, tiles per warp
  const int lane = threadIdx.x & 31, sp = lane & (SP - 1);
  const int ntile = (2 * K + 7) / 8 * 4, n4 = Wp / 4;
  for (int t0 = threadIdx.x / 32 * TPW; t0 < ntile; t0 += blockDim.x / 32 * TPW) {
    const int tile = t0 + (lane >> LB);  // (ntile is a multiple of 4)
    const int m0 = tile / 4 * 8, c0 = tile % 4 * 8;
    float acc[64];
#pragma unroll
    for (int q = 0; q < 64; ++q) acc[q] = 0.f;
    const float* t = tw + (long)m0 * tp;
    const int left = 2 * K - 1 - m0;  // rows beyond 2K repeat the last one and are dropped
    for (int x4 = sp; x4 < n4; x4 += SP) {
      float4 b[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) b[j] = f4(vs + (c0 + j) * P + 4 * x4);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 a = TWS ? f4(t + min(i, left) * tp + 4 * x4) : ldg4(t + (long)min(i, left) * tp + 4 * x4);
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i * 8 + j] = dot4(a, b[j], acc[i * 8 + j]);
      }
    }
    reduce_scatter<64, LB, 0>(acc, lane);  // lane sp: entries q = SP k + sp
#pragma unroll
    for (int k = 0; k < 64 / SP; ++k) {
      const int q = SP * k + sp, m = m0 + q / 8, c = c0 + q % 8;
      if (m < 2 * K) (reinterpret_cast<float*>(A + m / 2 * kFC + c))[m & 1] = acc[k];
    }
  }
}

// Element q = threadIdx.x, + blockDim.x, ... of rows of n: its row and place, without a
// division per element.
struct RowWalk {
  int r, c, dr, dc, n;
  __device__ __forceinline__ explicit RowWalk(int n) : n(n) {
    r = threadIdx.x / n;
    c = threadIdx.x - r * n;
    dr = blockDim.x / n;
    dc = blockDim.x - dr * n;
  }
  __device__ __forceinline__ void next() {
    r += dr;
    c += dc;
    if (c >= n) {
      c -= n;
      ++r;
    }
  }
};

// The twiddle rows into shared memory (pitch P): constants, so before the
// dependency wait, which hides their latency where a launch has few blocks.
__device__ __forceinline__ void fno_stage_tw(float* dst, const float* __restrict__ tw, int Wp, int P, int K) {
  for (RowWalk q(Wp / 4); q.r < 2 * K; q.next())
    *reinterpret_cast<float4*>(dst + q.r * P + q.c * 4) = ldg4(tw + q.r * Wp + q.c * 4);
}

// 16-byte asynchronous copies of a row's planes into shared memory, one group
__device__ __forceinline__ void fno_copy_row(float* vs, const float* v, int Wp, int P) {
  for (RowWalk q(Wp / 4); q.r < kFC; q.next()) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(vs + q.r * P + q.c * 4);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(v + q.r * Wp + q.c * 4) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// LIFT: v0[c][x] = p[c] + sum_k P[c][k] xn[k] of a row, xn = (m - mean) / std,
// stored, and its row DFT.  Otherwise the row DFT of the stored row v.
template <bool LIFT, bool SMALL>
__global__ void __launch_bounds__(SMALL ? 384 : 128)
    fno_first_kernel(const float4* m, float3 mean, float3 inv_std, const float* Pw,
                     const float* pb, float* __restrict__ v, float2* __restrict__ A, int W, int Wp, int K,
                     const float* __restrict__ tw) {
  extern __shared__ __align__(16) float fsm[];
  const int P = fno_pitch(Wp);
  float *vs = fsm, *ts = fsm + kFC * P;
  const long r = blockIdx.x;
  float* row = v + r * kFC * Wp;
  if (SMALL) fno_stage_tw(ts, tw, Wp, P, K);
  pdl_wait_next();
  if (LIFT) {
    // a thread takes one cell and eight channels
    for (int q = threadIdx.x; q < Wp * 4; q += blockDim.x) {
      const int x = q % Wp, c0 = q / Wp * 8;
      float nx = 0.f, ny = 0.f, nz = 0.f;
      const bool in = x < W;
      if (in) {
        const float4 a = m[r * W + x];
        nx = (a.x - mean.x) * inv_std.x;
        ny = (a.y - mean.y) * inv_std.y;
        nz = (a.z - mean.z) * inv_std.z;
      }
#pragma unroll
      for (int c = c0; c < c0 + 8; ++c) {
        const float o = in ? pb[c] + Pw[c * 3] * nx + Pw[c * 3 + 1] * ny + Pw[c * 3 + 2] * nz : 0.f;
        vs[c * P + x] = o;
        row[(long)c * Wp + x] = o;
      }
    }
  } else {
    fno_copy_row(vs, row, Wp, P);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  __syncthreads();
  fno_row_dft<SMALL>(vs, P, Wp, K, SMALL ? ts : tw, SMALL ? P : Wp, A + r * K * kFC);
}

// ---------------------------------------------------------------------------
// Column pass of one (kx, sample) on a cluster of eight CTAs.  CTA q takes modes
// m in [q MM, (q + 1) MM) of the 2K kept rows (ky = m, or H - 2K + m for m >=
// K): X[m][c] = sum_y A[y][c] e^{-2 pi i ky y / H} (kept in X when given), the mix
// Y[m][o] = sum_i X[m][i] F[i][o] with F = R[m] (ADJ: the conjugate transpose),
// then, with every CTA's Y in shared memory, rows y in [q HH, (q + 1) HH) of
// A[y][o] = sum_m Y[m][o] e^{+2 pi i ky y / H}, in place (the cluster barrier
// orders every read of A before the writes).  Sums are split over the warps
// that a mode or row leaves over.  twy[y][m] = e^{-2 pi i ky y / H}.
// Bound: latency of the three short sums; one launch instead of three, and the
// filters are read ahead of the dependency wait.
// ---------------------------------------------------------------------------
constexpr int kMidCl = 8, kMidWarps = 12, kMidChunk = 64, kMidTi = 512;
constexpr int kMidBatch = 5;  // samples from which the batch kernels below are taken

// Shares (warps) that a mode's sums, and a row's, are split over.
__host__ __device__ __forceinline__ int fno_mid_shares(int K) {
  return kMidWarps / ((2 * K + kMidCl - 1) / kMidCl);
}
__host__ __device__ __forceinline__ int fno_mid_row_shares(int H) {
  const int hh = (H + kMidCl - 1) / kMidCl;
  return hh <= kMidWarps / 2 ? kMidWarps / hh : 1;
}

struct FnoMidSmem {
  float2 col[kMidChunk][kFC];
  float2 red[kMidWarps][kFC];
  float2 X[2 * kFMaxK / kMidCl][kFC];
  float2 Y[2 * kFMaxK][kFC];
  float2 F[2 * kFMaxK / kMidCl][kFC][kFC + 1];
  float2 tf[kMidChunk][2 * kFMaxK / kMidCl];  // forward twiddles of a chunk of rows
  float2 ti[kMidTi];                          // inverse twiddles of this CTA's rows, where they fit
};

template <bool ADJ>
__global__ void __cluster_dims__(kMidCl, 1, 1) __launch_bounds__(kMidWarps * 32)
    fno_mid_kernel(float2* A, float2* __restrict__ X, const float* __restrict__ R, int B, int H, int K,
                   const float2* __restrict__ twy) {
  extern __shared__ __align__(16) unsigned char midraw[];
  FnoMidSmem& s = *reinterpret_cast<FnoMidSmem*>(midraw);
  const int rank = (int)cluster_rank();
  const int kx = (blockIdx.x / kMidCl) % K, b = blockIdx.x / (kMidCl * K);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int M2 = 2 * K, MM = (M2 + kMidCl - 1) / kMidCl;
  const int m0 = rank * MM, nm = max(0, min(MM, M2 - m0));
  // this CTA's filters (parameters, last written before the kernel before this one)
  for (int q = threadIdx.x; q < nm * kFC * kFC; q += blockDim.x) {
    const int j = q / (kFC * kFC), i = (q / kFC) % kFC, o = q % kFC;
    s.F[j][i][o] = __ldg(reinterpret_cast<const float2*>(R) + ((long)(m0 + j) * K + kx) * kFC * kFC + i * kFC + o);
  }
  auto stage_fwd = [&](int y0) {
    for (int q = threadIdx.x; q < min(kMidChunk, H - y0) * nm; q += blockDim.x)
      s.tf[q / nm][q % nm] = __ldg(&twy[(long)(y0 + q / nm) * M2 + m0 + q % nm]);
  };
  stage_fwd(0);
  const int HH = (H + kMidCl - 1) / kMidCl;
  const int yb = rank * HH, ye = min(H, yb + HH);
  const bool ti = HH * M2 <= kMidTi;
  if (ti)
    for (int q = threadIdx.x; q < (ye - yb) * M2; q += blockDim.x) s.ti[q] = __ldg(&twy[(long)yb * M2 + q]);
  pdl_wait_next();
  // warp -> (mode of this CTA, share of the sum)
  const int ns = fno_mid_shares(K), mj = warp % MM, sp = warp / MM;
  const bool sums = sp < ns && mj < nm;
  float2* col0 = A + ((long)b * H * K + kx) * kFC;
  const long ys = (long)K * kFC;
  float re = 0.f, im = 0.f;
  for (int y0 = 0; y0 < H; y0 += kMidChunk) {
    const int ny = min(kMidChunk, H - y0);
    if (y0) {
      __syncthreads();
      stage_fwd(y0);
    }
    for (int q = threadIdx.x; q < ny * kFC; q += blockDim.x)
      s.col[q / kFC][q % kFC] = col0[(long)(y0 + q / kFC) * ys + q % kFC];
    __syncthreads();
    if (sums) {
#pragma unroll 4
      for (int y = sp; y < ny; y += ns) {
        const float2 a = s.col[y][lane];
        const float2 w = s.tf[y][mj];
        re = fmaf(a.x, w.x, fmaf(-a.y, w.y, re));
        im = fmaf(a.x, w.y, fmaf(a.y, w.x, im));
      }
    }
  }
  s.red[warp][lane] = make_float2(re, im);
  __syncthreads();
  if (warp < nm) {  // (MM <= 4 < the number of warps)
    float2 t = s.red[warp][lane];
    for (int q = 1; q < ns; ++q) t = cadd(t, s.red[warp + q * MM][lane]);
    s.X[warp][lane] = t;
    if (X) X[(((long)(m0 + warp) * K + kx) * B + b) * kFC + lane] = t;
  }
  __syncthreads();
  re = im = 0.f;
  if (sums) {
    for (int i = sp; i < kFC; i += ns) {
      const float2 x = s.X[mj][i];
      float2 f = ADJ ? s.F[mj][lane][i] : s.F[mj][i][lane];
      if (ADJ) f.y = -f.y;
      re = fmaf(x.x, f.x, fmaf(-x.y, f.y, re));
      im = fmaf(x.x, f.y, fmaf(x.y, f.x, im));
    }
  }
  s.red[warp][lane] = make_float2(re, im);
  __syncthreads();
  // Y of this CTA's modes into every CTA of the cluster
  cluster_arrive_relaxed();
  for (int q = threadIdx.x; q < nm * kFC; q += blockDim.x) {
    const int j = q / kFC, o = q % kFC;
    float2 t = s.red[j][o];
    for (int u = 1; u < ns; ++u) t = cadd(t, s.red[j + u * MM][o]);
    s.X[j][o] = t;
  }
  __syncthreads();
  cluster_wait();  // every CTA has started
  for (int q = threadIdx.x; q < nm * kFC * kMidCl; q += blockDim.x) {
    const int dst = q / (nm * kFC), e = q % (nm * kFC);
    float2* y = const_cast<float2*>(cluster_map(&s.Y[m0][0], (unsigned)dst));
    y[e] = s.X[e / kFC][e % kFC];
  }
  cluster_sync_all();
  // inverse: warp -> (row, share of the modes)
  const int nsm = fno_mid_row_shares(H);  // shares per row
  const int rw = nsm > 1 ? HH : kMidWarps;                   // rows in flight
  const int sh = warp / rw;
  for (int y0 = yb; y0 < ye; y0 += rw) {
    const int y = y0 + warp % rw;
    re = im = 0.f;
    if (sh < nsm && y < ye) {
      const float2* w = ti ? s.ti + (y - yb) * M2 : twy + (long)y * M2;
#pragma unroll 4
      for (int m = sh; m < M2; m += nsm) {
        const float2 t = w[m], a = s.Y[m][lane];
        re = fmaf(a.x, t.x, fmaf(a.y, t.y, re));
        im = fmaf(a.y, t.x, fmaf(-a.x, t.y, im));
      }
    }
    if (nsm > 1) {  // (then one round)
      s.red[warp][lane] = make_float2(re, im);
      __syncthreads();
      if (sh > 0) continue;
      for (int q = 1; q < nsm; ++q) {
        re += s.red[warp + q * rw][lane].x;
        im += s.red[warp + q * rw][lane].y;
      }
    }
    if (y < ye) col0[(long)y * ys + lane] = make_float2(re, im);
  }
}

// Batches: the column pass as three kernels, each filter read once for the whole
// batch (the cluster kernel reads all filters per sample: a forward pass of four
// fields of 160 x 40 takes 115 us with it and 138 with these, one of six 151
// against 141, one of 32 506 against 344).  Every sum runs in the cluster
// kernel's order (its shares one after the other), so a sample's output does not
// depend on the size of its batch.
//
// Forward column DFT: thread (c) of column (b, kx) sums kMidM modes over all rows,
// eight rows' values in flight; the block's twiddles in shared memory by chunks of rows.
constexpr int kMidM = 8, kMidY = 8;
__global__ void __launch_bounds__(128) fno_dft_y_kernel(const float2* A, float2* __restrict__ X, int B,
                                                        int H, int K, const float2* __restrict__ twy) {
  __shared__ __align__(16) float2 ts[kMidChunk][kMidM];
  const int c = threadIdx.x & 31;
  const long col = (long)blockIdx.x * 4 + (threadIdx.x >> 5);  // b K + kx
  const int m0 = blockIdx.y * kMidM, M2 = 2 * K, ns = fno_mid_shares(K);
  const bool ok = col < (long)B * K;
  const int b = ok ? (int)(col / K) : 0, kx = (int)(col % K);
  const float2* a = A + ((long)b * H * K + kx) * kFC + c;
  float2 sum[kMidM], acc[kMidM];
  for (int sp = 0; sp < ns; ++sp) {
#pragma unroll
    for (int q = 0; q < kMidM; ++q) acc[q] = make_float2(0.f, 0.f);
    for (int yc = 0; yc < H; yc += kMidChunk) {
      const int ny = min(kMidChunk, H - yc);
      if (sp == 0 || H > kMidChunk) {
        __syncthreads();
        for (int q = threadIdx.x; q < ny * kMidM; q += 128)
          ts[q / kMidM][q % kMidM] = __ldg(&twy[(long)(yc + q / kMidM) * M2 + min(m0 + q % kMidM, M2 - 1)]);
        if (sp == 0 && yc == 0) pdl_wait_next();
        __syncthreads();
      }
      for (int y0 = sp; y0 < ny; y0 += 8 * ns) {
        float2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          v[u] = ok && y0 + u * ns < ny ? a[(long)(yc + y0 + u * ns) * K * kFC] : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (y0 + u * ns >= ny) break;
          const float4* t4 = reinterpret_cast<const float4*>(ts[y0 + u * ns]);
#pragma unroll
          for (int q = 0; q < kMidM / 2; ++q) {
            const float4 t = t4[q];
            float2 &x = acc[2 * q], &y = acc[2 * q + 1];
            x = make_float2(fmaf(v[u].x, t.x, fmaf(-v[u].y, t.y, x.x)), fmaf(v[u].x, t.y, fmaf(v[u].y, t.x, x.y)));
            y = make_float2(fmaf(v[u].x, t.z, fmaf(-v[u].y, t.w, y.x)), fmaf(v[u].x, t.w, fmaf(v[u].y, t.z, y.y)));
          }
        }
      }
    }
#pragma unroll
    for (int q = 0; q < kMidM; ++q) sum[q] = sp ? cadd(sum[q], acc[q]) : acc[q];
  }
  if (!ok) return;
#pragma unroll
  for (int q = 0; q < kMidM; ++q)
    if (m0 + q < M2) X[(((long)(m0 + q) * K + kx) * B + b) * kFC + c] = sum[q];
}

// Channel mix per kept mode over the batch: Y[mode][b][o] = sum_i X[mode][b][i] F[i][o]
// with F = R[mode] or (ADJ) its conjugate transpose; a thread takes one o of kMixB samples.
constexpr int kMixB = 4;
template <bool ADJ>
__global__ void __launch_bounds__(256) fno_mix_kernel(const float2* X, float2* __restrict__ Y,
                                                       const float* __restrict__ R, int B, int K) {
  __shared__ float2 F[kFC][kFC + 1];
  __shared__ __align__(16) float2 xs[8 * kMixB][kFC];
  const int mode = blockIdx.x, ns = fno_mid_shares(K);
  const float2* Rm = (const float2*)(R + (long)mode * kFC * kFC * 2);
  for (int q = threadIdx.x; q < kFC * kFC; q += 256) {
    const int i = q / kFC, o = q % kFC;  // R[mode][i][o]
    const float2 r = __ldg(&Rm[q]);
    if (ADJ)
      F[o][i] = make_float2(r.x, -r.y);
    else
      F[i][o] = r;
  }
  pdl_wait_next();
  const int o = threadIdx.x & 31, w = threadIdx.x >> 5;
  const float2* Xm = X + (long)mode * B * kFC;
  float2* Ym = Y + (long)mode * B * kFC;
  for (int b0 = 0; b0 < B; b0 += 8 * kMixB) {
    __syncthreads();
    for (int q = threadIdx.x; q < 8 * kMixB * kFC; q += 256)
      (&xs[0][0])[q] = b0 + q / kFC < B ? Xm[(long)b0 * kFC + q] : make_float2(0.f, 0.f);
    __syncthreads();
    float2 sum[kMixB], acc[kMixB];
    for (int sp = 0; sp < ns; ++sp) {
#pragma unroll
      for (int q = 0; q < kMixB; ++q) acc[q] = make_float2(0.f, 0.f);
#pragma unroll 4
      for (int i = sp; i < kFC; i += ns) {
        const float2 f = F[i][o];
#pragma unroll
        for (int q = 0; q < kMixB; ++q) {
          const float2 x = xs[w * kMixB + q][i];
          acc[q] = make_float2(fmaf(x.x, f.x, fmaf(-x.y, f.y, acc[q].x)), fmaf(x.x, f.y, fmaf(x.y, f.x, acc[q].y)));
        }
      }
#pragma unroll
      for (int q = 0; q < kMixB; ++q) sum[q] = sp ? cadd(sum[q], acc[q]) : acc[q];
    }
#pragma unroll
    for (int q = 0; q < kMixB; ++q) {
      const int b = b0 + w * kMixB + q;
      if (b < B) Ym[(long)b * kFC + o] = sum[q];
    }
  }
}

// Inverse column DFT: thread (o) of column (b, kx) forms kMidY rows from all modes.
__global__ void __launch_bounds__(128) fno_idft_y_kernel(const float2* Y, float2* __restrict__ A, int B,
                                                         int H, int K, const float2* __restrict__ twy) {
  __shared__ __align__(16) float2 ts[2 * kFMaxK][kMidY];
  const int o = threadIdx.x & 31;
  const long col = (long)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int y0 = blockIdx.y * kMidY, M2 = 2 * K, ns = fno_mid_row_shares(H);
  const bool ok = col < (long)B * K;
  const int b = ok ? (int)(col / K) : 0, kx = (int)(col % K);
  for (int q = threadIdx.x; q < M2 * kMidY; q += 128)
    ts[q % M2][q / M2] = __ldg(&twy[(long)min(y0 + q / M2, H - 1) * M2 + q % M2]);
  pdl_wait_next();
  __syncthreads();
  if (!ok) return;
  const float2* v = Y + ((long)kx * B + b) * kFC + o;
  float2 sum[kMidY], acc[kMidY];
  for (int sp = 0; sp < ns; ++sp) {
#pragma unroll
    for (int q = 0; q < kMidY; ++q) acc[q] = make_float2(0.f, 0.f);
    for (int mc = sp; mc < M2; mc += 8 * ns) {
      float2 a[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        a[u] = mc + u * ns < M2 ? v[(long)(mc + u * ns) * K * B * kFC] : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (mc + u * ns >= M2) break;
        const float4* t4 = reinterpret_cast<const float4*>(ts[mc + u * ns]);
#pragma unroll
        for (int q = 0; q < kMidY / 2; ++q) {
          const float4 t = t4[q];
          float2 &x = acc[2 * q], &y = acc[2 * q + 1];
          x = make_float2(fmaf(a[u].x, t.x, fmaf(a[u].y, t.y, x.x)), fmaf(a[u].y, t.x, fmaf(-a[u].x, t.y, x.y)));
          y = make_float2(fmaf(a[u].x, t.z, fmaf(a[u].y, t.w, y.x)), fmaf(a[u].y, t.z, fmaf(-a[u].x, t.w, y.y)));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < kMidY; ++q) sum[q] = sp ? cadd(sum[q], acc[q]) : acc[q];
  }
#pragma unroll
  for (int q = 0; q < kMidY; ++q)
    if (y0 + q < H) A[(((long)b * H + y0 + q) * K + kx) * kFC + o] = sum[q];
}

// ---------------------------------------------------------------------------
// Row pass.  For output channel o of cell x, with the inverse row DFT
//   s = (1/(H W)) [Re A[0][o] + 2 sum_{kx>=1} Re(A[kx][o] e^{+2 pi i kx x / W})]:
// FWD: u = s + sum_i Wl[o][i] vin[i][x] + wl[o];  pre = u (if kept); out = act(u)
// BWD: u = s + sum_i Wl[i][o] vin[i][x]  (vin = dL/du of this layer, o = input channel);
//      out = u gelu'(gpre[o][x]) when gpre is given (the layer below's pre-activation, kept
//      from the forward pass, so that it may be read ahead of the wait: 60 us a launch for
//      32 fields of 160 x 40, 66 otherwise)
// and, with next, the row DFT of out into A (in place: the block owns its row).
// u is one product over 32 + 2K terms: a thread holds T cells x T channels and
// reads T floats of cells (vin, or the twiddle rows) and T of channels per T^2
// FMA.  T = 8 for batches: a float4 load occupies the load path for four cycles
// whatever its addresses, so 4 x 4 tiles are bound by it at half the FMA rate.
// T = 4 with the twiddle rows in shared memory where there are few rows, for the
// shorter chain.  Bound: for batches FP32 issue (a pass of 32 fields of 160 x 40
// is 34.9 M warp instructions at 63 % of the issue slots, 16.4 M of them the FMAs of
// the products and of the row DFT); 51 us in the chain of a training step where the
// lane-per-channel kernel took 85.  Not kept: persistent
// blocks with two row buffers (97 us at 8 warps per SM, 71 with one buffer).
// ---------------------------------------------------------------------------
template <bool BWD, int T>
__global__ void __launch_bounds__(T == 8 ? 256 : 512, T == 8 ? 2 : 1)
    fno_row_kernel(float2* A, const float* vin, const float* __restrict__ Wl,
                   const float* __restrict__ wl, float* __restrict__ pre, float* __restrict__ out,
                   const float* __restrict__ gpre, int W, int Wp, int K, float scale, int gelu_out, int next,
                   const float* __restrict__ tw) {
  constexpr bool TWS = T == 4;
  constexpr int OG = kFC / T, H4 = T / 4;  // channel groups; float4 per operand
  extern __shared__ __align__(16) float fsm[];
  const int P = fno_pitch(Wp), tid = threadIdx.x, NT = blockDim.x;
  float* Bs = fsm;                           // [32 + 2K][32]: W, then the scaled A
  float* vs = fsm + (kFC + 2 * K) * kFC;     // [32][P]
  float* ts = vs + kFC * P;                  // [2K][P] (TWS)
  const long r = blockIdx.x, base = r * kFC * Wp;
  for (int q = tid; q < kFC * kFC; q += NT) {
    const int j = q / kFC, l = q % kFC;
    Bs[BWD ? q : l * kFC + j] = __ldg(&Wl[q]);  // Bs[j][l] multiplies vin[j]
  }
  if (TWS) fno_stage_tw(ts, tw, Wp, P, K);
  const int og = tid % OG, n4 = Wp / 4, span = (n4 + H4 - 1) / H4;  // 4-cell groups per operand half
  // channels 4 og .. + 3 (and 16 + 4 og .. + 3); cells 4 xi .. + 3 (and 4 (xi + span) .. + 3)
  float bias[T];
#pragma unroll
  for (int j = 0; j < T; ++j) bias[j] = (!BWD && wl) ? __ldg(&wl[j / 4 * 16 + 4 * og + j % 4]) : 0.f;
  pdl_wait_next();
  fno_copy_row(vs, vin + base, Wp, P);
  float2* Ar = A + r * K * kFC;
  for (int q = tid; q < K * kFC; q += NT) {
    const float2 a = Ar[q];
    const int kx = q / kFC, o = q % kFC;
    const float ck = kx == 0 ? scale : 2.f * scale;
    Bs[(kFC + 2 * kx) * kFC + o] = a.x * ck;
    Bs[(kFC + 2 * kx + 1) * kFC + o] = a.y * ck;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  for (int x0 = 0; x0 < span; x0 += NT / OG) {
    const int xi = x0 + tid / OG;
    const bool in = xi < span;
    float acc[T][T];
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
      for (int j = 0; j < T; ++j) acc[i][j] = bias[j];
    if (in) {
      const int xa = 4 * xi, xb = xi + span < n4 ? 4 * (xi + span) : xa;
      const float* w = Bs + 4 * og;
#pragma unroll 4
      for (int k = 0; k < kFC; ++k, w += kFC) {
        const float* a = vs + k * P;
        if constexpr (T == 8)
          outer8(acc, f4(a + xa), f4(a + xb), f4(w), f4(w + 16));
        else
          outer4(acc, f4(a + xa), f4(w));
      }
#pragma unroll 4
      for (int k = 0; k < 2 * K; ++k, w += kFC) {
        if constexpr (T == 8) {
          const float* a = tw + (long)k * Wp;
          outer8(acc, ldg4(a + xa), ldg4(a + xb), f4(w), f4(w + 16));
        } else {
          outer4(acc, f4(ts + k * P + xa), f4(w));
        }
      }
    }
    if (next) __syncthreads();  // this round's cells of vs are read
#pragma unroll
    for (int p = 0; p < H4; ++p) {
      const int x = 4 * (xi + p * span);
      if (!in || xi + p * span >= n4) continue;
#pragma unroll
      for (int j = 0; j < T; ++j) {
        const int o = j / 4 * 16 + 4 * og + j % 4;
        const long at = base + (long)o * Wp + x;
        float u[4];
        float4 gp = make_float4(0.f, 0.f, 0.f, 0.f);
        if (BWD && gpre) gp = f4(gpre + at);
        const float gv[4] = {gp.x, gp.y, gp.z, gp.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          u[i] = acc[4 * p + i][j];
          if (BWD && gpre) u[i] *= fgelu_grad(gv[i]);
          if (x + i >= W) u[i] = 0.f;
        }
        if (!BWD && pre) *reinterpret_cast<float4*>(pre + at) = make_float4(u[0], u[1], u[2], u[3]);
        if (!BWD && gelu_out) {
#pragma unroll
          for (int i = 0; i < 4; ++i) u[i] = fgelu(u[i]);
        }
        const float4 o4 = make_float4(u[0], u[1], u[2], u[3]);
        *reinterpret_cast<float4*>(out + at) = o4;
        if (next) *reinterpret_cast<float4*>(vs + o * P + x) = o4;
      }
    }
  }
  if (!next) return;
  __syncthreads();
  fno_row_dft<TWS>(vs, P, Wp, K, TWS ? ts : tw, TWS ? P : Wp, Ar);
}

// ---------------------------------------------------------------------------
// Projection q = Q2 gelu(Q1 v + q1) + q2 of a tile of 64 cells (16 groups of 4
// cells, counted through the rows, so no tile is cut at a row's end) by 256
// threads: thread (xg, jg) holds hidden values 4 jg .. + 3 of cells 4 xg .. + 3
// and 32 + 4 xg .. + 3.
// ---------------------------------------------------------------------------
constexpr int kPT = 64;         // cells per tile
constexpr int kPP = kPT + 4;    // pitch of [.][cell] tiles
constexpr int kPN = 256;        // threads per block

// z[x][j] of the thread's 8 x 4 tile
__device__ __forceinline__ void fno_hidden(float (&z)[8][4], const float* Q1t, const float* q1s, const float* vs,
                                           int xg, int jg) {
  const float4 b = f4(q1s + 4 * jg);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    z[i][0] = b.x;
    z[i][1] = b.y;
    z[i][2] = b.z;
    z[i][3] = b.w;
  }
#pragma unroll 4
  for (int k = 0; k < kFC; ++k) {
    const float4 v0 = f4(vs + k * kPP + 4 * xg), v1 = f4(vs + k * kPP + 32 + 4 * xg);
    const float4 w = f4(Q1t + k * (kFH + 4) + 4 * jg);
    const float vv[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w}, ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) z[i][j] = fmaf(vv[i], ww[j], z[i][j]);
  }
}

// Q1^T [i][j] (pitch 132), q1, Q2 into shared memory
__device__ __forceinline__ void fno_proj_weights(float* Q1t, float* q1s, float* Q2s, const float* __restrict__ Q1,
                                                 const float* __restrict__ q1, const float* __restrict__ Q2) {
  for (int q = threadIdx.x; q < kFH * kFC; q += blockDim.x) Q1t[(q % kFC) * (kFH + 4) + q / kFC] = __ldg(&Q1[q]);
  for (int q = threadIdx.x; q < kFH; q += blockDim.x) q1s[q] = __ldg(&q1[q]);
  for (int q = threadIdx.x; q < 3 * kFH; q += blockDim.x) Q2s[q] = __ldg(&Q2[q]);
}

// the tile's v planes (zero beyond the last group)
__device__ __forceinline__ void fno_load_tile(float* vs, const float* v, long tile, long groups, int Wp) {
  const int n4 = Wp / 4, g = threadIdx.x % (kPT / 4);
  const long gg = tile * (kPT / 4) + g;
  const long r = (int)gg / n4;  // (a group has 6 kB of activations, so their number fits 31 bits)
  const float* src = v + r * kFC * Wp + (gg - r * n4) * 4;
#pragma unroll
  for (int q = 0; q < kFC * (kPT / 4) / kPN; ++q) {
    const int c = threadIdx.x / (kPT / 4) + q * (kPN / (kPT / 4));
    *reinterpret_cast<float4*>(vs + c * kPP + 4 * g) = gg < groups ? f4(src + (long)c * Wp) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// cell i of the tile: its index in the compact [row][W] fields, -1 for padding
__device__ __forceinline__ long fno_cell(long tile, int i, long groups, int W, int Wp) {
  const long gg = tile * (kPT / 4) + i / 4;
  const long r = (int)gg / (Wp / 4);
  const int x = (int)(gg - r * (Wp / 4)) * 4 + i % 4;
  return gg < groups && x < W ? r * W + x : -1;
}

// o[k][i] over the thread's 4 hidden values, summed over the four jg of its
// warp and left in red[warp][k][cell]
__device__ __forceinline__ void fno_reduce_pred(float (&o)[3][8], float (*red)[3][kPT], int xg) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    reduce_scatter<8, 2, 3>(o[k], lane);  // lane bits 3, 4 = idx: entries idx, idx + 4
    const int i = (lane >> 3) & 3;
    red[warp][k][4 * xg + i] = o[k][0];
    red[warp][k][32 + 4 * xg + i] = o[k][1];
  }
}

// Inference: h = q std + mean (float4 per cell), one tile per block.
__global__ void __launch_bounds__(kPN) fno_proj_kernel(const float* v, long groups, int W, int Wp,
                                                       const float* __restrict__ Q1, const float* __restrict__ q1,
                                                       const float* __restrict__ Q2, const float* __restrict__ q2,
                                                       float4* __restrict__ out, float3 mean, float3 sd) {
  __shared__ __align__(16) float Q1t[kFC * (kFH + 4)], q1s[kFH], Q2s[3 * kFH], vs[kFC * kPP];
  __shared__ float red[8][3][kPT];
  fno_proj_weights(Q1t, q1s, Q2s, Q1, q1, Q2);
  pdl_wait_next();
  fno_load_tile(vs, v, blockIdx.x, groups, Wp);
  __syncthreads();
  const int tid = threadIdx.x, xg = tid & 7, jg = tid >> 3;
  float z[8][4];
  fno_hidden(z, Q1t, q1s, vs, xg, jg);
  float o[3][8] = {};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float a = Q2s[4 * jg + j], b = Q2s[kFH + 4 * jg + j], c = Q2s[2 * kFH + 4 * jg + j];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float h = fgelu(z[i][j]);
      o[0][i] = fmaf(a, h, o[0][i]);
      o[1][i] = fmaf(b, h, o[1][i]);
      o[2][i] = fmaf(c, h, o[2][i]);
    }
  }
  fno_reduce_pred(o, red, xg);
  __syncthreads();
  const long cell = tid < kPT ? fno_cell(blockIdx.x, tid, groups, W, Wp) : -1;
  if (cell >= 0) {
    float q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      q[k] = __ldg(&q2[k]);
#pragma unroll
      for (int w = 0; w < 8; ++w) q[k] += red[w][k][tid];
    }
    out[cell] = make_float4(q[0] * sd.x + mean.x, q[1] * sd.y + mean.y, q[2] * sd.z + mean.z, 0.f);
  }
}

// Training: projection, SmoothL1 (beta 1) against the normalised target, and
// the projection's backward pass, over the tiles of a persistent block:
//   dz[j] = gelu'(z[j]) sum_k Q2[k][j] g[k];  dv[i] = sum_j Q1[j][i] dz[j]
// (the last spectral layer has no activation), and dQ1, dq1, dQ2, dq2 summed in
// registers and added once per block.  Per cell 13 k FMA and 128 erf and exp;
// the separate kernels moved z and dz (1 KB per cell) through memory five times.
// Bound: the load path of the tiled products (8 x 4 and 8 x 8 values per thread)
// and FP32 issue: 232 us for 32 fields of 160 x 40 (the five kernels it replaces
// took 630); 64-thread blocks with 8 x 8 tiles throughout (255 registers, 8 warps
// per SM) took 241.
struct FnoTrainSmem {
  float Q1t[kFC * (kFH + 4)];  // [i][j]
  float q1s[kFH], Q2s[3 * kFH];
  float vs[kFC * kPP];         // [i][x]
  float hs[kFH * kPP];         // [j][x]: gelu(z), then dz
  float red[8][3][kPT];
  float g[3][kPP];             // dL/dq
};

__global__ void __launch_bounds__(kPN, 2)
    fno_proj_train_kernel(const float* v, const float4* h_target, long groups, int W, int Wp,
                          const float* __restrict__ Q1, const float* __restrict__ q1, const float* __restrict__ Q2,
                          const float* __restrict__ q2, float3 mean, float3 inv_std, float inv_count,
                          float* __restrict__ dv, float* __restrict__ dQ1, float* __restrict__ dq1,
                          float* __restrict__ dQ2, float* __restrict__ dq2, float* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char trraw[];
  FnoTrainSmem& s = *reinterpret_cast<FnoTrainSmem*>(trraw);
  const int tid = threadIdx.x, xg = tid & 7, jg = tid >> 3, lane = tid & 31, warp = tid >> 5;
  fno_proj_weights(s.Q1t, s.q1s, s.Q2s, Q1, q1, Q2);
  pdl_wait_next();
  const long ntiles = (groups + kPT / 4 - 1) / (kPT / 4);
  // dQ1[jr + 16 a][ir + 8 b] over half kh of the tile's cells
  const int jr = tid & 15, ir = (tid >> 4) & 7, kh = tid >> 7;
  float aQ1[8][4] = {};
  float aq1 = 0.f;        // dq1[tid / 2], half tid % 2 of the cells
  float aQ2[3] = {};      // dQ2[k][tid / 2], likewise
  float aq2 = 0.f;        // dq2[warp] (lane 0 after the sum; warps 0..2)
  double aloss = 0.0;
  for (long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    __syncthreads();  // the previous tile's vs and hs are read
    fno_load_tile(s.vs, v, tile, groups, Wp);
    __syncthreads();
    float z[8][4];
    fno_hidden(z, s.Q1t, s.q1s, s.vs, xg, jg);
    {
      float o[3][8] = {};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int jj = 4 * jg + j;
        const float a = s.Q2s[jj], b = s.Q2s[kFH + jj], c = s.Q2s[2 * kFH + jj];
        float h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          // gelu and, in z's place, its derivative
          const float y = z[i][j], e = 0.5f * (1.f + erff(y * 0.70710678118654752f));
          h[i] = y * e;
          z[i][j] = e + y * 0.39894228040143268f * expf(-0.5f * y * y);
          o[0][i] = fmaf(a, h[i], o[0][i]);
          o[1][i] = fmaf(b, h[i], o[1][i]);
          o[2][i] = fmaf(c, h[i], o[2][i]);
        }
        *reinterpret_cast<float4*>(s.hs + jj * kPP + 4 * xg) = make_float4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<float4*>(s.hs + jj * kPP + 32 + 4 * xg) = make_float4(h[4], h[5], h[6], h[7]);
      }
      fno_reduce_pred(o, s.red, xg);
    }
    __syncthreads();
    if (tid < kPT) {
      float gg[3] = {0.f, 0.f, 0.f};
      const long cell = fno_cell(tile, tid, groups, W, Wp);
      if (cell >= 0) {
        const float4 t = h_target[cell];
        const float tn[3] = {(t.x - mean.x) * inv_std.x, (t.y - mean.y) * inv_std.y, (t.z - mean.z) * inv_std.z};
        float l = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          float q = __ldg(&q2[k]);
#pragma unroll
          for (int w = 0; w < 8; ++w) q += s.red[w][k][tid];
          const float d = q - tn[k], ad = fabsf(d);
          l += ad < 1.f ? 0.5f * d * d : ad - 0.5f;
          gg[k] = fminf(fmaxf(d, -1.f), 1.f) * inv_count;
        }
        aloss += (double)l;
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) s.g[k][tid] = gg[k];
    }
    __syncthreads();
    // dQ2[k][j] += sum_x g[k][x] h[j][x]: two threads per hidden row
    {
      const float* hr = s.hs + (tid >> 1) * kPP + 4 * (tid & 1);
      const float* gr = s.g[0] + 4 * (tid & 1);
#pragma unroll
      for (int x = 0; x < kPT; x += 8) {
        const float4 h = f4(hr + x);
#pragma unroll
        for (int k = 0; k < 3; ++k) aQ2[k] = dot4(f4(gr + k * kPP + x), h, aQ2[k]);
      }
    }
    if (warp < 3) aq2 += s.g[warp][lane] + s.g[warp][lane + 32];
    __syncthreads();  // gelu(z) is read
    {
      float g[3][8];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float4 a = f4(s.g[k] + 4 * xg), b = f4(s.g[k] + 32 + 4 * xg);
        g[k][0] = a.x, g[k][1] = a.y, g[k][2] = a.z, g[k][3] = a.w;
        g[k][4] = b.x, g[k][5] = b.y, g[k][6] = b.z, g[k][7] = b.w;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int jj = 4 * jg + j;
        const float a = s.Q2s[jj], b = s.Q2s[kFH + jj], c = s.Q2s[2 * kFH + jj];
        float d[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) d[i] = z[i][j] * (a * g[0][i] + b * g[1][i] + c * g[2][i]);
        *reinterpret_cast<float4*>(s.hs + jj * kPP + 4 * xg) = make_float4(d[0], d[1], d[2], d[3]);
        *reinterpret_cast<float4*>(s.hs + jj * kPP + 32 + 4 * xg) = make_float4(d[4], d[5], d[6], d[7]);
      }
    }
    __syncthreads();
    // dv[i][x] = sum_j Q1[j][i] dz[j][x]: an eighth sp of the hidden sum, channels 8 ig .. + 7, cells 4 xq .. + 3
    // and 32 + 4 xq .. + 3
    {
      const int sp = tid & 7, xq = (tid >> 3) & 7, ig = tid >> 6;
      float a[64];
#pragma unroll
      for (int q = 0; q < 64; ++q) a[q] = 0.f;
#pragma unroll 1
      for (int j4 = sp; j4 < kFH / 4; j4 += 8) {
        float4 w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = f4(s.Q1t + (8 * ig + i) * (kFH + 4) + 4 * j4);
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const float* d = s.hs + (4 * j4 + jj) * kPP + 4 * xq;
          const float4 d0 = f4(d), d1 = f4(d + 32);
          const float dx[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float wi = jj == 0 ? w[i].x : (jj == 1 ? w[i].y : (jj == 2 ? w[i].z : w[i].w));
#pragma unroll
            for (int x = 0; x < 8; ++x) a[i * 8 + x] = fmaf(wi, dx[x], a[i * 8 + x]);
          }
        }
      }
      reduce_scatter<64, 3, 0>(a, lane);  // entries q = 8 k + sp: channel k, cell entry sp
      const long gg = tile * (kPT / 4) + (sp < 4 ? 0 : 8) + xq;
      const long r = (int)gg / (Wp / 4);
      if (gg < groups) {
        float* dst = dv + (r * kFC + 8 * ig) * Wp + (gg - r * (Wp / 4)) * 4 + (sp & 3);
        // (dz is zero in the padding, so dv is too)
#pragma unroll
        for (int k = 0; k < 8; ++k) dst[(long)k * Wp] = a[k];
      }
    }
    // dQ1[j][i] += sum_x dz[j][x] v[i][x]
#pragma unroll 1
    for (int x = 32 * kh; x < 32 * kh + 32; x += 4) {
      float4 u[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) u[b] = f4(s.vs + (ir + 8 * b) * kPP + x);
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const float4 d = f4(s.hs + (jr + 16 * a) * kPP + x);
#pragma unroll
        for (int b = 0; b < 4; ++b) aQ1[a][b] = dot4(d, u[b], aQ1[a][b]);
      }
    }
    {
      const float* d = s.hs + (tid >> 1) * kPP + 4 * (tid & 1);
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int x = 0; x < kPT; x += 8) {
        const float4 q = f4(d + x);
        t = make_float4(t.x + q.x, t.y + q.y, t.z + q.z, t.w + q.w);
      }
      aq1 += (t.x + t.y) + (t.z + t.w);
    }
  }
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) atomicAdd(&dQ1[(jr + 16 * a) * kFC + ir + 8 * b], aQ1[a][b]);
  atomicAdd(&dq1[tid >> 1], aq1);
#pragma unroll
  for (int k = 0; k < 3; ++k) atomicAdd(&dQ2[k * kFH + (tid >> 1)], aQ2[k]);
  if (warp < 3) {
    for (int o = 16; o > 0; o >>= 1) aq2 += __shfl_down_sync(0xffffffffu, aq2, o);
    if (lane == 0) atomicAdd(&dq2[warp], aq2);
  }
  if (warp < 2) {
    for (int o = 16; o > 0; o >>= 1) aloss += __shfl_down_sync(0xffffffffu, aloss, o);
    if (lane == 0) atomicAdd(loss, (float)(aloss * (double)inv_count));
  }
}

// Pointwise weight gradient of a layer: dW[o][i] += sum du[o][x] v[i][x], db[o] +=
// sum du[o][x] over the cells of the block's rows.  Four groups of 64 threads
// take a quarter of a chunk's cells each, a thread 4 x 4 outputs (channels 8
// apart, so a warp's float4 reads meet no bank twice): 64 FMA per 8 loads.
constexpr int kWgX = 64, kWgP = kWgX + 4;
__global__ void __launch_bounds__(256) fno_wgrad_kernel(const float* du, const float* v,
                                                        long rows, int Wp, float* __restrict__ dW,
                                                        float* __restrict__ db) {
  __shared__ __align__(16) float as[2 * kFC * kWgP];
  float* bs = as + kFC * kWgP;
  const int tid = threadIdx.x, o0 = tid & 7, i0 = (tid >> 3) & 7, grp = tid >> 6;
  float acc[4][4] = {}, ab[4] = {};
  pdl_wait_next();
  const int per = (Wp + kWgX - 1) / kWgX;
  // the next chunk's loads are in flight while this one is summed
  constexpr int NL = kFC * (kWgX / 4) / 256;
  const int lc = tid / (kWgX / 4), lx = tid % (kWgX / 4) * 4;
  float4 na[NL], nb[NL];
  auto load = [&](long t) {
    const long r = t / per;
    const int x = (int)(t % per) * kWgX + lx;
    const bool in = t < rows * per && x < Wp;
#pragma unroll
    for (int q = 0; q < NL; ++q) {
      const long at = (r * kFC + lc + q * (kFC / NL)) * Wp + x;
      na[q] = in ? f4(du + at) : make_float4(0.f, 0.f, 0.f, 0.f);
      nb[q] = in ? f4(v + at) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  load(blockIdx.x);
  for (long t = blockIdx.x; t < rows * per; t += gridDim.x) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NL; ++q) {
      *reinterpret_cast<float4*>(as + (lc + q * (kFC / NL)) * kWgP + lx) = na[q];
      *reinterpret_cast<float4*>(bs + (lc + q * (kFC / NL)) * kWgP + lx) = nb[q];
    }
    __syncthreads();
    load(t + gridDim.x);
#pragma unroll
    for (int x = grp * (kWgX / 4); x < (grp + 1) * (kWgX / 4); x += 4) {
      float4 a[4], b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a[q] = f4(as + (o0 + 8 * q) * kWgP + x);
        b[q] = f4(bs + (i0 + 8 * q) * kWgP + x);
      }
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        if (i0 == 0) ab[p] += (a[p].x + a[p].y) + (a[p].z + a[p].w);
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = dot4(a[p], b[q], acc[p][q]);
      }
    }
  }
  // the four groups' sums through shared memory, then one addition per output and block
  float* part = as;  // [group][o][i | sum]: 4 x 32 x 33 floats fit as and bs together
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    if (i0 == 0) part[(grp * kFC + o0 + 8 * p) * (kFC + 1) + kFC] = ab[p];
#pragma unroll
    for (int q = 0; q < 4; ++q) part[(grp * kFC + o0 + 8 * p) * (kFC + 1) + i0 + 8 * q] = acc[p][q];
  }
  __syncthreads();
  for (int q = tid; q < kFC * (kFC + 1); q += 256) {
    constexpr int G = kFC * (kFC + 1);
    const float t = (part[q] + part[G + q]) + (part[2 * G + q] + part[3 * G + q]);
    const int o = q / (kFC + 1), i = q % (kFC + 1);
    atomicAdd(i == kFC ? &db[o] : &dW[o * kFC + i], t);
  }
}

// Lifting layer's gradient: dP[o][k] += sum du[o][x] xn[k][x], dp[o] += sum
// du[o][x]; warp o of the block, lanes over x.
__global__ void __launch_bounds__(1024) fno_lift_grad_kernel(const float* du, const float4* m,
                                                             long rows, int W, int Wp, float3 mean, float3 inv_std,
                                                             float* __restrict__ dP, float* __restrict__ dp) {
  const int o = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float a[4] = {};
  pdl_wait_next();
  for (long r = blockIdx.x; r < rows; r += gridDim.x) {
    const float* d = du + (r * kFC + o) * Wp;
    for (int x = lane; x < W; x += 32) {
      const float u = d[x];
      const float4 c = m[r * W + x];
      a[0] = fmaf(u, (c.x - mean.x) * inv_std.x, a[0]);
      a[1] = fmaf(u, (c.y - mean.y) * inv_std.y, a[1]);
      a[2] = fmaf(u, (c.z - mean.z) * inv_std.z, a[2]);
      a[3] += u;
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    for (int q = 16; q > 0; q >>= 1) a[k] += __shfl_down_sync(0xffffffffu, a[k], q);
  if (lane == 0) {
    for (int k = 0; k < 3; ++k) atomicAdd(&dP[o * 3 + k], a[k]);
    atomicAdd(&dp[o], a[3]);
  }
}

// Filter gradient per kept mode: dR[mode][i][o] = s_kx sum_b conj(X[mode][b][i]) Xg[mode][b][o],
// s_kx = (kx == 0 ? 1 : 2) / (H W).  One block of 32 x 32 threads per mode.
__global__ void __launch_bounds__(1024) fno_rgrad_kernel(const float2* X, const float2* Xg,
                                                         float* __restrict__ dR, int B, int K, float scale) {
  __shared__ float2 xs[kFC][kFC];
  __shared__ float2 gs[kFC][kFC];
  const int mode = blockIdx.x, kx = mode % K;
  pdl_wait_next();
  const int i = threadIdx.x >> 5, o = threadIdx.x & 31;
  const float2* Xm = X + (long)mode * B * kFC;
  const float2* Gm = Xg + (long)mode * B * kFC;
  float re = 0.f, im = 0.f;
  for (int b0 = 0; b0 < B; b0 += kFC) {
    const int nb = min(kFC, B - b0);
    __syncthreads();
    if (i < nb) {
      xs[i][o] = Xm[(long)(b0 + i) * kFC + o];
      gs[i][o] = Gm[(long)(b0 + i) * kFC + o];
    }
    __syncthreads();
    for (int b = 0; b < nb; ++b) {
      const float2 a = xs[b][i], g = gs[b][o];
      re = fmaf(a.x, g.x, fmaf(a.y, g.y, re));  // conj(a) g
      im = fmaf(a.x, g.y, fmaf(-a.y, g.x, im));
    }
  }
  const float s = kx == 0 ? scale : 2.f * scale;
  float2* out = (float2*)(dR + (long)mode * kFC * kFC * 2);
  out[i * kFC + o] = make_float2(re * s, im * s);
}

}  // namespace mx

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
struct mx_fno {
  int nx, ny, K, max_batch;
  int wp;      // nx rounded up to 4: columns of a stored row
  long cells;  // per sample
  long np;
  float* params = nullptr;
  float* grad = nullptr;
  float* am = nullptr;
  float* av = nullptr;
  int adam_t = 0;
  float* twx = nullptr;   // [2 kx, 2 kx + 1][x]: cos, -sin of 2 pi kx x / W, zero in the padding
  float2* twy = nullptr;  // [y][m]: e^{-2 pi i ky(m) y / H}
  float* v[mx::kFL + 1] = {};
  float* pre[mx::kFL - 1] = {};
  float2* A = nullptr;
  float2* X[mx::kFL] = {};
  float2* Xg = nullptr;
  float2* Y = nullptr;
  float* du[2] = {};
  float* loss = nullptr;
  float stats[12] = {0, 0, 0, 1, 1, 1, 0, 0, 0, 1, 1, 1};
};

namespace mx {

struct FnoOffsets {
  long P, p, R[kFL], W[kFL], w[kFL], Q1, q1, Q2, q2, total;
};

static FnoOffsets fno_offsets(int K) {
  FnoOffsets f;
  long o = 0;
  f.P = o; o += kFC * 3;
  f.p = o; o += kFC;
  for (int l = 0; l < kFL; ++l) {
    f.R[l] = o; o += 2L * K * K * kFC * kFC * 2;
    f.W[l] = o; o += kFC * kFC;
    f.w[l] = o; o += kFC;
  }
  f.Q1 = o; o += kFH * kFC;
  f.q1 = o; o += kFH;
  f.Q2 = o; o += 3 * kFH;
  f.q2 = o; o += 3;
  f.total = o;
  return f;
}

// Launch shape of the row kernels (a block per row): the small variant (4 x 4
// tiles, more threads, staged twiddles) where at most one row falls to an SM and
// its buffers fit.  One field of 160 x 40 takes 72 us with it and 96 without; four
// fields 138 us with it (two rows on some SMs) and 115 without.
struct FnoRowShape {
  bool small;
  int threads;
  size_t smem;
};
constexpr size_t kFnoMaxSmem = 220 * 1024;
static FnoRowShape row_shape(const mx_fno* n, int B, bool first) {
  const size_t pitch = sizeof(float) * (size_t)fno_pitch(n->wp);
  const size_t bs = first ? 0 : sizeof(float) * (size_t)(kFC + 2 * n->K) * kFC;
  FnoRowShape r;
  r.smem = bs + (kFC + 2 * n->K) * pitch;
  r.small = (long)B * n->ny <= 152 && r.smem <= kFnoMaxSmem;
  if (!r.small) r.smem = bs + kFC * pitch;
  const int n4 = n->wp / 4;
  const int want = first ? (r.small ? 384 : 128) : (r.small ? n4 * 8 : (n4 + 1) / 2 * 4);
  const int most = r.small ? 512 : 256;
  r.threads = (want + 31) / 32 * 32 < most ? (want + 31) / 32 * 32 : most;
  return r;
}

struct FnoNorm {
  float3 mean, inv_std, hmean, hstd, hinv;
};
static FnoNorm fno_norm(const mx_fno* n) {
  const float* s = n->stats;
  return FnoNorm{make_float3(s[0], s[1], s[2]), make_float3(1.f / s[3], 1.f / s[4], 1.f / s[5]),
                 make_float3(s[6], s[7], s[8]), make_float3(s[9], s[10], s[11]),
                 make_float3(1.f / s[9], 1.f / s[10], 1.f / s[11])};
}

// Column pass of layer l on n->A (ADJ: with the conjugate-transposed filters);
// X receives the kept modes unless null.
template <bool ADJ> static mx_status fno_mid(mx_fno* n, int l, float2* X, int B, cudaStream_t st) {
  const FnoOffsets f = fno_offsets(n->K);
  if (B >= kMidBatch) {
    const int K = n->K, H = n->ny;
    const unsigned cols = (unsigned)(((long)B * K + 3) / 4);
    float2* Xb = X ? X : n->X[0];
    launch_pdl(fno_dft_y_kernel, dim3(cols, (2 * K + kMidM - 1) / kMidM), dim3(128), 0, st, n->A, Xb, B, H, K, n->twy);
    MX_TRY(launch_check("fno_dft_y_kernel"));
    launch_pdl(fno_mix_kernel<ADJ>, dim3(2 * K * K), dim3(256), 0, st, Xb, n->Y, n->params + f.R[l], B, K);
    MX_TRY(launch_check("fno_mix_kernel"));
    launch_pdl(fno_idft_y_kernel, dim3(cols, (H + kMidY - 1) / kMidY), dim3(128), 0, st, n->Y, n->A, B, H, K, n->twy);
    return launch_check("fno_idft_y_kernel");
  }
  launch_pdl(fno_mid_kernel<ADJ>, dim3(kMidCl * n->K * B), dim3(kMidWarps * 32), sizeof(FnoMidSmem), st, n->A, X,
             n->params + f.R[l], B, n->ny, n->K, n->twy);
  return launch_check("fno_mid_kernel");
}

template <bool LIFT>
static mx_status fno_first(mx_fno* n, const float4* m, float* v, int B, cudaStream_t st) {
  const FnoOffsets f = fno_offsets(n->K);
  const FnoNorm nm = fno_norm(n);
  const FnoRowShape rs = row_shape(n, B, true);
  launch_pdl(rs.small ? fno_first_kernel<LIFT, true> : fno_first_kernel<LIFT, false>, dim3((unsigned)(B * n->ny)),
             dim3(rs.threads), rs.smem, st, m, nm.mean, nm.inv_std, n->params + f.P, n->params + f.p, v, n->A, n->nx,
             n->wp, n->K, n->twx);
  return launch_check("fno_first_kernel");
}

template <bool BWD>
static mx_status fno_row(mx_fno* n, int l, const float* vin, float* pre, float* out, const float* gpre, bool gelu_out,
                         bool next, int B, cudaStream_t st) {
  const FnoOffsets f = fno_offsets(n->K);
  const FnoRowShape rs = row_shape(n, B, false);
  const float scale = 1.f / ((float)n->ny * (float)n->nx);
  launch_pdl(rs.small ? fno_row_kernel<BWD, 4> : fno_row_kernel<BWD, 8>, dim3((unsigned)(B * n->ny)),
             dim3(rs.threads), rs.smem, st, n->A, vin, n->params + f.W[l], BWD ? nullptr : n->params + f.w[l], pre, out, gpre, n->nx, n->wp, n->K,
             scale, gelu_out ? 1 : 0, next ? 1 : 0, n->twx);
  return launch_check("fno_row_kernel");
}

// Lifting and the four spectral layers; returns v_4 in *v4.
static mx_status fno_layers(mx_fno* n, const float4* m, int B, bool train, const float** v4, cudaStream_t st) {
  MX_TRY(fno_first<true>(n, m, n->v[0], B, st));
  for (int l = 0; l < kFL; ++l) {
    // inference ping-pongs v[0] / v[1] and keeps no spectra
    const float* vin = train ? n->v[l] : n->v[l & 1];
    float* vout = train ? n->v[l + 1] : n->v[(l + 1) & 1];
    const bool last = l == kFL - 1;
    MX_TRY(fno_mid<false>(n, l, train ? n->X[l] : nullptr, B, st));
    MX_TRY(fno_row<false>(n, l, vin, train && !last ? n->pre[l] : nullptr, vout, nullptr, !last, !last, B, st));
  }
  *v4 = train ? n->v[kFL] : n->v[kFL & 1];
  return MX_OK;
}

static mx_status fno_forward(mx_fno* n, const float4* m, int B, float4* h_out, cudaStream_t st) {
  const FnoOffsets f = fno_offsets(n->K);
  const float* P = n->params;
  const FnoNorm nm = fno_norm(n);
  const float* v4 = nullptr;
  MX_TRY(fno_layers(n, m, B, false, &v4, st));
  const long groups = (long)B * n->ny * (n->wp / 4);
  launch_pdl(fno_proj_kernel, dim3((unsigned)((groups + kPT / 4 - 1) / (kPT / 4))), dim3(kPN), 0, st, v4, groups, n->nx,
             n->wp, P + f.Q1, P + f.q1, P + f.Q2, P + f.q2, h_out, nm.hmean, nm.hstd);
  return launch_check("fno_proj_kernel");
}

// Loss and gradient of a batch: forward, then backward, into n->loss and
// n->grad (zeroed by the caller).
static mx_status fno_train(mx_fno* n, const float4* m, const float4* h_target, int B, cudaStream_t st) {
  const FnoOffsets f = fno_offsets(n->K);
  const float* P = n->params;
  float* G = n->grad;
  const FnoNorm nm = fno_norm(n);
  const int W = n->nx, H = n->ny, K = n->K, Wp = n->wp;
  const long rows = (long)B * H;
  const float scale = 1.f / ((float)H * (float)W);
  const float* v4 = nullptr;
  MX_TRY(fno_layers(n, m, B, true, &v4, st));
  const long groups = rows * (Wp / 4), tiles = (groups + kPT / 4 - 1) / (kPT / 4);
  const long most = 2 * 152;  // persistent blocks, two per SM
  launch_pdl(fno_proj_train_kernel, dim3((unsigned)(tiles < most ? tiles : most)), dim3(kPN), sizeof(FnoTrainSmem), st,
             v4, h_target, groups, W, Wp, P + f.Q1, P + f.q1, P + f.Q2, P + f.q2, nm.hmean, nm.hinv,
             1.f / (3.f * (float)(n->cells * B)), n->du[0], G + f.Q1, G + f.q1, G + f.Q2, G + f.q2, n->loss);
  MX_TRY(launch_check("fno_proj_train_kernel"));
  // dL/du_3's row DFT; the others come with the row pass that forms dL/du_l
  MX_TRY(fno_first<false>(n, nullptr, n->du[0], B, st));
  const long chunks = rows * ((Wp + kWgX - 1) / kWgX);
  const unsigned wgrid = (unsigned)(chunks < 2 * 152 ? chunks : 2 * 152);
  int cur = 0;
  for (int l = kFL - 1; l >= 0; --l) {
    const float* du = n->du[cur];
    float* dnext = n->du[cur ^ 1];
    launch_pdl(fno_wgrad_kernel, dim3(wgrid), dim3(256), 0, st, du, n->v[l], rows, Wp, G + f.W[l], G + f.w[l]);
    MX_TRY(launch_check("fno_wgrad_kernel"));
    MX_TRY(fno_mid<true>(n, l, n->Xg, B, st));
    launch_pdl(fno_rgrad_kernel, dim3(2 * K * K), dim3(1024), 0, st, n->X[l], n->Xg, G + f.R[l], B, K, scale);
    MX_TRY(launch_check("fno_rgrad_kernel"));
    MX_TRY(fno_row<true>(n, l, du, nullptr, dnext, l > 0 ? n->pre[l - 1] : nullptr, false, l > 0, B, st));
    cur ^= 1;
  }
  launch_pdl(fno_lift_grad_kernel, dim3((unsigned)(rows < 152 ? rows : 152)), dim3(1024), 0, st, n->du[cur], m, rows, W,
             Wp, nm.mean, nm.inv_std, G + f.P, G + f.p);
  return launch_check("fno_lift_grad_kernel");
}

bool fno_matches(const mx_fno* n, const Grid& g) { return n->nx == g.nx && n->ny == g.ny && g.nz == 1; }

mx_status fno_demag(mx_fno* n, const float4* m, float4* h, cudaStream_t st) {
  return fno_forward(n, m, 1, h, st);
}

}  // namespace mx

using namespace mx;

extern "C" {

int mx_fno_num_params(int modes) {
  if (modes < 1 || modes > kFMaxK) return -1;
  return (int)fno_offsets(modes).total;
}

mx_status mx_fno_destroy(mx_fno* n) {
  if (!n) return MX_OK;
  std::vector<void*> ptrs = {n->params, n->grad, n->am, n->av, n->twx, n->twy, n->A, n->Xg, n->Y, n->du[0], n->du[1],
                             n->loss};
  for (int l = 0; l <= kFL; ++l) ptrs.push_back(n->v[l]);
  for (int l = 0; l < kFL - 1; ++l) ptrs.push_back(n->pre[l]);
  for (int l = 0; l < kFL; ++l) ptrs.push_back(n->X[l]);
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete n;
  return MX_OK;
}

mx_status mx_fno_create(mx_fno** out, int nx, int ny, int modes, int max_batch) {
  clear_error();
  if (!out || modes < 1 || modes > kFMaxK || nx < 2 * modes || ny < 2 * modes || nx > kFMaxN || ny > kFMaxN ||
      max_batch < 1 || max_batch > 65535) {
    set_error("mx_fno_create: need out != NULL, 1 <= modes <= 16, 2*modes <= nx, ny <= 1024 and "
              "1 <= max_batch <= 65535");
    return MX_ERR_INVALID_ARG;
  }
  *out = nullptr;
  mx_fno* n = new mx_fno();
  n->nx = nx;
  n->ny = ny;
  n->K = modes;
  n->max_batch = max_batch;
  n->wp = (nx + 3) / 4 * 4;
  n->cells = (long)nx * ny;
  n->np = fno_offsets(modes).total;
  const long nv = (long)n->wp * ny * max_batch * kFC;  // floats of one activation
  const long nspec = 2L * modes * modes * max_batch * kFC;
  bool ok = true;
  auto alloc = [&](void** p, size_t bytes) {
    if (ok && cudaMalloc(p, bytes) != cudaSuccess) {
      cudaGetLastError();
      ok = false;
    }
  };
  alloc((void**)&n->params, sizeof(float) * n->np);
  alloc((void**)&n->grad, sizeof(float) * n->np);
  alloc((void**)&n->am, sizeof(float) * n->np);
  alloc((void**)&n->av, sizeof(float) * n->np);
  alloc((void**)&n->twx, sizeof(float) * 2 * modes * n->wp);
  alloc((void**)&n->twy, sizeof(float2) * 2 * modes * ny);
  for (int l = 0; l <= kFL; ++l) alloc((void**)&n->v[l], sizeof(float) * nv);
  for (int l = 0; l < kFL - 1; ++l) alloc((void**)&n->pre[l], sizeof(float) * nv);
  alloc((void**)&n->A, sizeof(float2) * (size_t)max_batch * ny * modes * kFC);
  for (int l = 0; l < kFL; ++l) alloc((void**)&n->X[l], sizeof(float2) * nspec);
  alloc((void**)&n->Xg, sizeof(float2) * nspec);
  alloc((void**)&n->Y, sizeof(float2) * nspec);
  alloc((void**)&n->du[0], sizeof(float) * nv);
  alloc((void**)&n->du[1], sizeof(float) * nv);
  alloc((void**)&n->loss, sizeof(float));
  if (!ok) {
    mx_fno_destroy(n);
    set_error("mx_fno_create: device allocation failed");
    return MX_ERR_OOM;
  }
  // twiddles, in double on the host
  std::vector<float> tx((size_t)2 * modes * n->wp, 0.f);
  for (int kx = 0; kx < modes; ++kx)
    for (int x = 0; x < nx; ++x) {
      const double a = 2.0 * kPi * (double)(((long)kx * x) % nx) / (double)nx;
      tx[(size_t)(2 * kx) * n->wp + x] = (float)cos(a);
      tx[(size_t)(2 * kx + 1) * n->wp + x] = (float)-sin(a);
    }
  std::vector<float2> ty((size_t)2 * modes * ny);
  for (int y = 0; y < ny; ++y)
    for (int q = 0; q < 2 * modes; ++q) {
      const long ky = q < modes ? q : ny - 2 * modes + q;
      const double a = 2.0 * kPi * (double)((ky * y) % ny) / (double)ny;
      ty[(size_t)y * 2 * modes + q] = make_float2((float)cos(a), (float)-sin(a));
    }
  bool okc = true;
  okc = okc && cudaMemcpy(n->twx, tx.data(), sizeof(float) * tx.size(), cudaMemcpyHostToDevice) == cudaSuccess;
  okc = okc && cudaMemcpy(n->twy, ty.data(), sizeof(float2) * ty.size(), cudaMemcpyHostToDevice) == cudaSuccess;
  okc = okc && cudaMemset(n->params, 0, sizeof(float) * n->np) == cudaSuccess;
  okc = okc && cudaMemset(n->am, 0, sizeof(float) * n->np) == cudaSuccess;
  okc = okc && cudaMemset(n->av, 0, sizeof(float) * n->np) == cudaSuccess;
  auto smem = [&](const void* k, size_t bytes) {
    okc = okc && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
  };
  smem((const void*)fno_first_kernel<true, false>, kFnoMaxSmem);
  smem((const void*)fno_first_kernel<true, true>, kFnoMaxSmem);
  smem((const void*)fno_first_kernel<false, false>, kFnoMaxSmem);
  smem((const void*)fno_first_kernel<false, true>, kFnoMaxSmem);
  smem((const void*)fno_row_kernel<false, 4>, kFnoMaxSmem);
  smem((const void*)fno_row_kernel<false, 8>, kFnoMaxSmem);
  smem((const void*)fno_row_kernel<true, 4>, kFnoMaxSmem);
  smem((const void*)fno_row_kernel<true, 8>, kFnoMaxSmem);
  smem((const void*)fno_mid_kernel<false>, sizeof(FnoMidSmem));
  smem((const void*)fno_mid_kernel<true>, sizeof(FnoMidSmem));
  smem((const void*)fno_proj_train_kernel, sizeof(FnoTrainSmem));
  if (!okc) {
    cudaGetLastError();
    mx_fno_destroy(n);
    set_error("mx_fno_create: device set-up failed");
    return MX_ERR_CUDA;
  }
  *out = n;
  return MX_OK;
}

mx_status mx_fno_set_params(mx_fno* n, const float* params, mx_stream_t stream) {
  if (!n || !params) {
    set_error("mx_fno_set_params: NULL argument");
    return MX_ERR_INVALID_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  MX_CUDA_TRY(cudaMemcpyAsync(n->params, params, sizeof(float) * n->np, cudaMemcpyDeviceToDevice, st));
  MX_CUDA_TRY(cudaMemsetAsync(n->am, 0, sizeof(float) * n->np, st));
  MX_CUDA_TRY(cudaMemsetAsync(n->av, 0, sizeof(float) * n->np, st));
  n->adam_t = 0;
  return MX_OK;
}

mx_status mx_fno_get_params(const mx_fno* n, float* params, mx_stream_t stream) {
  if (!n || !params) {
    set_error("mx_fno_get_params: NULL argument");
    return MX_ERR_INVALID_ARG;
  }
  MX_CUDA_TRY(cudaMemcpyAsync(params, n->params, sizeof(float) * n->np, cudaMemcpyDeviceToDevice,
                              (cudaStream_t)stream));
  return MX_OK;
}

mx_status mx_fno_set_normalizer(mx_fno* n, const double stats[12]) {
  if (!n || !stats) {
    set_error("mx_fno_set_normalizer: NULL argument");
    return MX_ERR_INVALID_ARG;
  }
  for (int q = 0; q < 12; ++q) {
    if (!isfinite(stats[q]) || ((q % 6) >= 3 && !(stats[q] > 0))) {
      set_error("mx_fno_set_normalizer: standard deviations must be > 0 and every entry finite");
      return MX_ERR_INVALID_ARG;
    }
  }
  for (int q = 0; q < 12; ++q) n->stats[q] = (float)stats[q];
  return MX_OK;
}

static mx_status fno_check(const mx_fno* n, const float* m, int batch, const char* what) {
  if (!n || !m || batch < 1 || batch > n->max_batch || (((uintptr_t)m) & 15)) {
    set_error(std::string(what) + ": bad network, pointer or batch (1..max_batch)");
    return MX_ERR_INVALID_ARG;
  }
  return MX_OK;
}

mx_status mx_fno_forward(mx_fno* n, const float* m, float* h, int batch, mx_stream_t stream) {
  MX_TRY(fno_check(n, m, batch, "mx_fno_forward"));
  if (!h || (((uintptr_t)h) & 15)) {
    set_error("mx_fno_forward: h must be a 16-byte aligned device pointer");
    return MX_ERR_INVALID_ARG;
  }
  return fno_forward(n, (const float4*)m, batch, (float4*)h, (cudaStream_t)stream);
}

mx_status mx_fno_loss_grad(mx_fno* n, const float* m, const float* h_target, int batch, float* loss_out,
                           float* grad_out, mx_stream_t stream) {
  MX_TRY(fno_check(n, m, batch, "mx_fno_loss_grad"));
  if (!h_target || (((uintptr_t)h_target) & 15)) {
    set_error("mx_fno_loss_grad: h_target must be a 16-byte aligned device pointer");
    return MX_ERR_INVALID_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  MX_CUDA_TRY(cudaMemsetAsync(n->loss, 0, sizeof(float), st));
  MX_CUDA_TRY(cudaMemsetAsync(n->grad, 0, sizeof(float) * n->np, st));
  MX_TRY(fno_train(n, (const float4*)m, (const float4*)h_target, batch, st));
  if (loss_out) MX_CUDA_TRY(cudaMemcpyAsync(loss_out, n->loss, sizeof(float), cudaMemcpyDeviceToDevice, st));
  if (grad_out)
    MX_CUDA_TRY(cudaMemcpyAsync(grad_out, n->grad, sizeof(float) * n->np, cudaMemcpyDeviceToDevice, st));
  return MX_OK;
}

mx_status mx_fno_adam_step(mx_fno* n, double lr, double weight_decay, mx_stream_t stream) {
  if (!n || !(lr > 0) || !(weight_decay >= 0)) {
    set_error("mx_fno_adam_step: need a network, lr > 0 and weight_decay >= 0");
    return MX_ERR_INVALID_ARG;
  }
  n->adam_t += 1;
  return adam_update(n->params, n->grad, n->am, n->av, n->np, lr, weight_decay, n->adam_t, (cudaStream_t)stream);
}

}  // extern "C"
