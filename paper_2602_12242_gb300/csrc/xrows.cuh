// Row pieces of the compile-time-sized x transforms (demag_fast.cu, and the
// row kernels of the RK4 step and of the adjoint's reverse sweep): r2c of
// Ms m rows into the spectrum w1[c][row][kx], c2r of spectrum rows into
// shared memory, and the few-row block configuration of each size.  The same
// arithmetic as demag.cu's generic x kernels (Sec. II-B: zero-padded FFT
// convolution).
#pragma once

#include "common.cuh"
#include "fft.cuh"
#include "regfft.cuh"

namespace mx {

// ---------------------------------------------------------------------------
// Line8<M>: an M-point transform (M = 16 .. 1024, a power of two) on TL = M/8
// threads of eight elements: Stockham passes of radix 8, the last of radix
// 2, 4 or 8.  Thread j holds x[j + u TL], u < 8, before and X[j + u TL] after,
// in registers; between passes the line goes through shared memory (element i
// at i + i/8, which keeps the strided stores of a pass free of bank
// conflicts), the two halves of its buffer in turn so that a pass costs one
// barrier of the line.
// The grids that use it have a block or two per SM and every launch runs its code
// once, so time is the chain of instructions of a thread and of exposed
// latencies: eight elements a thread are the shortest chain without more
// passes (16 x 8 points on eight threads in two register steps took 2100 to 2500
// cycles per line on the SM's clock), and the twiddles are in
// registers, loaded before the wait for the previous kernel.
// ---------------------------------------------------------------------------
template <int M> struct Line8 {
  static constexpr int TL = M / 8;
  static constexpr int NP = M > 512 ? 4 : (M > 64 ? 3 : 2);  // passes
  // line pitch in float2 of one half of the buffer: neighbouring lines 4 or 8 mod 16 apart
  static constexpr int P0 = M + M / 8;
  static constexpr int PITCH = TL >= 16 ? P0 + 4 - P0 % 8 : (P0 % 16 == 8 ? P0 : (P0 + 15) / 16 * 16 + (TL == 2 ? 4 : 8));
  __host__ __device__ static constexpr int ns(int p) { return 1 << (3 * p); }
  __host__ __device__ static constexpr int radix(int p) { return M / ns(p) >= 8 ? 8 : M / ns(p); }
  __device__ __forceinline__ static int at(int i) { return i + (i >> 3); }

  struct Tw {
    float2 w[NP - 1][8];  // pass p + 1, element u (1 where none)
  };
  // twM[q] = W_M^q
  __device__ __forceinline__ static void load(Tw& tw, int j, const float2* __restrict__ twM) {
#pragma unroll
    for (int p = 1; p < NP; ++p) {
      const int R = radix(p), NS = ns(p), B = 8 / R;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = u / B, jj = j + (u % B) * TL;
        tw.w[p - 1][u] = t ? __ldg(&twM[t * (jj % NS) * (M / (NS * R))]) : make_float2(1.f, 0.f);
      }
    }
  }
  // barrier of N threads that hold whole lines (id: a barrier of their own where they span warps)
  template <int N> __device__ __forceinline__ static void sync(int id) {
    if (N <= 32)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(N) : "memory");
  }
  // `a`, `b`: the line in the two halves of the buffer; the first exchange goes
  // through a.  N: threads that a barrier joins (TL, or more that run in step).
  template <bool INV, int N = TL>
  __device__ __forceinline__ static void run(float2 (&v)[8], float2* a, float2* b, int j, const Tw& tw, int id) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int R = radix(p), NS = ns(p), B = 8 / R;
      if (p > 0) {
        float2* L = (p & 1) ? a : b;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float2 x = L[at(j + u * TL)];
          const float2 w = tw.w[p - 1][u];
          v[u] = u < B ? x : (INV ? cmul(x, cconj(w)) : cmul(x, w));
        }
      }
#pragma unroll
      for (int q = 0; q < B; ++q) {
        float2 t[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i < R) t[i] = v[(q + i * B) & 7];
        if (R == 8) Dft<8, INV, float2>::run(t);
        if (R == 4) Dft<4, INV, float2>::run(t);
        if (R == 2) Dft<2, INV, float2>::run(t);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i < R) v[(q + i * B) & 7] = t[i];
      }
      if (p + 1 < NP) {
        // (a pass before the last is of radix 8)
        float2* L = (p & 1) ? b : a;
        const int base = j / NS * NS * 8 + j % NS;
#pragma unroll
        for (int u = 0; u < 8; ++u) L[at(base + u * NS)] = v[u];
        sync<N>(id);
      }
    }
  }
};

// Few-row x block of R rows of M = Px/2 points: lines (r, c), line l on threads
// l TL .. l TL + TL - 1; the threads that only fill the last warp have scratch lines.
template <int M, int R> struct RowShape {
  typedef Line8<M> L;
  static constexpr int NF = (3 * R * L::TL + 31) / 32 * 32;  // threads of the transforms
  static constexpr int lines = NF / L::TL;
  static constexpr int half = lines * L::PITCH;  // float2 of one half of the buffer
  static constexpr size_t smem = sizeof(float2) * 2 * half;
  static_assert(smem <= kMaxSmem, "row kernel shared memory");
  // (called before a launch of a kernel with these blocks; only M = 1024 needs it)
  template <typename K> static mx_status allow(K kernel) {
    return smem > 48 * 1024 ? allow_smem(kernel, smem) : MX_OK;
  }
  // The buffer half that the inverse rows are left in and the forward rows are
  // read from: after an inverse's exchanges the next half in turn, and the one after that.
  static constexpr int h_at = (L::NP - 1) & 1, m_at = L::NP & 1;
};

// A thread's constants in a row block: the passes' twiddles and W_2M^(j + u TL)
// (tables that nothing writes after set-up: loaded before pdl_wait).
template <int M> struct RowTw {
  typename Line8<M>::Tw t;
  float2 p[8];
  __device__ __forceinline__ void load(const float2* __restrict__ twM, const float2* __restrict__ twP) {
    const int j = threadIdx.x % Line8<M>::TL;
    Line8<M>::load(t, j, twM);
#pragma unroll
    for (int u = 0; u < 8; ++u) p[u] = __ldg(&twP[j + u * Line8<M>::TL]);
  }
};

// The c2r transforms of rows row0 .. row0 + R - 1 into shared memory (xi_cell),
// ending with a block barrier.  With Z[k] = S + i t, S = X[k] + conj X[M-k],
// t = conj(W_2M^k) (X[k] - conj X[M-k]); element n of the inverse transform of Z
// is cells 2n (real part) and 2n + 1 (imaginary part).
template <int M, int R>
__device__ __forceinline__ void xi_rows(float2* sm, const float2* w1, const Grid& g, int row0,
                                        const RowTw<M>& tw) {
  typedef RowShape<M, R> RS;
  typedef Line8<M> L;
  const int tid = threadIdx.x;
  if (tid < RS::NF) {
    const int line = tid / L::TL, j = tid % L::TL;
    const int row = row0 + line / 3;
    const bool in = line < 3 * R && row < g.ny * g.nz;
    const float2* X = w1 + ((long)(line % 3) * g.nz * g.ny + (in ? row : 0)) * g.Hx;
    float2 v[8], b[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = in ? X[j + u * L::TL] : make_float2(0.f, 0.f);
      b[u] = in ? X[M - j - u * L::TL] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float2 bc = cconj(b[u]);
      const float2 Sv = cadd(v[u], bc);
      const float2 t = cmul(cconj(tw.p[u]), csub(v[u], bc));
      v[u] = make_float2(Sv.x - t.y, Sv.y + t.x);
    }
    float2* A = sm + line * L::PITCH;
    L::template run<true>(v, A, A + RS::half, j, tw.t, 1 + line);
    // cells i < nx <= M need n < M/2
    float2* H = A + RS::h_at * RS::half;
#pragma unroll
    for (int u = 0; u < 4; ++u) H[L::at(j + u * L::TL)] = v[u];
  }
  __syncthreads();
}

// H_demag of cell i of row r from the c2r lines
template <int M, int R>
__device__ __forceinline__ float3 xi_cell(const float2* sm, int r, int i) {
  constexpr int P = Line8<M>::PITCH;
  const float* L = reinterpret_cast<const float*>(sm + RowShape<M, R>::h_at * RowShape<M, R>::half + 3 * r * P +
                                                  Line8<M>::at(i >> 1)) + (i & 1);
  return make_float3(L[0], L[2 * P], L[4 * P]);
}

// Cell i < nx of row r of Ms m for xf_rows.
template <int M, int R>
__device__ __forceinline__ void xf_cell(float2* sm, int r, int i, float3 v) {
  constexpr int P = Line8<M>::PITCH;
  float* L = reinterpret_cast<float*>(sm + RowShape<M, R>::m_at * RowShape<M, R>::half + 3 * r * P +
                                      Line8<M>::at(i >> 1)) + (i & 1);
  L[0] = v.x;
  L[2 * P] = v.y;
  L[4 * P] = v.z;
}

// xf_cell for the cells of rows row0 .. row0 + R - 1 of Ms m in global memory.
template <int M, int R, int NT>
__device__ __forceinline__ void xf_stage(float2* sm, const float4* m, const Grid& g, float ms,
                                         const float* __restrict__ ms_map, int row0) {
  const int total = min(R, g.ny * g.nz - row0) * g.nx;
#pragma unroll 4
  for (int e = threadIdx.x; e < total; e += NT) {
    const int r = R == 1 ? 0 : e / g.nx, i = e - r * g.nx;
    const long idx = (long)row0 * g.nx + e;
    const float4 a = m[idx];
    const float s = ms_map ? __ldg(&ms_map[idx]) : ms;
    xf_cell<M, R>(sm, r, i, make_float3(s * a.x, s * a.y, s * a.z));
  }
}

// The r2c transforms of the rows in shared memory (xf_cell; a block barrier
// first) into w1: with E = (Z[k] + conj Z[M-k]) / 2, O = (Z[k] - conj Z[M-k]) / 2i
// and T = W_2M^k O, X[k] = E + T and X[M-k] = conj(E - T).
template <int M, int R>
__device__ __forceinline__ void xf_rows(float2* sm, const Grid& g, float2* __restrict__ w1, int row0,
                                        const RowTw<M>& tw) {
  typedef RowShape<M, R> RS;
  typedef Line8<M> L;
  const int tid = threadIdx.x;
  __syncthreads();
  if (tid >= RS::NF) return;
  const int line = tid / L::TL, j = tid % L::TL;
  const int row = row0 + line / 3;
  float2* A = sm + line * L::PITCH;
  float2* in = A + RS::m_at * RS::half;
  float2* other = A + (1 - RS::m_at) * RS::half;
  float2 v[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int n = j + u * L::TL;
    // zero outside the grid: cells 2n, 2n + 1 >= nx
    const float2 x = u < 4 ? in[L::at(n)] : make_float2(0.f, 0.f);
    v[u] = make_float2(2 * n < g.nx ? x.x : 0.f, 2 * n + 1 < g.nx ? x.y : 0.f);
  }
  L::template run<false>(v, other, in, j, tw.t, 1 + line);
  // the last exchange went through `other` (two or four passes) or `in` (three)
  float2* z = L::NP == 3 ? other : in;
#pragma unroll
  for (int u = 4; u < 8; ++u) z[L::at(j + u * L::TL)] = v[u];
  L::template sync<L::TL>(1 + line);
  if (line >= 3 * R || row >= g.ny * g.nz) return;
  float2* X = w1 + ((long)(line % 3) * g.nz * g.ny + row) * g.Hx;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int k = j + u * L::TL;
    const float2 zk = v[u];
    const float2 zc = cconj(k == 0 ? zk : z[L::at(M - k)]);
    const float2 Ev = cscale(cadd(zk, zc), 0.5f);
    const float2 D = csub(zk, zc);
    const float2 T = cmul(tw.p[u], make_float2(0.5f * D.y, -0.5f * D.x));
    X[k] = cadd(Ev, T);
    X[M - k] = cconj(csub(Ev, T));
  }
  if (j == 0) X[M / 2] = cconj(v[4]);
}

// x blocks of a grid: many rows per block (many_rows(M) of them) unless that
// gives fewer than kMinBlocks blocks; then the few-row blocks below.
constexpr int kMinBlocks = 2 * 152;
inline int many_rows(int half) {
  switch (half) {
    case 1024: return 2;
    case 512:
    case 256: return 4;
    case 128:
    case 64: return 8;
    default: return 32;
  }
}
inline bool few_rows(const Grid& g) {
  const int rb = many_rows(g.Px / 2);
  return (g.ny * g.nz + rb - 1) / rb < kMinBlocks;
}

// Calls f.template run<M, R, NT>() for the few-row x configuration of M = Px/2
// (R rows and NT threads per block; where the grid fills its padding, a cell or two
// per thread); MX_ERR_UNSUPPORTED for sizes without one.
template <class F> mx_status few_rows_dispatch(int half, F& f) {
  switch (half) {
    case 1024: return f.template run<1024, 1, 384>();
    case 512: return f.template run<512, 1, 256>();
    case 256: return f.template run<256, 1, 256>();
    case 128: return f.template run<128, 1, 128>();
    case 64: return f.template run<64, 2, 128>();
    case 32: return f.template run<32, 4, 128>();
    case 16: return f.template run<16, 4, 64>();
    default: return MX_ERR_UNSUPPORTED;
  }
}

}  // namespace mx
