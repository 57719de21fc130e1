// Compile-time-sized x passes of the demag convolution (the same arithmetic as demag.cu's generic
// kernels, Sec. II-B: zero-padded FFT convolution with the tensor spectrum),
// built from the register FFTs of regfft.cuh.
//
//   xf    r2c along x: M = Px/2 complex points per row (the real row packed
//         as z[n] = x[2n] + i x[2n+1]) plus the split step.
//   xi    c2r along x, cells i < nx written as float4.
#include "common.cuh"
#include "fft.cuh"
#include "kernels.cuh"
#include "local.cuh"
#include "regfft.cuh"
#include "xrows.cuh"

namespace mx {

template <int M, int R, int NT>
__global__ void __launch_bounds__(NT) xf_kernel(const float4* m, Grid g, float ms,
                                                const float* __restrict__ ms_map, float2* __restrict__ w1,
                                                const float2* __restrict__ twM, const float2* __restrict__ twP) {
  extern __shared__ float2 sm[];
  RowTw<M> tw;
  tw.load(twM, twP);
  pdl_wait_next();
  xf_stage<M, R, NT>(sm, m, g, ms, ms_map, blockIdx.x * R);
  xf_rows<M, R>(sm, g, w1, blockIdx.x * R, tw);
}

// ---------------------------------------------------------------------------
// x inverse (c2r).
// ---------------------------------------------------------------------------
template <int M, int R, int NT>
__global__ void __launch_bounds__(NT) xi_kernel(const float2* w1, Grid g, float4* __restrict__ hd,
                                                const float2* __restrict__ twM, const float2* __restrict__ twP) {
  extern __shared__ float2 sm[];
  const int row0 = blockIdx.x * R;
  RowTw<M> tw;
  tw.load(twM, twP);
  pdl_wait_next();
  xi_rows<M, R>(sm, w1, g, row0, tw);
  const int total = min(R, g.ny * g.nz - row0) * g.nx;
  for (int e = threadIdx.x; e < total; e += NT) {
    const int r = R == 1 ? 0 : e / g.nx, i = e - r * g.nx;
    const float3 h = xi_cell<M, R>(sm, r, i);
    hd[(long)row0 * g.nx + e] = make_float4(h.x, h.y, h.z, 0.f);
  }
}

// ---------------------------------------------------------------------------
// Many-row x passes: R rows per block, lines (r, c) of M = E*S points by S
// threads each, every thread transforming (NT = 3 R S), the product twiddles
// and a bank-conflict-free line layout in shared memory.  Outputs and inputs
// of the r2c split come in pairs (k, M - k): with E = (Z[k] + conj Z[M-k]) / 2,
// O = (Z[k] - conj Z[M-k]) / 2i and T = W_2M^k O, X[k] = E + T and X[M-k] =
// conj(E - T), one twiddle for two outputs; the inverse pairs them the same way.
// Measured at 128^3 against the lines of the few-row blocks with R = 8 (scattered
// twiddle loads, two-way bank conflicts): forward 73 -> 27 us, inverse 66 -> 33.
// ---------------------------------------------------------------------------
template <int E, int S, int R> struct ManyRows {
  static constexpr int M = E * S, NT = 3 * R * S, lines = 3 * R;
  static constexpr size_t smem = sizeof(float2) * (BankLine<E, S>::size(lines) + M);
};

template <int E, int S, int R>
__global__ void __launch_bounds__(3 * R * S) xf_many_kernel(const float4* m, Grid g, float ms,
                                                           const float* __restrict__ ms_map, float2* __restrict__ w1,
                                                           const float2* __restrict__ twM,
                                                           const float2* __restrict__ twP) {
  typedef BankLine<E, S> BL;
  constexpr int M = E * S, NT = 3 * R * S, HALF = M / 2;
  extern __shared__ __align__(16) float2 sm[];
  float2* twS = sm + BL::size(3 * R);
  const int nrows = g.ny * g.nz, row0 = blockIdx.x * R, tid = threadIdx.x;
  for (int q = tid; q < M; q += NT) twS[q] = __ldg(&twM[(q % S) * (q / S)]);
  pdl_wait();
  // nx <= M, so only the packed pairs n < M/2 are non-zero
  constexpr int NLD = (R * HALF + NT - 1) / NT;
  float4 va[NLD], vb[NLD];
  float sa[NLD], sb[NLD];
#pragma unroll
  for (int j = 0; j < NLD; ++j) {
    const int e = tid + j * NT;
    const int r = e / HALF, i = 2 * (e % HALF);
    const bool in = e < R * HALF && row0 + r < nrows;
    const long cell = (long)(row0 + r) * g.nx + i;
    va[j] = in && i < g.nx ? m[cell] : make_float4(0.f, 0.f, 0.f, 0.f);
    vb[j] = in && i + 1 < g.nx ? m[cell + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
    sa[j] = sb[j] = ms;
    if (ms_map) {
      if (in && i < g.nx) sa[j] = __ldg(&ms_map[cell]);
      if (in && i + 1 < g.nx) sb[j] = __ldg(&ms_map[cell + 1]);
    }
  }
#pragma unroll
  for (int j = 0; j < NLD; ++j) {
    const int e = tid + j * NT;
    if (e >= R * HALF) break;
    const int r = e / HALF, n = e % HALF;
    float2 *l0 = sm + BL::off(3 * r), *l1 = sm + BL::off(3 * r + 1), *l2 = sm + BL::off(3 * r + 2);
    l0[n] = make_float2(sa[j] * va[j].x, sb[j] * vb[j].x);
    l1[n] = make_float2(sa[j] * va[j].y, sb[j] * vb[j].y);
    l2[n] = make_float2(sa[j] * va[j].z, sb[j] * vb[j].z);
    l0[n + HALF] = l1[n + HALF] = l2[n + HALF] = make_float2(0.f, 0.f);
  }
  __syncthreads();
  line_fft<E, S, false, true, true>(sm + BL::off(tid / S), tid % S, twS);
  __syncthreads();
  const long cs = (long)nrows * g.Hx;
#pragma unroll 4
  for (int e = tid; e < 3 * R * (HALF + 1); e += NT) {
    const int line = e / (HALF + 1), k = e % (HALF + 1);
    const int row = row0 + line / 3;
    if (row >= nrows) break;
    const float2* L = sm + BL::off(line);
    float2* dst = w1 + (line % 3) * cs + (long)row * g.Hx;
    const float2 a = L[k];
    if (k == 0) {
      dst[0] = make_float2(a.x + a.y, 0.f);
      dst[M] = make_float2(a.x - a.y, 0.f);
    } else if (k == HALF) {
      dst[k] = cconj(a);
    } else {
      const float2 b = L[M - k];
      const float2 Ev = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
      const float2 O = make_float2(0.5f * (a.y + b.y), -0.5f * (a.x - b.x));
      const float2 t = cmul(__ldg(&twP[k]), O);
      dst[k] = cadd(Ev, t);
      dst[M - k] = cconj(csub(Ev, t));
    }
  }
}

template <int E, int S, int R>
__global__ void __launch_bounds__(3 * R * S) xi_many_kernel(const float2* w1, Grid g,
                                                           float4* __restrict__ hd, const float2* __restrict__ twM,
                                                           const float2* __restrict__ twP) {
  typedef BankLine<E, S> BL;
  constexpr int M = E * S, NT = 3 * R * S, HALF = M / 2;
  extern __shared__ __align__(16) float2 sm[];
  float2* twS = sm + BL::size(3 * R);
  const int nrows = g.ny * g.nz, row0 = blockIdx.x * R, tid = threadIdx.x;
  for (int q = tid; q < M; q += NT) twS[q] = __ldg(&twM[(q % S) * (q / S)]);
  pdl_wait();
  const long cs = (long)nrows * g.Hx;
  constexpr int NE = 3 * R * (HALF + 1), kB = 5;  // pairs per thread in flight
  for (int e0 = tid; e0 < NE; e0 += NT * kB) {
    float2 a[kB], b[kB];
#pragma unroll
    for (int u = 0; u < kB; ++u) {
      const int e = e0 + u * NT;
      const int line = e / (HALF + 1), k = e % (HALF + 1);
      const int row = row0 + line / 3;
      a[u] = b[u] = make_float2(0.f, 0.f);
      if (e < NE && row < nrows) {
        const float2* X = w1 + (line % 3) * cs + (long)row * g.Hx;
        a[u] = X[k];
        b[u] = cconj(X[M - k]);
      }
    }
#pragma unroll
    for (int u = 0; u < kB; ++u) {
      const int e = e0 + u * NT;
      if (e >= NE) break;
      const int line = e / (HALF + 1), k = e % (HALF + 1);
      float2* L = sm + BL::off(line);
      const float2 Sv = cadd(a[u], b[u]);
      const float2 t = cmul(cconj(__ldg(&twP[k])), csub(a[u], b[u]));
      L[k] = make_float2(Sv.x - t.y, Sv.y + t.x);
      if (k > 0 && k < HALF) L[M - k] = make_float2(Sv.x + t.y, t.x - Sv.y);
    }
  }
  __syncthreads();
  line_fft<E, S, true, true, true>(sm + BL::off(tid / S), tid % S, twS);
  __syncthreads();
  // cells 2n and 2n + 1 of row r are the real and imaginary parts of element n
#pragma unroll 3
  for (int e = tid; e < R * HALF; e += NT) {
    const int r = e / HALF, n = e % HALF, i = 2 * n;
    if (row0 + r >= nrows || i >= g.nx) continue;
    const float2 hx = sm[BL::off(3 * r) + n], hy = sm[BL::off(3 * r + 1) + n], hz = sm[BL::off(3 * r + 2) + n];
    float4* row = hd + (long)(row0 + r) * g.nx;
    row[i] = make_float4(hx.x, hy.x, hz.x, 0.f);
    if (i + 1 < g.nx) row[i + 1] = make_float4(hx.y, hy.y, hz.y, 0.f);
  }
}

// ---------------------------------------------------------------------------
// Row kernel of the RK4 and Euler steps: the inverse x pass of rows row0 .. row0 + R - 1,
// the local stage of `mode` on their cells (demag term from shared memory),
// and, with `xf_next`, the forward x pass of the stage output io.out for the
// next stage, so that between the y/z passes of two stages there is one
// kernel and H_demag never goes to global memory.  A thread's cells and their
// neighbours are loaded before the inverse transforms; the stage output goes to
// the forward transforms through shared memory.  The four stages share one piece
// of code (their coefficients are run-time values): a launch runs it once per block.
// Bound: its chain of dependent phases (load, two to four FFT passes, the cell
// update, the passes again, store).  us per stage of kernel and
// boundaries, the row kernel's and the y/z kernel's changes together (RK4 step / 4), with
// the kernels before: 512x128 15.7 -> 11.0, 128x128 9.5 -> 6.9, 1000x100 31.7 -> 19.3,
// 201x77x3 15.6 -> 13.6, 32x32x4 7.4 -> 6.9.
// ---------------------------------------------------------------------------
// HEFF: the effective field of io.m instead of a stage.
template <int M, int R, int NT, bool DMI, bool HEFF>
__global__ void __launch_bounds__(NT) xr_kernel(float2* __restrict__ w1, Grid g, const float2* __restrict__ twM,
                                                const float2* __restrict__ twP, StageIO io, LocalCoef c, int mode,
                                                int xf_next, float4* __restrict__ hd_out, int* flag) {
  extern __shared__ float2 sm[];
  constexpr int KC = (R * M + NT - 1) / NT;  // cells per thread (nx <= M)
  const int row0 = blockIdx.x * R;
  RowTw<M> tw;
  tw.load(twM, twP);
  const int total = min(R, g.ny * g.nz - row0) * g.nx;
  pdl_wait_next();
  StageCell v[KC];
#pragma unroll
  for (int u = 0; u < KC; ++u) {
    const int e = threadIdx.x + u * NT;
    if (e < total) {
      const int r = R == 1 ? 0 : e / g.nx;
      const int row = row0 + r;
      v[u].load(io, g, c, e - r * g.nx, row % g.ny, row / g.ny, (long)row0 * g.nx + e, HEFF ? (int)LM_HEFF : mode);
    }
  }
  xi_rows<M, R>(sm, w1, g, row0, tw);
#pragma unroll
  for (int u = 0; u < KC; ++u) {
    const int e = threadIdx.x + u * NT;
    if (e < total) {
      const int r = R == 1 ? 0 : e / g.nx, i = e - r * g.nx;
      const long idx = (long)row0 * g.nx + e;
      const float3 h = xi_cell<M, R>(sm, r, i);
      if (HEFF) {
        v[u].template heff<DMI>(io, c, idx, h, flag);
        continue;
      }
      if (hd_out) hd_out[idx] = make_float4(h.x, h.y, h.z, 0.f);
      const float3 out = v[u].template stage<DMI>(io, c, idx, h, mode, flag);
      xf_cell<M, R>(sm, r, i, v[u].ms * out);
    }
  }
  if (!HEFF && xf_next) xf_rows<M, R>(sm, g, w1, row0, tw);
}

// ---------------------------------------------------------------------------
// y transform + tensor multiply + inverse y of a one-z-plane spectrum
// (Pz == 1, so no z transform and N_xz = N_yz = 0), T kx columns per block,
// small-grid layout w1[c][y][kx].  The Py-point transform of the zero-padded
// column (inputs y < ny <= Py/2) splits into its even outputs, a Py/2-point
// FFT of x, and its odd outputs, a Py/2-point FFT of x W_Py^y; the inverse
// restricted to y < ny is even + W_Py^-y odd.  Lines (c, t, half) of LH =
// Py/2 points are Line8 transforms; the tensor entries and every twiddle are
// loaded before the wait.  Bound: as the row kernel, its chain of phases (load,
// transforms, multiply, transforms, store).  256 threads: with 384 the film of
// 512x128 cells takes 46.0 us per step, with 256 44.0.
// ---------------------------------------------------------------------------
// PAIR: a column's two lines are on the same threads, one after the other.
template <int LH, int T, bool PAIR> struct Yz2d {
  typedef Line8<LH> L;
  static constexpr int NF = ((PAIR ? 3 : 6) * T * L::TL + 31) / 32 * 32;  // threads of the transforms
  static constexpr int NT = NF > 256 ? NF : 256;                         // (the others only load, multiply and store)
  static constexpr int MB = NT <= 384 ? 2 : 1;                            // blocks per SM
  static constexpr int lines = (PAIR ? 2 : 1) * NF / L::TL;
  static constexpr int half = lines * L::PITCH;
  static constexpr size_t smem = sizeof(float2) * 2 * half;
};

template <int LH, int T, bool PAIR>
__global__ void __launch_bounds__(Yz2d<LH, T, PAIR>::NT, Yz2d<LH, T, PAIR>::MB)
    yz2d_kernel(float2* __restrict__ w1, Grid g, const float* __restrict__ nhat, const float2* __restrict__ twH,
                const float2* __restrict__ twPy) {
  typedef Yz2d<LH, T, PAIR> D;
  typedef Line8<LH> L;
  constexpr int NT = D::NT, PITCH = L::PITCH;
  extern __shared__ __align__(16) float2 sm[];
  const int kx0 = blockIdx.x * T;
  const int tid = threadIdx.x;
  const int ny = g.ny;
  const long wc = (long)g.ny * g.Hx;  // component stride of w1 (one z plane)
  // line (c T + t) 2 + h; with PAIR the first of the thread's two
  const int line = PAIR ? 2 * (tid / L::TL) : tid / L::TL, j = tid % L::TL;
  const bool fft = tid < D::NF, odd = line & 1;
  typename L::Tw tw;
  float2 wy[8];  // W_Py^(j + u TL)
  if (fft) {
    L::load(tw, j, twH);
#pragma unroll
    for (int u = 0; u < 8; ++u) wy[u] = PAIR || odd ? __ldg(&twPy[j + u * L::TL]) : make_float2(1.f, 0.f);
  }
  // this thread's tensor entries for the multiply below
  constexpr int NMUL = T * 2 * LH, KM = (NMUL + NT - 1) / NT;
  const long no = (long)g.Hx * g.Oy * g.Oz;
  float4 nt[KM];
#pragma unroll
  for (int u = 0; u < KM; ++u) {
    const int e = tid + u * NT;
    const int q = e % LH, h = (e / LH) % 2, t = e / (2 * LH);
    const int kx = kx0 + t;
    nt[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < NMUL && kx < g.Hx) {
      const int ky = 2 * q + h;
      const bool fy = ky > (g.Py >> 1);
      const long o = (long)(fy ? g.Py - ky : ky) * g.Hx + kx;
      nt[u] = make_float4(__ldg(&nhat[o]), __ldg(&nhat[no + o]), __ldg(&nhat[2 * no + o]),
                          (fy ? -1.f : 1.f) * __ldg(&nhat[3 * no + o]));
    }
  }
  pdl_wait_next();  // the tables are constants; w1 is the previous kernel's
  // column (c, t) to the slot of its even line in the second half; every load of a thread in flight at once
  float2* sb = sm + D::half;
  {
    constexpr int NE = 3 * T * LH, KB = (NE + NT - 1) / NT;
    float2 v[KB];
#pragma unroll
    for (int u = 0; u < KB; ++u) {
      const int e = tid + u * NT;
      const int t = e % T, y = (e / T) % LH, c = e / (T * LH);
      const int kx = kx0 + t;
      v[u] = (e < NE && y < ny && kx < g.Hx) ? w1[c * wc + (long)y * g.Hx + kx] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < KB; ++u) {
      const int e = tid + u * NT;
      if (e >= NE) break;
      const int t = e % T, y = (e / T) % LH, c = e / (T * LH);
      sb[(c * T + t) * 2 * PITCH + L::at(y)] = v[u];
    }
  }
  __syncthreads();
  // Where both lines' threads read the column, the barriers of the transforms are theirs together.
  constexpr int NB = PAIR ? L::TL : 2 * L::TL;
  constexpr int NZ = L::NP == 3 ? 0 : 1;  // half that the forward outputs go to (the one free after the exchanges)
  float2* A = sm + line * PITCH;
  float2* Z = A + NZ * D::half;
  float2* O = A + (1 - NZ) * D::half;
  if (fft) {
    const float2* x = sb + (line & ~1) * PITCH;
    float2 v[8], xo[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = x[L::at(j + u * L::TL)];
      if (PAIR) xo[u] = cmul(v[u], wy[u]);
      if (!PAIR && odd) v[u] = cmul(v[u], wy[u]);
    }
    L::template run<false, NB>(v, A, A + D::half, j, tw, 1 + line / 2);
#pragma unroll
    for (int u = 0; u < 8; ++u) Z[L::at(j + u * L::TL)] = v[u];
    if (PAIR) {
      L::template run<false, NB>(xo, A + PITCH, A + PITCH + D::half, j, tw, 1 + line / 2);
#pragma unroll
      for (int u = 0; u < 8; ++u) Z[PITCH + L::at(j + u * L::TL)] = xo[u];
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < KM; ++u) {
    const int e = tid + u * NT;
    const int q = e % LH, h = (e / LH) % 2, t = e / (2 * LH);
    if (e >= NMUL) continue;
    const float nxx = nt[u].x, nyy = nt[u].y, nzz = nt[u].z, nxy = nt[u].w;
    float2* px = sm + NZ * D::half + (t * 2 + h) * PITCH + L::at(q);
    float2* py = px + 2 * T * PITCH;
    float2* pz = py + 2 * T * PITCH;
    const float2 mx = *px, my = *py, mz = *pz;
    *px = make_float2(nxx * mx.x + nxy * my.x, nxx * mx.y + nxy * my.y);
    *py = make_float2(nxy * mx.x + nyy * my.x, nxy * mx.y + nyy * my.y);
    *pz = make_float2(nzz * mz.x, nzz * mz.y);
  }
  __syncthreads();
  constexpr int NO = L::NP == 3 ? 1 - NZ : NZ;  // half that the inverse outputs go to
  if (fft) {
    float2 v[8], vo[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = Z[L::at(j + u * L::TL)];
    L::template run<true, NB>(v, O, Z, j, tw, 1 + line / 2);
    if (PAIR) {
#pragma unroll
      for (int u = 0; u < 8; ++u) vo[u] = Z[PITCH + L::at(j + u * L::TL)];
      L::template run<true, NB>(vo, O + PITCH, Z + PITCH, j, tw, 1 + line / 2);
    }
    float2* out = A + NO * D::half;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (PAIR) v[u] = cadd(v[u], cmul(vo[u], cconj(wy[u])));
      out[L::at(j + u * L::TL)] = !PAIR && odd ? cmul(v[u], cconj(wy[u])) : v[u];
    }
  }
  __syncthreads();
  for (int e = tid; e < 3 * T * LH; e += NT) {
    const int t = e % T, y = (e / T) % LH, c = e / (T * LH);
    const int kx = kx0 + t;
    if (y >= ny || kx >= g.Hx) continue;
    const float2* H = sm + NO * D::half + (c * T + t) * 2 * PITCH + L::at(y);
    w1[c * wc + (long)y * g.Hx + kx] = PAIR ? H[0] : cadd(H[0], H[PITCH]);
  }
}

template <int LH, int T, bool PAIR>
static mx_status yz2d_run(mx_ctx* ctx, cudaStream_t st, bool setup) {
  typedef Yz2d<LH, T, PAIR> D;
  if (setup) {
    MX_CUDA_TRY(cudaFuncSetAttribute(yz2d_kernel<LH, T, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)D::smem));
    return MX_OK;
  }
  launch_pdl(yz2d_kernel<LH, T, PAIR>, dim3((ctx->g.Hx + T - 1) / T), dim3(D::NT), D::smem, st, ctx->w1, ctx->g,
             ctx->nhat, ctx->tw_yh, ctx->tw_y);
  return launch_check("yz2d_kernel");
}

// ---------------------------------------------------------------------------
// The same on many columns of 256 or 512 points: the register line FFT of
// E x S points, S threads a line, so that a block is a quarter of the threads and
// half the shared memory of Line8's, and one wave holds twice the columns.
// ---------------------------------------------------------------------------
template <int E, int S, int T, int NT>
__global__ void __launch_bounds__(NT) yz2d_wide_kernel(float2* __restrict__ w1, Grid g, const float* __restrict__ nhat,
                                                  const float2* __restrict__ twH,
                                                  const float2* __restrict__ twPy) {
  constexpr int LH = E * S;
  constexpr int PITCH = LineFft<E, S>::kPitch;
  constexpr int NF = 6 * T * S;  // threads of the FFT phases
  static_assert(NT >= NF && NT % 32 == 0 && NF % 32 == 0, "yz2d thread count");
  extern __shared__ __align__(16) float2 sm[];
  float2* twS = sm + 6 * T * PITCH;  // W_LH^(s k) at [k S + s]
  float2* twS2 = twS + LH;           // W_Py^y, y < LH
  const int kx0 = blockIdx.x * T;
  const int tid = threadIdx.x;
  const int ny = g.ny;
  const long wc = (long)g.ny * g.Hx;  // component stride of w1 (one z plane)
  for (int q = tid; q < LH; q += NT) {
    twS[q] = __ldg(&twH[(q % S) * (q / S)]);
    twS2[q] = __ldg(&twPy[q]);
  }
  // this thread's tensor entries for the multiply below (constants, so read
  // while the previous kernel may still run)
  constexpr int NMUL = T * 2 * LH, KM = (NMUL + NT - 1) / NT;
  const long no = (long)g.Hx * g.Oy * g.Oz;
  float4 nt[KM];
#pragma unroll
  for (int u = 0; u < KM; ++u) {
    const int e = tid + u * NT;
    const int j = e % LH, h = (e / LH) % 2, t = e / (2 * LH);
    const int kx = kx0 + t;
    nt[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < NMUL && kx < g.Hx) {
      const int ky = 2 * j + h;
      const bool fy = ky > (g.Py >> 1);
      const long o = (long)(fy ? g.Py - ky : ky) * g.Hx + kx;
      nt[u] = make_float4(__ldg(&nhat[o]), __ldg(&nhat[no + o]), __ldg(&nhat[2 * no + o]),
                          (fy ? -1.f : 1.f) * __ldg(&nhat[3 * no + o]));
    }
  }
  pdl_wait();  // the tables are constants; w1 is the previous kernel's
  __syncthreads();
  // line (c, t, h) at ((c T + t) 2 + h) PITCH; every load of a thread in flight at once
  {
    constexpr int NE = 3 * T * LH, KB = (NE + NT - 1) / NT;
    float2 v[KB];
#pragma unroll
    for (int u = 0; u < KB; ++u) {
      const int e = tid + u * NT;
      const int t = e % T, y = (e / T) % LH, c = e / (T * LH);
      const int kx = kx0 + t;
      v[u] = (e < NE && y < ny && kx < g.Hx) ? w1[c * wc + (long)y * g.Hx + kx] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < KB; ++u) {
      const int e = tid + u * NT;
      if (e >= NE) break;
      const int t = e % T, y = (e / T) % LH, c = e / (T * LH);
      float2* L = sm + ((c * T + t) * 2) * PITCH;
      L[y] = v[u];
      L[PITCH + y] = cmul(v[u], twS2[y]);
    }
  }
  __syncthreads();
  if (tid < NF) line_fft<E, S, false, true, true>(sm + (tid / S) * PITCH, tid % S, twS);
  __syncthreads();
#pragma unroll
  for (int u = 0; u < KM; ++u) {
    const int e = tid + u * NT;
    const int j = e % LH, h = (e / LH) % 2, t = e / (2 * LH);
    const int kx = kx0 + t;
    if (e >= NMUL || kx >= g.Hx) continue;
    const float nxx = nt[u].x, nyy = nt[u].y, nzz = nt[u].z, nxy = nt[u].w;
    float2* px = sm + ((0 * T + t) * 2 + h) * PITCH + j;
    float2* py = sm + ((1 * T + t) * 2 + h) * PITCH + j;
    float2* pz = sm + ((2 * T + t) * 2 + h) * PITCH + j;
    const float2 mx = *px, my = *py, mz = *pz;
    *px = make_float2(nxx * mx.x + nxy * my.x, nxx * mx.y + nxy * my.y);
    *py = make_float2(nxy * mx.x + nyy * my.x, nxy * mx.y + nyy * my.y);
    *pz = make_float2(nzz * mz.x, nzz * mz.y);
  }
  __syncthreads();
  if (tid < NF) line_fft<E, S, true, true, true>(sm + (tid / S) * PITCH, tid % S, twS);
  __syncthreads();
  for (int e = tid; e < 3 * T * LH; e += NT) {
    const int t = e % T, y = (e / T) % LH, c = e / (T * LH);
    const int kx = kx0 + t;
    if (y >= ny || kx >= g.Hx) continue;
    const float2* L = sm + ((c * T + t) * 2) * PITCH;
    w1[c * wc + (long)y * g.Hx + kx] = cadd(L[y], cmul(L[PITCH + y], cconj(twS2[y])));
  }
}

// 384 threads per block at least: most of them only load, multiply and store
template <int E, int S, int T>
static mx_status yz2d_wide_run(mx_ctx* ctx, cudaStream_t st, bool setup) {
  constexpr int NT = 6 * T * S > 384 ? 6 * T * S : 384;
  const size_t sm = sizeof(float2) * (6 * T * LineFft<E, S>::kPitch + 2 * E * S);
  if (setup) {
    MX_CUDA_TRY(cudaFuncSetAttribute(yz2d_wide_kernel<E, S, T, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    return MX_OK;
  }
  launch_pdl(yz2d_wide_kernel<E, S, T, NT>, dim3((ctx->g.Hx + T - 1) / T), dim3(NT), sm, st, ctx->w1, ctx->g,
             ctx->nhat, ctx->tw_yh, ctx->tw_y);
  return launch_check("yz2d_wide_kernel");
}

// One column per block where that is at most a block per SM, two where two blocks
// per SM hold them all, else four with their lines in pairs.  At 513
// columns of 128 points one, two and four (paired): RK4 step 48.2, 44.2, 56.1 us; at
// 1025 one, two, four and four paired: 93.4, 83.0, 81.0, 77.2; at 129 columns one and
// two (the block before): yz 8.4 and 9.3 us.
template <int LH>
static mx_status yz2d_cols(mx_ctx* ctx, cudaStream_t st, bool setup) {
  if (setup) {
    MX_TRY((yz2d_run<LH, 1, false>(ctx, st, true)));
    MX_TRY((yz2d_run<LH, 2, false>(ctx, st, true)));
    return yz2d_run<LH, 4, true>(ctx, st, true);
  }
  if (ctx->g.Hx <= kSMs) return yz2d_run<LH, 1, false>(ctx, st, false);
  if (ctx->g.Hx <= 4 * kSMs) return yz2d_run<LH, 2, false>(ctx, st, false);
  return yz2d_run<LH, 4, true>(ctx, st, false);
}

// Rows of up to 32 points: two columns per block, eight where those would be more
// than four blocks per SM.  RK4 step of 200x30 cells with
// two 25.5 us, with eight 28.7; of 64x30 23.4 and 27.6.
template <int LH>
static mx_status yz2d_short(mx_ctx* ctx, cudaStream_t st, bool setup) {
  if (setup) {
    MX_TRY((yz2d_run<LH, 2, false>(ctx, st, true)));
    return yz2d_run<LH, 8, false>(ctx, st, true);
  }
  return ctx->g.Hx <= 8 * kSMs ? yz2d_run<LH, 2, false>(ctx, st, false) : yz2d_run<LH, 8, false>(ctx, st, false);
}

// Long columns: RK4 step of 300x300 cells (513 columns of 512 points) with the wide
// kernel 114.6 us, else 139; of 640x160 (1025 of 256) 134.6 and 145; of 500x250 (513 of
// 256) 76.8 and 83.0; of 250x250 (257 of 256) the other way, 48.1 and 46.1; yz of
// 200x500 (257 of 512) 16.1 us and 19.3, of 128x500 (129 of 512) 14.7 and 13.3.
bool yz2d_wide(const Grid& g) { return (g.Py == 1024 && g.Hx > kSMs) || (g.Py == 512 && g.Hx > 2 * kSMs); }

static mx_status yz2d_dispatch(mx_ctx* ctx, cudaStream_t st, bool setup) {
  const bool wide = yz2d_wide(ctx->g);
  switch (ctx->g.Py / 2) {
    case 512: return wide ? yz2d_wide_run<32, 16, 2>(ctx, st, setup) : yz2d_run<512, 1, false>(ctx, st, setup);
    case 256:
      if (wide) return yz2d_wide_run<16, 16, 2>(ctx, st, setup);
      return ctx->g.Hx <= kSMs ? yz2d_run<256, 1, false>(ctx, st, setup) : yz2d_run<256, 2, true>(ctx, st, setup);
    case 128: return yz2d_cols<128>(ctx, st, setup);
    case 64: return yz2d_cols<64>(ctx, st, setup);
    case 32: return yz2d_short<32>(ctx, st, setup);
    case 16: return yz2d_short<16>(ctx, st, setup);
    default: return MX_ERR_UNSUPPORTED;
  }
}

mx_status yz2d_pass(mx_ctx* ctx, cudaStream_t st) { return yz2d_dispatch(ctx, st, false); }

// ---------------------------------------------------------------------------
// Dispatch
// ---------------------------------------------------------------------------
template <int M, int R, int NT>
static mx_status run_xf(mx_ctx* ctx, const float4* m, cudaStream_t st) {
  const Grid& g = ctx->g;
  MX_TRY((RowShape<M, R>::allow(xf_kernel<M, R, NT>)));
  launch_pdl(xf_kernel<M, R, NT>, dim3((g.ny * g.nz + R - 1) / R), dim3(NT), RowShape<M, R>::smem, st, m, g,
             (float)ctx->p.Ms, ctx->ms_map, ctx->w1, ctx->tw_m, ctx->tw_x);
  return launch_check("xf_kernel");
}

template <int M, int R, int NT>
static mx_status run_xi(mx_ctx* ctx, float4* hd, cudaStream_t st) {
  const Grid& g = ctx->g;
  MX_TRY((RowShape<M, R>::allow(xi_kernel<M, R, NT>)));
  launch_pdl(xi_kernel<M, R, NT>, dim3((g.ny * g.nz + R - 1) / R), dim3(NT), RowShape<M, R>::smem, st, ctx->w1, g, hd,
             ctx->tw_m, ctx->tw_x);
  return launch_check("xi_kernel");
}

template <int M, int R, int NT>
static mx_status run_xr(mx_ctx* ctx, int mode, const StageIO& io, bool xf_next, float4* hd_out, cudaStream_t st) {
  const Grid& g = ctx->g;
  const LocalCoef c = local_coef(ctx);
  auto k = mode == LM_HEFF ? (c.dmi ? xr_kernel<M, R, NT, true, true> : xr_kernel<M, R, NT, false, true>)
                           : (c.dmi ? xr_kernel<M, R, NT, true, false> : xr_kernel<M, R, NT, false, false>);
  MX_TRY((RowShape<M, R>::allow(k)));
  launch_pdl(k, dim3((g.ny * g.nz + R - 1) / R), dim3(NT), RowShape<M, R>::smem, st, ctx->w1, g, ctx->tw_m, ctx->tw_x, io, c, mode, xf_next ? 1 : 0, hd_out,
             ctx->flag);
  return launch_check("xr_kernel");
}

// x pass for M = Px/2 (returns MX_ERR_UNSUPPORTED when no specialisation fits).
// Each size has a many-rows-per-block variant and a few-rows one; grids whose
// row count would give fewer than two blocks per SM with the first take the
// second.

template <int E, int S, int R>
static mx_status run_many(mx_ctx* ctx, const float4* m, float4* hd, bool inverse, cudaStream_t st, bool setup) {
  typedef ManyRows<E, S, R> D;
  if (setup) {
    MX_CUDA_TRY(cudaFuncSetAttribute(xf_many_kernel<E, S, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)D::smem));
    MX_CUDA_TRY(cudaFuncSetAttribute(xi_many_kernel<E, S, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)D::smem));
    return MX_OK;
  }
  const Grid& g = ctx->g;
  const dim3 grid((g.ny * g.nz + R - 1) / R);
  if (inverse)
    launch_pdl(xi_many_kernel<E, S, R>, grid, dim3(D::NT), D::smem, st, ctx->w1, g, hd, ctx->tw_m, ctx->tw_x);
  else
    launch_pdl(xf_many_kernel<E, S, R>, grid, dim3(D::NT), D::smem, st, m, g, (float)ctx->p.Ms, ctx->ms_map, ctx->w1,
               ctx->tw_m, ctx->tw_x);
  return launch_check(inverse ? "xi_many_kernel" : "xf_many_kernel");
}

// The few-row kernels, by few_rows_dispatch.
struct RowLaunch {
  mx_ctx* ctx;
  const float4* m;
  float4* hd;
  bool inverse;
  cudaStream_t st;
  template <int M, int R, int NT> mx_status run() {
    return inverse ? run_xi<M, R, NT>(ctx, hd, st) : run_xf<M, R, NT>(ctx, m, st);
  }
};

// The row kernel exists for the few-row blocks only (grids whose x passes
// have fewer blocks than two per SM, where the step is bound by its kernel
// boundaries); MX_ERR_UNSUPPORTED for the others.
struct XrLaunch {
  mx_ctx* ctx;
  int mode;
  const StageIO* io;
  bool xf_next;
  float4* hd_out;
  cudaStream_t st;
  bool setup;
  template <int M, int R, int NT> mx_status run() {
    return setup ? MX_OK : run_xr<M, R, NT>(ctx, mode, *io, xf_next, hd_out, st);
  }
};

static mx_status xr_pass(mx_ctx* ctx, int mode, const StageIO& io, bool xf_next, float4* hd_out, cudaStream_t st,
                         bool setup) {
  if (!few_rows(ctx->g)) return MX_ERR_UNSUPPORTED;
  XrLaunch L{ctx, mode, &io, xf_next, hd_out, st, setup};
  return few_rows_dispatch(ctx->g.Px / 2, L);
}

static mx_status x_pass(mx_ctx* ctx, const float4* m, float4* hd, bool inverse, cudaStream_t st, bool setup) {
  if (!setup && few_rows(ctx->g)) {
    RowLaunch L{ctx, m, hd, inverse, st};
    return few_rows_dispatch(ctx->g.Px / 2, L);
  }
  switch (ctx->g.Px / 2) {
    case 1024: return run_many<32, 32, 2>(ctx, m, hd, inverse, st, setup);
    case 512: return run_many<32, 16, 4>(ctx, m, hd, inverse, st, setup);
    case 256: return run_many<16, 16, 4>(ctx, m, hd, inverse, st, setup);
    case 128: return run_many<16, 8, 8>(ctx, m, hd, inverse, st, setup);
    case 64: return run_many<8, 8, 8>(ctx, m, hd, inverse, st, setup);
    case 32: return run_many<8, 4, 32>(ctx, m, hd, inverse, st, setup);
    case 16: return run_many<4, 4, 32>(ctx, m, hd, inverse, st, setup);
    default: return MX_ERR_UNSUPPORTED;
  }
}

mx_status fast_setup(mx_ctx* ctx) {
  MX_TRY(upload_w32());
  ctx->fast_x = ctx->p.demag_path != MX_DEMAG_GENERIC &&
                x_pass(ctx, nullptr, nullptr, false, nullptr, true) == MX_OK &&
                x_pass(ctx, nullptr, nullptr, true, nullptr, true) == MX_OK;
  ctx->yz2d = ctx->fused_yz && ctx->g.Pz == 1 && yz2d_dispatch(ctx, nullptr, true) == MX_OK;
  StageIO none{};
  ctx->xrow = ctx->fast_x && xr_pass(ctx, LM_RK4_S0, none, false, nullptr, nullptr, true) == MX_OK;
  clear_error();
  return MX_OK;
}

mx_status fast_row_stage(mx_ctx* ctx, int mode, const StageIO& io, bool xf_next, float4* hd_out, cudaStream_t st) {
  if (mode == LM_RHS) {
    set_error("fast_row_stage: bad mode");
    return MX_ERR_INVALID_ARG;
  }
  return xr_pass(ctx, mode, io, xf_next, hd_out, st, false);
}

mx_status fast_x_pass(mx_ctx* ctx, const float4* m, float4* hd, bool inverse, cudaStream_t st) {
  return x_pass(ctx, m, hd, inverse, st, false);
}

}  // namespace mx
