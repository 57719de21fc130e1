// y and z passes of the demag convolution on deep grids (Sec. II-B: zero-padded
// FFT convolution with the tensor spectrum), where a kx plane fits neither one
// block nor a cluster: three kernels between the x passes, on the small-grid
// spectrum w1[c][z][y][kx] and w2[c][z][ky][kx].
//
//   yf   forward y: T kx columns of one (c, z) plane per block; w1 -> w2
//   zc   forward z, 3x3 tensor multiply, inverse z of T kx columns at one ky,
//        all three components; w2 in place
//   yi   inverse y, rows y < ny; w2 -> w1
//
// The P-point transform of a zero-padded line (inputs n < P/2 = L) splits into
// its even outputs (half h = 0), an L-point FFT of x, and its odd outputs (h =
// 1), an L-point FFT of x W_P^n; the inverse restricted to n < L is even +
// W_P^-n odd.  So the padding is never transformed.
//
// A half line of L = E S points is transformed by S threads in two register
// steps with one exchange through shared memory.  Thread s takes x[s + S n]
// straight from global memory, an E-point FFT over n, the twiddle W_P^(s (2 k1
// + h)) (which holds the odd half's W_P^s; its W_2E^n goes in before the FFT),
// and after the exchange S-point FFTs give X[k1 + E k2] for its k1 = s + S j.
// The spectrum is used where it lies: the inverse starts with the S-point FFTs
// over k2 of the same registers and ends with E-point ones, whose outputs s + S
// n go straight to global memory, so natural order is never formed.  In zc a
// thread holds the three components of its wavenumbers and multiplies in
// registers.  Neighbouring lanes take neighbouring kx (T of them contiguous).
//
// Bound: instruction issue (128^3: 76 M warp instructions in zc, 57 % of the
// issue slots), shared memory (51 % of its wavefronts) and the latency of the
// phases between barriers; a first version
// that kept lines in natural order moved every value through shared memory 14
// times where this one does 5 (9 in zc of long lines).  Measured at 128^3 (256^3
// padded), against the size-generic passes: yf 36 us (266), zc 113 us (884; 136
// in natural order), yi 41 us (330).
#include <math.h>

#include "common.cuh"
#include "fft.cuh"
#include "kernels.cuh"
#include "regfft.cuh"
#include "zcol.cuh"

namespace mx {

// Block shape of a half length L = P/2: E x S points per line, T kx columns.
// The exchange holds element (k1, s) of a line at k1 S + (s xor k1 mod S): a
// half-warp (T neighbouring lines, then s) meets no bank twice, whether its
// lanes share k1 (first steps) or each takes its own row (second steps), with
// the line pitch L + 16 / T (odd for T = 16).  Padding the rows instead would
// take 12 % more shared memory and one block per SM in zc.
template <int L> struct DeepShape;
template <> struct DeepShape<16> { static constexpr int E = 4, S = 4, T = 16, PITCH = 17; };
template <> struct DeepShape<32> { static constexpr int E = 8, S = 4, T = 16, PITCH = 33; };
template <> struct DeepShape<64> { static constexpr int E = 8, S = 8, T = 8, PITCH = 66; };
template <> struct DeepShape<128> { static constexpr int E = 16, S = 8, T = 8, PITCH = 130; };
template <> struct DeepShape<256> { static constexpr int E = 16, S = 16, T = 4, PITCH = 260; };
template <> struct DeepShape<512> { static constexpr int E = 32, S = 16, T = 4, PITCH = 516; };

template <int L> struct Deep {
  typedef DeepShape<L> D;
  static constexpr int E = D::E, S = D::S, T = D::T, J = E / S, PITCH = D::PITCH;
  static constexpr int NT = 2 * T * S;          // threads: t fastest, then s, then h
  static constexpr int TW = 2 * E * (S + 1);    // twiddle table: W_P^(s (2 k1 + h)) at (h E + k1)(S + 1) + s
  static constexpr size_t smem(int lines) { return sizeof(float2) * (TW + (size_t)lines * PITCH); }

  __device__ __forceinline__ static void table(float2* tw, const float2* __restrict__ twP) {
    for (int q = threadIdx.x; q < 2 * E * S; q += NT) {
      const int s = q % S, k1 = (q / S) % E, h = q / (E * S);
      tw[(h * E + k1) * (S + 1) + s] = __ldg(&twP[s * (2 * k1 + h)]);
    }
  }
  // W_2E^n
  __device__ __forceinline__ static float2 w2e(int n, const float2* __restrict__ twP) {
    if constexpr (2 * E <= 32)
      return c_w32[n * (32 / (2 * E))];
    else
      return __ldg(&twP[S * n]);
  }
  __device__ __forceinline__ static int at(int k1, int s) { return k1 * S + (s ^ (k1 & (S - 1))); }
  // first step of the forward transform: v[n] = x[s + S n] -> row k1, column s of the exchange
  __device__ __forceinline__ static void fwd1(float2 (&v)[E], float2* line, int s, int h, const float2* tw,
                                              const float2* __restrict__ twP) {
    if (h) {
#pragma unroll
      for (int n = 1; n < E; ++n) v[n] = cmul(v[n], w2e(n, twP));
    }
    RegFft<E, false>::run(v);
    const float2* w = tw + h * E * (S + 1) + s;
#pragma unroll
    for (int k = 0; k < E; ++k) line[at(k, s)] = cmul(v[k], w[k * (S + 1)]);
  }
  // second step: v[j S + k2] = X[k1 + E k2], k1 = s + S j
  __device__ __forceinline__ static void fwd2(float2 (&v)[E], const float2* line, int s) {
#pragma unroll
    for (int j = 0; j < J; ++j) {
#pragma unroll
      for (int q = 0; q < S; ++q) v[j * S + q] = line[at(s + S * j, q)];
      RegFft<S, false>::run(&v[j * S]);
    }
  }
  // first step of the inverse, from the same arrangement, into the same rows of the exchange
  __device__ __forceinline__ static void inv1(float2 (&v)[E], float2* line, int s, int h, const float2* tw) {
#pragma unroll
    for (int j = 0; j < J; ++j) {
      RegFft<S, true>::run(&v[j * S]);
      const float2* w = tw + (h * E + s + S * j) * (S + 1);
#pragma unroll
      for (int q = 0; q < S; ++q) line[at(s + S * j, q)] = cmul(v[j * S + q], cconj(w[q]));
    }
  }
  // second step: v[n] = this half's share of x[s + S n]
  __device__ __forceinline__ static void inv2(float2 (&v)[E], const float2* line, int s, int h,
                                              const float2* __restrict__ twP) {
#pragma unroll
    for (int k = 0; k < E; ++k) v[k] = line[at(k, s)];
    RegFft<E, true>::run(v);
    if (h) {
#pragma unroll
      for (int n = 1; n < E; ++n) v[n] = cmul(v[n], cconj(w2e(n, twP)));
    }
  }
  // the halves finish E/2 of the outputs each: thread h hands over those of the other half ...
  __device__ __forceinline__ static void give(const float2 (&v)[E], float2* line, int s, int h) {
#pragma unroll
    for (int n = 0; n < E / 2; ++n) line[at(n, s)] = h ? v[n] : v[n + E / 2];
  }
  // ... and adds what the other handed over to its own: o[n] = x[s + S (n + h E/2)]
  __device__ __forceinline__ static void take(const float2 (&v)[E], const float2* other, int s, int h,
                                              float2 (&o)[E / 2]) {
#pragma unroll
    for (int n = 0; n < E / 2; ++n) o[n] = cadd(h ? v[n + E / 2] : v[n], other[at(n, s)]);
  }
};

// ---------------------------------------------------------------------------
// y passes of one (c, z) plane: line (h, t) at (h T + t) PITCH.
// ---------------------------------------------------------------------------
template <int L>
__global__ void __launch_bounds__(Deep<L>::NT)
    deep_yf_kernel(const float2* w1, float2* w2, Grid g, const float2* __restrict__ twP) {
  typedef Deep<L> D;
  constexpr int E = D::E, S = D::S, T = D::T;
  extern __shared__ __align__(16) float2 sm[];
  const int ntile = (g.Hx + T - 1) / T;
  const int cz = blockIdx.x / ntile, kx = (blockIdx.x % ntile) * T + threadIdx.x % T;
  const int t = threadIdx.x % T, s = (threadIdx.x / T) % S, h = threadIdx.x / (T * S);
  const bool ok = kx < g.Hx;
  D::table(sm, twP);
  pdl_wait();
  const float2* src = w1 + (long)cz * g.ny * g.Hx + kx;
  float2 v[E];
#pragma unroll
  for (int n = 0; n < E; ++n) {
    const int y = s + S * n;
    v[n] = ok && y < g.ny ? src[(long)y * g.Hx] : make_float2(0.f, 0.f);
  }
  __syncthreads();  // the table
  float2* line = sm + D::TW + (h * T + t) * D::PITCH;
  D::fwd1(v, line, s, h, sm, twP);
  __syncthreads();
  D::fwd2(v, line, s);
  if (!ok) return;
  float2* dst = w2 + (long)cz * g.Py * g.Hx + kx;
#pragma unroll
  for (int j = 0; j < D::J; ++j)
#pragma unroll
    for (int q = 0; q < S; ++q) dst[(long)(2 * (s + S * j + E * q) + h) * g.Hx] = v[j * S + q];
}

template <int L>
__global__ void __launch_bounds__(Deep<L>::NT)
    deep_yi_kernel(const float2* w2, float2* w1, Grid g, const float2* __restrict__ twP) {
  typedef Deep<L> D;
  constexpr int E = D::E, S = D::S, T = D::T;
  extern __shared__ __align__(16) float2 sm[];
  const int ntile = (g.Hx + T - 1) / T;
  const int cz = blockIdx.x / ntile, kx = (blockIdx.x % ntile) * T + threadIdx.x % T;
  const int t = threadIdx.x % T, s = (threadIdx.x / T) % S, h = threadIdx.x / (T * S);
  const bool ok = kx < g.Hx;
  D::table(sm, twP);
  pdl_wait();
  const float2* src = w2 + (long)cz * g.Py * g.Hx + kx;
  float2 v[E];
#pragma unroll
  for (int j = 0; j < D::J; ++j)
#pragma unroll
    for (int q = 0; q < S; ++q)
      v[j * S + q] = ok ? src[(long)(2 * (s + S * j + E * q) + h) * g.Hx] : make_float2(0.f, 0.f);
  __syncthreads();
  float2* line = sm + D::TW + (h * T + t) * D::PITCH;
  D::inv1(v, line, s, h, sm);
  __syncthreads();
  D::inv2(v, line, s, h, twP);
  D::give(v, line, s, h);  // (this thread's own column of the exchange, read above)
  __syncthreads();
  float2 o[E / 2];
  D::take(v, sm + D::TW + ((1 - h) * T + t) * D::PITCH, s, h, o);
  float2* dst = w1 + (long)cz * g.ny * g.Hx + kx;
#pragma unroll
  for (int n = 0; n < E / 2; ++n) {
    const int y = s + S * (n + h * (E / 2));
    if (ok && y < g.ny) dst[(long)y * g.Hx] = o[n];
  }
}

// ---------------------------------------------------------------------------
// z pass at one ky: line (h, c, t) at ((h 3 + c) T + t) PITCH.
// ---------------------------------------------------------------------------
template <int L>
__global__ void __launch_bounds__(Deep<L>::NT, 5)
    deep_z_kernel(float2* w2, Grid g, const float* __restrict__ nhat, const float2* __restrict__ twP) {
  typedef Deep<L> D;
  constexpr int E = D::E, S = D::S, T = D::T;
  extern __shared__ __align__(16) float2 sm[];
  const int ntile = (g.Hx + T - 1) / T;
  // ky and Py - ky read the same octant rows: neighbours in launch order
  const int b = blockIdx.x / ntile;
  const int ky = (b % 2 == 0) ? b / 2 : g.Py - 1 - b / 2;
  const int kx = (blockIdx.x % ntile) * T + threadIdx.x % T;
  const int t = threadIdx.x % T, s = (threadIdx.x / T) % S, h = threadIdx.x / (T * S);
  const bool ok = kx < g.Hx;
  const long zs = (long)g.Py * g.Hx;  // from z to z + 1
  const bool fy = ky > (g.Py >> 1);
  const float2* oct = reinterpret_cast<const float2*>(nhat) +
                      plane_octant_index(g, ok ? kx : 0, 0, 0, fy ? g.Py - ky : ky) / 2;
  D::table(sm, twP);
  pdl_wait();
  __syncthreads();
  float2* line = sm + D::TW + (h * 3 * T + t) * D::PITCH;
  constexpr int CS = T * D::PITCH;  // from component to component
  float2* col = w2 + (long)ky * g.Hx + kx;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float2 v[E];
#pragma unroll
    for (int n = 0; n < E; ++n) {
      const int z = s + S * n;
      v[n] = ok && z < g.nz ? col[((long)c * g.nz + z) * zs] : make_float2(0.f, 0.f);
    }
    D::fwd1(v, line + c * CS, s, h, sm, twP);
  }
  __syncthreads();
  {
    float2 v[3][E];
#pragma unroll
    for (int c = 0; c < 3; ++c) D::fwd2(v[c], line + c * CS, s);
    const float sy = fy ? -1.f : 1.f;
#pragma unroll
    for (int j = 0; j < D::J; ++j)
#pragma unroll
      for (int q = 0; q < S; ++q) {
        const int kz = 2 * (s + S * j + E * q) + h;
        const bool fz = kz > L;
        const float2* n = oct + (long)(fz ? 2 * L - kz : kz) * 3 * g.Hx;
        const float2 t01 = __ldg(n), t23 = __ldg(n + g.Hx), t45 = __ldg(n + 2 * g.Hx);
        const int i = j * S + q;
        tensor_apply(v[0][i], v[1][i], v[2][i], t01.x, t01.y, t23.x, sy * t23.y, fz ? -t45.x : t45.x,
                     fz ? -sy * t45.y : sy * t45.y);
      }
#pragma unroll
    for (int c = 0; c < 3; ++c) D::inv1(v[c], line + c * CS, s, h, sm);
  }
  __syncthreads();
  float2 v[3][E];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    D::inv2(v[c], line + c * CS, s, h, twP);
    D::give(v[c], line + c * CS, s, h);
  }
  __syncthreads();
  const float2* other = sm + D::TW + ((1 - h) * 3 * T + t) * D::PITCH;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float2 o[E / 2];
    D::take(v[c], other + c * CS, s, h, o);
#pragma unroll
    for (int n = 0; n < E / 2; ++n) {
      const int z = s + S * (n + h * (E / 2));
      if (ok && z < g.nz) col[((long)c * g.nz + z) * zs] = o[n];
    }
  }
}

// The same with one component per thread (t fastest, then c, s, h): the spectrum
// goes back to its place in the exchange and is multiplied there.
template <int L>
__global__ void __launch_bounds__(3 * Deep<L>::NT, L <= 128 ? 3 : (L <= 256 ? 2 : 1))
    deep_z3_kernel(float2* w2, Grid g, const float* __restrict__ nhat, const float2* __restrict__ twP) {
  typedef Deep<L> D;
  constexpr int E = D::E, S = D::S, T = D::T, NT = 3 * D::NT;
  extern __shared__ __align__(16) float2 sm[];
  const int ntile = (g.Hx + T - 1) / T;
  const int b = blockIdx.x / ntile;
  const int ky = (b % 2 == 0) ? b / 2 : g.Py - 1 - b / 2;
  const int kx0 = (blockIdx.x % ntile) * T;
  const int t = threadIdx.x % T, s = (threadIdx.x / T) % S, r = threadIdx.x / (T * S);
  const int h = r / 3, c = r % 3;
  const bool ok = kx0 + t < g.Hx;
  const long zs = (long)g.Py * g.Hx;
  for (int q = threadIdx.x; q < 2 * E * S; q += NT) {
    const int qs = q % S, k1 = (q / S) % E, qh = q / (E * S);
    sm[(qh * E + k1) * (S + 1) + qs] = __ldg(&twP[qs * (2 * k1 + qh)]);
  }
  pdl_wait();
  float2* line = sm + D::TW + (r * T + t) * D::PITCH;
  float2* col = w2 + (long)c * g.nz * zs + (long)ky * g.Hx + kx0 + t;
  float2 v[E];
#pragma unroll
  for (int n = 0; n < E; ++n) {
    const int z = s + S * n;
    v[n] = ok && z < g.nz ? col[(long)z * zs] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  D::fwd1(v, line, s, h, sm, twP);
  __syncthreads();
  D::fwd2(v, line, s);
#pragma unroll
  for (int j = 0; j < D::J; ++j)
#pragma unroll
    for (int q = 0; q < S; ++q) line[D::at(s + S * j, q)] = v[j * S + q];
  __syncthreads();
  {
    const bool fy = ky > (g.Py >> 1);
    const float sy = fy ? -1.f : 1.f;
    const float2* oct = reinterpret_cast<const float2*>(nhat) +
                        plane_octant_index(g, kx0, 0, 0, fy ? g.Py - ky : ky) / 2;
    // wavenumber idx of half hh is kz = 2 idx + hh; kz and its mirror P - kz share an octant entry
    for (int e = threadIdx.x; e < T * (L + 1); e += NT) {
      const int tt = e % T, k = e / T;
      if (kx0 + tt >= g.Hx) continue;
      const int hh = k > L / 2 ? 1 : 0, i = hh ? k - L / 2 - 1 : k, im = L - i - hh;
      const float2* n = oct + (long)(2 * i + hh) * 3 * g.Hx + tt;
      const float2 t01 = __ldg(n), t23 = __ldg(n + g.Hx), t45 = __ldg(n + 2 * g.Hx);
      float2* p = sm + D::TW + (hh * 3 * T + tt) * D::PITCH;
      constexpr int CS = T * D::PITCH;
      auto mul = [&](int idx, float sz) {
        float2* o = p + D::at(idx % E, idx / E);
        float2 x = o[0], y = o[CS], z = o[2 * CS];
        tensor_apply(x, y, z, t01.x, t01.y, t23.x, sy * t23.y, sz * t45.x, sz * sy * t45.y);
        o[0] = x;
        o[CS] = y;
        o[2 * CS] = z;
      };
      mul(i, 1.f);
      if (im != i && im < L) mul(im, -1.f);
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < D::J; ++j)
#pragma unroll
    for (int q = 0; q < S; ++q) v[j * S + q] = line[D::at(s + S * j, q)];
  D::inv1(v, line, s, h, sm);
  __syncthreads();
  D::inv2(v, line, s, h, twP);
  D::give(v, line, s, h);
  __syncthreads();
  float2 o[E / 2];
  D::take(v, sm + D::TW + (((1 - h) * 3 + c) * T + t) * D::PITCH, s, h, o);
#pragma unroll
  for (int n = 0; n < E / 2; ++n) {
    const int z = s + S * (n + h * (E / 2));
    if (ok && z < g.nz) col[(long)z * zs] = o[n];
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
template <int L, bool INV> static mx_status deep_y_run(mx_ctx* ctx, cudaStream_t st, bool setup) {
  typedef Deep<L> D;
  auto k = INV ? deep_yi_kernel<L> : deep_yf_kernel<L>;
  const size_t sm = D::smem(2 * D::T);
  if (setup) {
    MX_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    return MX_OK;
  }
  const Grid& g = ctx->g;
  launch_pdl(k, dim3(3 * g.nz * ((g.Hx + D::T - 1) / D::T)), dim3(D::NT), sm, st, INV ? ctx->w2 : ctx->w1,
             INV ? ctx->w1 : ctx->w2, g, ctx->tw_y);
  return launch_check(INV ? "deep_yi_kernel" : "deep_yf_kernel");
}

template <int L> static mx_status deep_z_run(mx_ctx* ctx, cudaStream_t st, bool setup) {
  typedef Deep<L> D;
  // All three components of E <= 8 wavenumbers fit a thread's registers at five
  // blocks per SM; with E = 16 that leaves 12 to 16 warps per SM, and one
  // component per thread is faster although the spectrum passes through the
  // exchange once more (zc at 256x256x32: 88 us against 88, at 64^3 20 against
  // 21; at 128^3 133 against 119, at 30x200x200 186 against 152).
  constexpr bool SPLIT = L > 64;
  void (*k)(float2*, Grid, const float*, const float2*);
  if constexpr (SPLIT)
    k = deep_z3_kernel<L>;
  else
    k = deep_z_kernel<L>;
  const size_t sm = D::smem(6 * D::T);
  if (setup) {
    MX_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    return MX_OK;
  }
  const Grid& g = ctx->g;
  launch_pdl(k, dim3(g.Py * ((g.Hx + D::T - 1) / D::T)), dim3(SPLIT ? 3 * D::NT : D::NT), sm, st, ctx->w2, g,
             ctx->nhat, ctx->tw_z);
  return launch_check("deep_z_kernel");
}

static mx_status deep_y(mx_ctx* ctx, bool inverse, cudaStream_t st, bool setup) {
#define MX_DEEP_Y(L) \
  case L: return inverse ? deep_y_run<L, true>(ctx, st, setup) : deep_y_run<L, false>(ctx, st, setup)
  switch (ctx->g.Py / 2) {
    MX_DEEP_Y(512);
    MX_DEEP_Y(256);
    MX_DEEP_Y(128);
    MX_DEEP_Y(64);
    MX_DEEP_Y(32);
    MX_DEEP_Y(16);
    default: return MX_ERR_UNSUPPORTED;
  }
#undef MX_DEEP_Y
}

static mx_status deep_z(mx_ctx* ctx, cudaStream_t st, bool setup) {
  switch (ctx->g.Pz / 2) {
    case 512: return deep_z_run<512>(ctx, st, setup);
    case 256: return deep_z_run<256>(ctx, st, setup);
    case 128: return deep_z_run<128>(ctx, st, setup);
    case 64: return deep_z_run<64>(ctx, st, setup);
    case 32: return deep_z_run<32>(ctx, st, setup);
    case 16: return deep_z_run<16>(ctx, st, setup);
    default: return MX_ERR_UNSUPPORTED;
  }
}

mx_status deep_pass(mx_ctx* ctx, cudaStream_t st) {
  {
    ProfScope ps(ctx, KID_Y_FWD, st);
    MX_TRY(deep_y(ctx, false, st, false));
  }
  {
    ProfScope ps(ctx, KID_Z_MUL, st);
    MX_TRY(deep_z(ctx, st, false));
  }
  ProfScope ps(ctx, KID_Y_INV, st);
  return deep_y(ctx, true, st, false);
}

bool deep_setup(mx_ctx* ctx) {
  if (upload_w32() != MX_OK) return false;
  const bool ok = deep_y(ctx, false, nullptr, true) == MX_OK && deep_y(ctx, true, nullptr, true) == MX_OK &&
                  deep_z(ctx, nullptr, true) == MX_OK;
  clear_error();
  return ok;
}

}  // namespace mx
