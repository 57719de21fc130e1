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
// The P-point transform of a zero-padded line (inputs n < P/2) splits into its
// even outputs, a P/2-point FFT of x, and its odd outputs, a P/2-point FFT of
// x W_P^n; the inverse restricted to n < P/2 is even + W_P^-n odd.  So the
// padding is never transformed, and each half line is a register line FFT of E
// x S points by S threads that never leaves its warp (the size-generic passes
// meet two block barriers per radix pass and transform the zero half too).
//
// Bound: shared-memory and instruction throughput of the line FFTs, then the
// passes over w2 (read and written once by each of zc and yf/yi).  Measured at
// 128^3 (256^3 padded): MEASURED_DEEP
#include <math.h>

#include "common.cuh"
#include "fft.cuh"
#include "kernels.cuh"
#include "regfft.cuh"
#include "zcol.cuh"

namespace mx {

// Shared-memory line layout.  A half-warp of a line FFT covers H = 16 / S
// lines, and the load and store loops put T neighbouring lines on neighbouring
// lanes.  Both stay free of bank conflicts when the H lines of a group start
// 2 S words apart modulo 32 and the groups 4 words apart.
template <int E, int S> struct DeepLine {
  static constexpr int PITCH = LineFft<E, S>::kPitch;
  static constexpr int H = S >= 16 ? 1 : 16 / S;
  // shift of lines within a group (a multiple of 2 S words apart), and the group's stride
  static constexpr bool SHIFT = (S == 8 && PITCH % 16 == 0) || (S == 4 && PITCH % 16 == 8);
  static constexpr int GROUP = H * PITCH + (SHIFT ? 16 : 0) + 2;
  __device__ __forceinline__ static int off(int l) {
    const int r = l % H;
    return l / H * GROUP + r * PITCH + (SHIFT ? (S == 8 ? 8 * r : 4 * (r >> 1)) : 0);
  }
  static constexpr int size(int lines) { return (lines + H - 1) / H * GROUP; }  // float2 of `lines` lines
};

// Block shape of a half length L = P/2: E x S points per line, T kx columns.
template <int L> struct DeepShape;
template <> struct DeepShape<16> { static constexpr int E = 4, S = 4, T = 16; };
template <> struct DeepShape<32> { static constexpr int E = 8, S = 4, T = 16; };
template <> struct DeepShape<64> { static constexpr int E = 8, S = 8, T = 8; };
template <> struct DeepShape<128> { static constexpr int E = 16, S = 8, T = 8; };
template <> struct DeepShape<256> { static constexpr int E = 16, S = 16, T = 4; };
template <> struct DeepShape<512> { static constexpr int E = 32, S = 16, T = 4; };

// twiddle tables of a half length: twS[k S + s] = W_L^(s k), twS2[n] = W_2L^n
template <int L, int S, int NT>
__device__ __forceinline__ void deep_tables(float2* twS, float2* twS2, const float2* __restrict__ twL,
                                            const float2* __restrict__ twP) {
  for (int q = threadIdx.x; q < L; q += NT) {
    twS[q] = __ldg(&twL[(q % S) * (q / S)]);
    twS2[q] = __ldg(&twP[q]);
  }
}

// ---------------------------------------------------------------------------
// y passes: lines (t, half) of one (c, z) plane.
// ---------------------------------------------------------------------------
template <int L, bool INV>
__global__ void __launch_bounds__(2 * DeepShape<L>::T * DeepShape<L>::S)
    deep_y_kernel(const float2* __restrict__ in, float2* __restrict__ out, Grid g, const float2* __restrict__ twL,
                  const float2* __restrict__ twP) {
  typedef DeepShape<L> D;
  typedef DeepLine<D::E, D::S> DL;
  constexpr int T = D::T, S = D::S, NT = 2 * T * S;
  extern __shared__ __align__(16) float2 sm[];
  float2* twS = sm + DL::size(2 * T);
  float2* twS2 = twS + L;
  const int ntile = (g.Hx + T - 1) / T;
  const int kx0 = (blockIdx.x % ntile) * T;
  const int cz = blockIdx.x / ntile;
  const int tid = threadIdx.x, ny = g.ny, Hx = g.Hx;
  const int t = tid % T;  // NT is a multiple of T: a thread keeps its column
  const bool ok = kx0 + t < Hx;
  deep_tables<L, S, NT>(twS, twS2, twL, twP);
  pdl_wait();
  __syncthreads();
  // line (half, t) at off(half T + t)
  float2* l0 = sm + DL::off(t);
  float2* l1 = sm + DL::off(T + t);
  constexpr int ST = NT / T;  // rows between a thread's elements
  if (!INV) {
    const float2* src = in + (long)cz * ny * Hx + kx0 + t;
    constexpr int KB = L / ST < 8 ? L / ST : 8;
#pragma unroll
    for (int y0 = tid / T; y0 < L; y0 += ST * KB) {
      float2 v[KB];
#pragma unroll
      for (int u = 0; u < KB; ++u) {
        const int y = y0 + u * ST;
        v[u] = (ok && y < ny) ? __ldg(&src[(long)y * Hx]) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < KB; ++u) {
        const int y = y0 + u * ST;
        l0[y] = v[u];
        l1[y] = cmul(v[u], twS2[y]);
      }
    }
  } else {
    const float2* src = in + (long)cz * g.Py * Hx + kx0 + t;
    constexpr int KB = 2 * L / ST < 8 ? 2 * L / ST : 8;
#pragma unroll
    for (int y0 = tid / T; y0 < 2 * L; y0 += ST * KB) {
      float2 v[KB];
#pragma unroll
      for (int u = 0; u < KB; ++u) v[u] = ok ? __ldg(&src[(long)(y0 + u * ST) * Hx]) : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < KB; ++u) {
        const int ky = y0 + u * ST;
        ((ky & 1) ? l1 : l0)[ky >> 1] = v[u];
      }
    }
  }
  __syncthreads();
  line_fft<D::E, S, INV, true, true>(sm + DL::off(tid / S), tid % S, twS);
  __syncthreads();
  if (!ok) return;
  if (!INV) {
    float2* dst = out + (long)cz * g.Py * Hx + kx0 + t;
#pragma unroll 8
    for (int ky = tid / T; ky < 2 * L; ky += ST) dst[(long)ky * Hx] = ((ky & 1) ? l1 : l0)[ky >> 1];
  } else {
    float2* dst = out + (long)cz * ny * Hx + kx0 + t;
#pragma unroll 4
    for (int y = tid / T; y < ny; y += ST) dst[(long)y * Hx] = cadd(l0[y], cmul(l1[y], cconj(twS2[y])));
  }
}

// ---------------------------------------------------------------------------
// z pass: lines (half, c, t) at one ky.
// ---------------------------------------------------------------------------
template <int L>
__global__ void __launch_bounds__(6 * DeepShape<L>::T * DeepShape<L>::S, L <= 256 ? 2 : 1)
    deep_z_kernel(float2* __restrict__ w2, Grid g, const float* __restrict__ nhat, const float2* __restrict__ twL,
                  const float2* __restrict__ twP) {
  typedef DeepShape<L> D;
  typedef DeepLine<D::E, D::S> DL;
  constexpr int T = D::T, S = D::S, NT = 6 * T * S;
  static_assert(NT % (3 * T) == 0, "a thread keeps its line pair");
  extern __shared__ __align__(16) float2 sm[];
  float2* twS = sm + DL::size(6 * T);
  float2* twS2 = twS + L;
  const int ntile = (g.Hx + T - 1) / T;
  const int kx0 = (blockIdx.x % ntile) * T;
  // ky and Py - ky read the same octant rows: neighbours in launch order
  const int q = blockIdx.x / ntile;
  const int ky = (q % 2 == 0) ? q / 2 : g.Py - 1 - q / 2;
  const int tid = threadIdx.x, nz = g.nz, Hx = g.Hx;
  const long zs = (long)g.Py * Hx;  // from z to z + 1
  const int t = tid % T, c = (tid / T) % 3;
  const bool ok = kx0 + t < Hx;
  deep_tables<L, S, NT>(twS, twS2, twL, twP);
  pdl_wait();
  __syncthreads();
  float2* l0 = sm + DL::off(c * T + t);
  float2* l1 = sm + DL::off((3 + c) * T + t);
  float2* col = w2 + (long)c * nz * zs + (long)ky * Hx + kx0 + t;
  constexpr int ST = NT / (3 * T);  // planes between a thread's elements
  {
    constexpr int KB = L / ST < 8 ? L / ST : 8;
#pragma unroll
    for (int z0 = tid / (3 * T); z0 < L; z0 += ST * KB) {
      float2 v[KB];
#pragma unroll
      for (int u = 0; u < KB; ++u) {
        const int z = z0 + u * ST;
        v[u] = (ok && z < nz) ? col[(long)z * zs] : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < KB; ++u) {
        const int z = z0 + u * ST;
        l0[z] = v[u];
        l1[z] = cmul(v[u], twS2[z]);
      }
    }
  }
  __syncthreads();
  line_fft<D::E, S, false, true, true>(sm + DL::off(tid / S), tid % S, twS);
  __syncthreads();
  {
    // kz and its mirror P - kz (same half) share an octant entry: half 0 has
    // kz = 0, 2, .., L, half 1 kz = 1, 3, .., L - 1; neighbouring lanes take
    // neighbouring kz of one half (contiguous entries)
    const bool fy = ky > (g.Py >> 1);
    const int qy = fy ? g.Py - ky : ky;
    const float sy = fy ? -1.f : 1.f;
    for (int e = tid; e < T * (L + 1); e += NT) {
      const int tt = e / (L + 1), k = e % (L + 1);
      if (kx0 + tt >= Hx) break;
      const int h = k > L / 2 ? 1 : 0;
      const int j = h ? k - L / 2 - 1 : k;
      const ZEntry n = z_entry(nhat + plane_octant_index(g, kx0 + tt, 0, 2 * j + h, qy), 0, 0);
      float2* p0 = sm + DL::off((3 * h + 0) * T + tt);
      float2* p1 = sm + DL::off((3 * h + 1) * T + tt);
      float2* p2 = sm + DL::off((3 * h + 2) * T + tt);
      const float nxy = sy * n.t23.y, nyz = sy * n.t45.y;
      {
        float2 a = p0[j], b = p1[j], d = p2[j];
        tensor_apply(a, b, d, n.t01.x, n.t01.y, n.t23.x, nxy, n.t45.x, nyz);
        p0[j] = a;
        p1[j] = b;
        p2[j] = d;
      }
      const int jm = L - j - h;  // 2 jm + h = P - kz
      if (jm != j && jm < L) {
        float2 a = p0[jm], b = p1[jm], d = p2[jm];
        tensor_apply(a, b, d, n.t01.x, n.t01.y, n.t23.x, nxy, -n.t45.x, -nyz);
        p0[jm] = a;
        p1[jm] = b;
        p2[jm] = d;
      }
    }
  }
  __syncthreads();
  line_fft<D::E, S, true, true, true>(sm + DL::off(tid / S), tid % S, twS);
  __syncthreads();
  if (!ok) return;
#pragma unroll 4
  for (int z = tid / (3 * T); z < nz; z += ST) col[(long)z * zs] = cadd(l0[z], cmul(l1[z], cconj(twS2[z])));
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
template <int L, bool INV> static mx_status deep_y_run(mx_ctx* ctx, cudaStream_t st, bool setup) {
  typedef DeepShape<L> D;
  const size_t sm = sizeof(float2) * (DeepLine<D::E, D::S>::size(2 * D::T) + 2 * L);
  if (setup) {
    MX_CUDA_TRY(cudaFuncSetAttribute(deep_y_kernel<L, INV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    return MX_OK;
  }
  const Grid& g = ctx->g;
  launch_pdl(deep_y_kernel<L, INV>, dim3(3 * g.nz * ((g.Hx + D::T - 1) / D::T)), dim3(2 * D::T * D::S), sm, st,
             INV ? ctx->w2 : ctx->w1, INV ? ctx->w1 : ctx->w2, g, ctx->tw_yh, ctx->tw_y);
  return launch_check("deep_y_kernel");
}

template <int L> static mx_status deep_z_run(mx_ctx* ctx, cudaStream_t st, bool setup) {
  typedef DeepShape<L> D;
  const size_t sm = sizeof(float2) * (DeepLine<D::E, D::S>::size(6 * D::T) + 2 * L);
  if (setup) {
    MX_CUDA_TRY(cudaFuncSetAttribute(deep_z_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    return MX_OK;
  }
  const Grid& g = ctx->g;
  launch_pdl(deep_z_kernel<L>, dim3(g.Py * ((g.Hx + D::T - 1) / D::T)), dim3(6 * D::T * D::S), sm, st, ctx->w2, g,
             ctx->nhat, ctx->tw_zh, ctx->tw_z);
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
