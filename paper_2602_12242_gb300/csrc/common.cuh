// Shared definitions of libmx: context layout, error reporting, complex helpers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string>

#include "../../include/mx.h"

namespace mx {

constexpr double kPi = 3.14159265358979323846;
constexpr double kMu0 = 4e-7 * kPi;  // vacuum permeability [T m/A]
constexpr int kMaxPad = 4096;         // largest padded length per axis

// ---------------------------------------------------------------------------
// Error reporting: a per-thread message plus a status code.
// ---------------------------------------------------------------------------
void set_error(const std::string& msg);
void clear_error();

#define MX_CUDA_TRY(expr)                                                         \
  do {                                                                            \
    cudaError_t e_ = (expr);                                                      \
    if (e_ != cudaSuccess) {                                                      \
      ::mx::set_error(std::string(#expr) + ": " + cudaGetErrorString(e_));        \
      return MX_ERR_CUDA;                                                         \
    }                                                                             \
  } while (0)

#define MX_TRY(expr)                       \
  do {                                     \
    mx_status s_ = (expr);                 \
    if (s_ != MX_OK) return s_;            \
  } while (0)

// Check the launch that was just enqueued.
inline mx_status launch_check(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error(std::string(what) + ": " + cudaGetErrorString(e));
    return MX_ERR_CUDA;
  }
  return MX_OK;
}

// The dynamic shared memory a kernel may be launched with.  The limit belongs to the kernel,
// which every context shares: `bytes` is the most that any of them asks for (cut to a
// block's), never one context's own need, or the newest context would take it from the others.
constexpr size_t kMaxSmem = 227 * 1024;
template <typename K> inline mx_status allow_smem(K kernel, size_t bytes) {
  MX_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)(bytes < kMaxSmem ? bytes : kMaxSmem)));
  return MX_OK;
}

// Programmatic dependent launch.  A kernel launched by launch_pdl may be
// scheduled while the kernel before it in the stream is still running; it
// calls pdl_wait() before its first access to memory that kernel writes or
// reads (the wait returns once that kernel has completed and its writes are
// visible; without a programmatic dependency it returns at once).
//
// What such a kernel reads of the kernels before it goes through plain loads: no
// __ldg and no `const __restrict__` kernel parameter.  Those are non-coherent loads,
// which the compiler takes for constants and may move above the wait (memory clobber
// or not).  deep_yf_kernel did so behind row kernels of at most a block per SM: a deep
// grid of 26x25x20 cells took the spectrum of the stage before.  Both are for tables,
// parameters and maps that no kernel of the chain writes.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// pdl_wait_next: after the wait, a grid of at most a block per SM lets the next
// launch_pdl kernel be scheduled as soon as its last block has got here, so that
// the next one's blocks are placed and have their constants while this one runs.
// (That one waits for all of this one, and this one has waited for what ran before.)
// Used by the chains of short kernels: one field of the Fourier operator 67.9 -> 57.9 us,
// of the convolutional surrogate 27.0 -> 25.2, the adjoint of the 128x128 film 6.03 -> 5.75
// ms.  Larger grids do not: blocks placed among the last of a full grid end up unevenly
// spread (RK4 step of the 512x128 film 63 -> 72 us, of the bulk grid 1630 -> 1750).
constexpr int kSMs = 152;
__device__ __forceinline__ void pdl_wait_next() {
  pdl_wait();
  if (gridDim.x * gridDim.y * gridDim.z <= kSMs) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
inline void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);  // errors reach launch_check
}

// ---------------------------------------------------------------------------
// Complex arithmetic on float2 / double2.
// ---------------------------------------------------------------------------
template <typename C> struct real_of;
template <> struct real_of<float2> { typedef float type; };
template <> struct real_of<double2> { typedef double type; };

template <typename C> __host__ __device__ __forceinline__ C mkc(typename real_of<C>::type r, typename real_of<C>::type i) {
  C c; c.x = r; c.y = i; return c;
}
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return mkc<C>(a.x + b.x, a.y + b.y); }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return mkc<C>(a.x - b.x, a.y - b.y); }
// Single-precision sums as one packed instruction: the pipes take it in two cycles, as
// two scalar ones, but it is one issue slot, and the transforms are bound by issue and
// latency.  With the tensor multiply packed too (zcol.cuh): bulk grid y/z kernel 231 -> 211 us
// per launch and step 1606 -> 1521 us, cube step (128^3) 266 -> 257, 640x160x4 multirate step
// 415 -> 404.  The complex multiply stays scalar (packed, with its swapped operand: 1568 and
// 1607 us for the bulk step).
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  float2 d;
  asm("{.reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; add.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z;}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  float2 d;
  asm("{.reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; sub.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z;}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  return mkc<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C cconj(C a) { return mkc<C>(a.x, -a.y); }
template <typename C> __device__ __forceinline__ C cscale(C a, typename real_of<C>::type s) { return mkc<C>(a.x * s, a.y * s); }
// multiply by -i (forward) or +i (inverse)
template <bool INV, typename C> __device__ __forceinline__ C cmul_mi(C a) {
  return INV ? mkc<C>(-a.y, a.x) : mkc<C>(a.y, -a.x);
}

// ---------------------------------------------------------------------------
// Derived per-context constants passed to kernels by value.
// ---------------------------------------------------------------------------
// Bits of the context's device status flag (read and cleared by mx_sync).
constexpr int kFlagNonfinite = 1;  // a kernel produced a non-finite value
constexpr int kFlagTimeout = 2;    // a bounded wait on a bulk copy ran out

struct Grid {
  int nx, ny, nz;      // cells
  int Px, Py, Pz;      // padded lengths
  int Hx;              // Px/2 + 1 (half spectrum along x); 1 when Px == 1
  int Oy, Oz;          // Py/2 + 1, Pz/2 + 1 (octant extents of the spectrum)
  long ncell;
  int oct4;            // tensor octant layout of plane_octant_index (0, 1 or 2)
};

// Tensor octant layouts of the per-kx plane path (6 comps innermost, so one
// (qz, qy) is three float2 loads):
//   oct4 == 0: [kx][qz][qy mod 2][qy / 2][comp], the even-ky and odd-ky halves
//              of a plane (two-CTA plane kernel) each read contiguous rows;
//   oct4 == 1: [kx][qz][qy mod 4][qy / 4][comp], Py/8 + 1 entries per class, so
//              each CTA of the four-CTA plane kernel (one residue of ky mod 4)
//              reads contiguous rows;
//   oct4 == 2: [qy][qz][comp / 2][kx][comp mod 2], so the deep-grid z kernel (one
//              ky, neighbouring kx on neighbouring lanes) reads contiguous pairs.
__host__ __device__ __forceinline__ int plane_oct4_rows(const Grid& g) { return (g.Py >> 3) + 1; }
__host__ __device__ __forceinline__ long plane_octant_index(const Grid& g, int kx, int comp, int qz, int qy) {
  if (g.oct4 == 1) return ((((long)kx * g.Oz + qz) * 4 + (qy & 3)) * plane_oct4_rows(g) + (qy >> 2)) * 6 + comp;
  if (g.oct4 == 2) return ((((long)qy * g.Oz + qz) * 3 + (comp >> 1)) * g.Hx + kx) * 2 + (comp & 1);
  const int oyh = (g.Oy + 1) >> 1;
  return ((((long)kx * g.Oz + qz) * 2 + (qy & 1)) * oyh + (qy >> 1)) * 6 + comp;
}
// floats to allocate for any of them
__host__ __device__ __forceinline__ long plane_octant_size(const Grid& g) {
  const long two = (long)g.Hx * g.Oz * 2 * ((g.Oy + 1) >> 1) * 6;
  const long four = (long)g.Hx * g.Oz * 4 * plane_oct4_rows(g) * 6;
  return two > four ? two : four;  // (the third is the octant without padding)
}

struct LocalCoef {
  float inv_dx2, inv_dy2, inv_dz2;   // 1/h^2
  float inv_2dx, inv_2dy;            // 1/(2h) for central differences
  float kdx, kdy;                    // h * D/(2A): chiral ghost strength
  float cA;                          // 2A/mu0      (divide by Ms_i)
  float cD;                          // 2D/mu0      (divide by Ms_i)
  float cK;                          // 2Ku/mu0     (scalar Ku; divide by Ms_i)
  float Ms;                          // scalar Ms
  float ax, ay, az;                  // scalar easy axis (unit)
  float hx, hy, hz;                  // bias
  float llg;                         // -gamma0/(1+alpha^2)
  float alpha;
  int dmi, precession;
  const float* ms_map;               // may be null
  const float* ku_map;               // may be null (then cK)
  const float4* axis_map;            // may be null (then ax, ay, az)
};

struct Profiler;
struct AdjWork;

}  // namespace mx

// The context (opaque to callers).
struct mx_ctx {
  mx_params p;
  int device;
  mx::Grid g;

  // material maps (context copies)
  float* ms_map = nullptr;
  float* ku_map = nullptr;
  float4* axis_map = nullptr;

  // demag
  bool built = false;
  float* nhat = nullptr;          // tensor octant: [comp][qz][qy][kx], or plane_octant_index() where octant6()
  float2* w1 = nullptr;           // 3 x nz x ny x Hx   (after the x pass)
  float2* w2 = nullptr;           // 3 x nz x Py x Hx   (after the y pass; unfused path)
  float2* tw_x = nullptr;         // W_Px^k, k < Px
  float2* tw_y = nullptr;         // W_Py^k, k < Py
  float2* tw_z = nullptr;         // W_Pz^k, k < Pz
  bool fused_yz = false;          // y/z passes in one kernel (plane fits on chip)
  bool fast_x = false;            // compile-time-sized x passes available
  bool yz3 = false;               // few-layer y/z kernel (whole kx planes in a block's shared memory) for the fused y/z pass
  bool deep = false;              // deep-grid y and z kernels (demag_deep.cu)
  bool yz2d = false;              // single-z-plane y kernel (Pz == 1) for the fused y/z pass
  float2* tw_m = nullptr;         // W_M^k, k < M = Px/2
  float2* tw_mk = nullptr;        // W_M^(s k) at [k * S + s] for the plane path's x line FFTs (M = E S)
  float2* tw_yh = nullptr;        // W_{Py/2}^k, k < Py/2
  // the octant is stored in plane_octant_index order
  bool octant6() const { return plane || yz3 || deep; }
  bool plane = false;             // per-kx plane kernel (kx-major spectra and tensor)
  bool quad = false;              // plane path uses the four-CTA y/z kernel (else the two-CTA one)
  int xfk_grid = 1;               // persistent grid of the plane path's x forward kernel
  bool xlocal = false;            // inverse x pass fused into the RK/Euler local stage
  bool xrow = false;              // few-row grids: inverse x, local stage and next forward x in one kernel
  bool inject_wait_timeout = false;  // mx_inject_wait_timeout: the two-CTA kernel's bulk-copy wait runs out
  void* dft_a = nullptr;          // split-BF16 DFT matrices (MX_FFT_SPLIT_BF16)
  int yz_tile = 1;                // kx columns per block in the fused kernel
  double* t_real = nullptr;       // FP64 real-space tensor octant (kept for checking)
  double spectrum_imag_ratio = 0; // max|Im| / max|Re| of the FP64 tensor spectrum

  // stage buffers
  float4* hd = nullptr;           // demag field
  float4* sa = nullptr;           // stage input A
  float4* sb = nullptr;           // stage input B
  float4* acc = nullptr;          // RK accumulator
  int* flag = nullptr;            // non-finite flag
  double* ered = nullptr;         // energy accumulators (5)

  // CUDA graph cache for mx_rk_step: a step, and two Euler steps
  cudaGraphExec_t graph = nullptr, pair = nullptr;
  const float* graph_m = nullptr;
  double graph_dt = 0.0;
  int graph_method = -1;
  cudaStream_t cap_stream = nullptr;

  // profiling hook (events around each launch when non-null)
  mx::Profiler* prof = nullptr;

  // adjoint workspaces (mx_adjoint_reserve)
  mx::AdjWork* adj = nullptr;

  // learned demag backend (mx_set_demag_surrogate / mx_set_demag_fno; at
  // most one is set); both NULL: FFT convolution
  struct mx_cnn* surrogate = nullptr;
  struct mx_fno* fno = nullptr;
  float4* mri_f = nullptr;        // MRI slow right-hand sides F_1..F_3 (allocated at first use)
  double* red2 = nullptr;         // 2 FP64 accumulators for mx_rel_l2
};
