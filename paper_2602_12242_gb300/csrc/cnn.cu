// Learned demag surrogate: a 3D conv net 3 -> 32 -> 64 -> 32 -> 3 (3x3x3
// kernels, zero padding 1, exact-erf GELU after the first three layers) that
// maps the normalised magnetisation to the normalised demag field, trained
// with SmoothL1 loss and Adam with L2 weight decay (the paper's ML module,
// Sec. II-D: a network trained offline on (M, H_demag) pairs from the FFT
// solver, per-channel Gaussian normaliser, Adam lr 1e-3, weight decay 1e-4).
//
// Activations are BF16 planes of eight channels, [b z][C/8][y][x][8] with C
// padded to a multiple of 16 (first input: 3 -> 16).  An operand tile, halo
// included, is a box of a tensor map over them: one bulk copy, which fills what
// leaves the grid with zeros (a step of one cell in x is 16 bytes, the alignment
// that a copy's start needs).  So nothing but the cells is stored, 832 bytes for
// each, and each thread of an epilogue stores 16 bytes next to its neighbour's.
// Weights are FP32 masters with BF16 copies in the layout of the tensor cores' operand.
//   forward     out = conv(a, W) + b, stored pre-activation y and a = gelu(y)
//   backward-x  dA_{l-1} = conv(dY_l, W'), W'[tap][ci][co] = W[26 - tap][co][ci],
//               times gelu'(y_{l-1}) in the epilogue -> dY_{l-1}
//   backward-W  dW[tap] = sum over cells of dY (x) x_shifted(tap)
// Every convolution and weight gradient is a tcgen05 (BF16 in, FP32 accumulator
// in tensor memory) kernel of three roles: a producer warp issues the bulk
// copies, one thread the MMAs, eight or sixteen warps (four in the weight
// gradient) run the epilogue of the tile before;
// they meet at mbarriers only (every wait bounded; one that runs out sets
// kFlagTimeout and its role stops).  The last layer's epilogue denormalises, or
// in training forms the loss and its gradient.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <string>
#include <vector>

#include "common.cuh"
#include "kernels.cuh"
#include "bulk.cuh"
#include "mma.cuh"
#include "tc05.cuh"

namespace mx {

static const int kCh[5] = {3, 32, 64, 32, 3};
static const int kCinPad[4] = {16, 32, 64, 32};
static const int kCoutPad[4] = {32, 64, 32, 16};

__device__ __forceinline__ float gelu_f(float y) { return 0.5f * y * (1.f + erff(y * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float y) {
  return 0.5f * (1.f + erff(y * 0.70710678118654752f)) + y * 0.39894228040143268f * expf(-0.5f * y * y);
}

// Grid and samples of an activation.
struct ConvDims {
  int nx, ny, nz, batch;
};
// cells from the start of a plane to cell (x, y)
__device__ __forceinline__ long cell_at(const ConvDims& d, int y, int x) { return (long)y * d.nx + x; }

// A CTA's tiles [t0, t1): tile t is layer z = t % nz of column t / nz.  The
// planes z - 1 .. z + 1 inside the grid are loaded once per column (or at the
// range's start) into a ring of slots, in order.  A tile holds at most three; the
// slots beyond them are what the producer can run ahead, and a copy's latency is
// about that of a tile's MMAs.
struct TileWalk {
  int t0, t1, nz;
  __device__ TileWalk(long ntiles, int cta, int ncta, int nz_) : nz(nz_) {
    t0 = (int)(ntiles * cta / ncta);
    t1 = (int)(ntiles * (cta + 1) / ncta);
  }
  // planes of tile t that are not loaded yet: [z0, z1]
  __device__ void fresh(int t, int& z0, int& z1) const {
    const int z = t % nz;
    z1 = min(nz - 1, z + 1);
    z0 = (t == t0 || z == 0) ? max(0, z - 1) : z + 1;
  }
};

// Bounded barrier wait of a role: false (and kFlagTimeout set) when it runs out.
__device__ __forceinline__ bool role_wait(uint64_t* bar, uint32_t parity, int* flag) {
  if (mbar_wait(bar, parity)) return true;
  atomicOr(flag, kFlagTimeout);
  return false;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32addr(bar)) : "memory");
}

enum ConvMode { CM_HIDDEN = 0, CM_BWD = 1, CM_OUT = 2, CM_LOSS = 3 };

struct ConvArgs {
  const bf16_t* wk;    // [27][CIN/8][NP][8]
  const float* bias;
  bf16_t* out;         // HIDDEN: gelu; BWD: dY of the layer below; LOSS: dY of the last layer (channels 0..7)
  bf16_t* ypre;        // HIDDEN: pre-activation (may be null); BWD: read
  const float4* target;  // LOSS: raw target field
  float4* field;       // OUT: denormalised field
  float* db;           // BWD, LOSS: bias gradient of the layer whose dY is written
  float* loss;         // LOSS
  float3 mean, sd;     // OUT: of the field; LOSS: mean and 1 / std
  float inv_count;     // LOSS
  ConvDims d;
  int* flag;
};

// ---------------------------------------------------------------------------
// Convolution as an implicit GEMM.  A tile is 8 (x) x 16 (y) x 1 output cells, M =
// 128 rows (row = 8 y + x); N = COUT (16 for the last layer); K = 27 taps x CIN.
// Operands in the canonical K-major layout without swizzle:
//   weights [tap][CIN/8][N][8]   B of tap t, K chunk c: 8-row groups (8 output
//                                channels) 128 B apart, K chunks N x 16 B apart
//   plane   [CIN/8][180][8]      (18 x 10 cells): A of tap (dz, dy, dx) starts at
//                                cell (dy, dx) of plane z + dz - 1; each output
//                                row y (8 cells) is one 8-row group, groups are
//                                10 x 16 B apart
// Taps of a plane outside the grid are left out (their products are zero).  A
// CTA walks z fastest, so each tile brings one new plane; the planes of tile t +
// 1 arrive and its MMAs start while the epilogue of tile t runs (two accumulators
// in tensor memory).
// Bound: the MMAs, at about 80 cycles each whatever N <= 64 is (their A operand is 4
// KB of shared memory; 78 over a whole launch of 64 -> 32 channels, 85 of 32 -> 3), and for 64 output channels the issue slots of the epilogue's
// erf.  Measured forward at 64 samples of 64x64x4, with the kernel before in brackets
// (256 threads copied three planes per tile with cp.async, waited for the MMAs and
// ran the epilogue in turn): 3 -> 32 channels 98 us (230), 32 -> 64 167 (362), 64 ->
// 32 191 (475), 32 -> 3 with the loss 104 (268 + 51).  On the way: planes as separate
// bulk copies of their 160-byte rows went out at one per 40 ns (64 -> 32 290 us); a
// single diverged thread issuing the MMAs took 20 cycles more for each than a
// converged warp with uniform operands; column coordinates divided out per tile cost
// 5 %.
// ---------------------------------------------------------------------------
constexpr int kTXc = 8, kTYc = 16;
constexpr int kHXc = kTXc + 2, kHYc = kTYc + 2;
constexpr int kPlaneC = kHXc * kHYc;

template <int CIN, int COUT> struct ConvTc {
  static constexpr int NP = COUT < 16 ? 16 : COUT;  // MMA N
  static constexpr int KC = CIN / 8;
  static constexpr int EW = COUT < 16 ? 8 : 16;     // epilogue warps: four lane quarters x EW / 4 column parts
  static constexpr int threads = 32 * (2 + EW);
  static constexpr uint32_t w_bytes = sizeof(bf16_t) * 8 * 27 * KC * NP;
  static constexpr uint32_t p_bytes = sizeof(bf16_t) * 8 * KC * kPlaneC;
  // as many plane slots as fit, at most 8 (at least 4)
  static constexpr int FIT = (int)((226 * 1024 - w_bytes) / p_bytes);
  static constexpr int RING = FIT < 8 ? FIT : 8;
  static_assert(RING >= 4, "three planes of a tile and one to load");
  static constexpr size_t smem = w_bytes + RING * p_bytes;
  // two accumulators of NP columns, allocated as a power of two >= 32
  static constexpr uint32_t TCOLS = 2 * NP <= 32 ? 32 : (2 * NP <= 64 ? 64 : 128);
};

template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(ConvTc<CIN, COUT>::threads, 1)
    conv_tc_kernel(const __grid_constant__ CUtensorMap in, const __grid_constant__ ConvArgs p) {
  typedef ConvTc<CIN, COUT> T;
  constexpr int RING = T::RING, NP = T::NP, KC = T::KC, NH = NP / (T::EW / 4);
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ __align__(8) uint64_t wbar, full[RING], empty[RING], tfull[2], tempty[2];
  __shared__ uint32_t tbase;
  const ConvDims& d = p.d;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t sw_a = smem_u32(smraw), sp_a = sw_a + T::w_bytes;
  if (tid == 0) {
    mbar_init(&wbar, 1);
    for (int q = 0; q < RING; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&tfull[q], 1);
      mbar_init(&tempty[q], T::EW);
    }
  }
  if (warp == 1) tmem_alloc(&tbase, T::TCOLS);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tb = tbase;
  const int tiles_x = (d.nx + kTXc - 1) / kTXc, tiles_y = (d.ny + kTYc - 1) / kTYc;
  const TileWalk walk((long)tiles_x * tiles_y * d.nz * d.batch, blockIdx.x, gridDim.x, d.nz);
  // column col: first cell of its tile, sample
  auto column = [&](int col, int& b, int& y0, int& x0) {
    x0 = col % tiles_x * kTXc;
    const int r = col / tiles_x;
    y0 = r % tiles_y * kTYc;
    b = r / tiles_y;
  };
  if (warp == 0) {
    // ---- producer: the weights (constants of this launch, last written before
    // the kernel before this one), then the planes
    if (lane == 0) mbar_arrive_expect_tx(&wbar, T::w_bytes);
    __syncwarp();
    if (lane < 27)
      bulk_load(smraw + lane * (T::w_bytes / 27), p.wk + (long)lane * (T::w_bytes / 27 / sizeof(bf16_t)),
                T::w_bytes / 27, &wbar);
    pdl_wait_next();
    if (lane == 0) {
      int seq = 0;
      bool ok = true;
      for (int t = walk.t0; t < walk.t1 && ok; ++t) {
        int b, y0, x0, z0, z1;
        column(t / d.nz, b, y0, x0);
        walk.fresh(t, z0, z1);
        for (int z = z0; z <= z1; ++z, ++seq) {
          const int slot = seq % RING;
          if (seq >= RING) ok = role_wait(&empty[slot], (uint32_t)(seq / RING - 1) & 1u, p.flag);
          if (!ok) break;
          mbar_arrive_expect_tx(&full[slot], T::p_bytes);
          // (zeros where the halo leaves the grid)
          tensor_load3(smraw + T::w_bytes + slot * T::p_bytes, &in, (x0 - 1) * 8, y0 - 1, (b * d.nz + z) * KC,
                       &full[slot]);
        }
      }
      // no copy is in flight when the block ends (each full barrier's last phase)
      for (int q = max(0, seq - RING); q < seq; ++q) mbar_wait(&full[q % RING], (uint32_t)(q / RING) & 1u);
      mbar_wait(&wbar, 0);
    }
    __syncwarp();
  } else if (warp == 1) {
    {
      // ---- MMA issue: the warp stays together (its operands are uniform), one thread issues
      pdl_wait();  // (the bounds of its waits do not count the kernel before)
      const uint32_t leader = tc_elect();
      constexpr uint32_t idesc = tc_idesc_bf16(128, NP);
      bool ok = __all_sync(0xffffffffu, role_wait(&wbar, 0, p.flag));
      int seq = 0, zfirst = 0, sfirst = 0;  // ring position of the column's plane zfirst is sfirst
      for (int t = walk.t0; t < walk.t1 && ok; ++t) {
        const int k = t - walk.t0, z = t % d.nz;
        int z0, z1;
        walk.fresh(t, z0, z1);
        if (t == walk.t0 || z == 0) {
          zfirst = z0;
          sfirst = seq;
        }
        for (int q = z0; q <= z1 && ok; ++q, ++seq)
          ok = __all_sync(0xffffffffu, role_wait(&full[seq % RING], (uint32_t)(seq / RING) & 1u, p.flag));
        if (k >= 2 && ok)
          ok = __all_sync(0xffffffffu, role_wait(&tempty[k & 1], (uint32_t)(k / 2 - 1) & 1u, p.flag));
        if (!ok) break;
        tc_fence_after_sync();
        const uint32_t dt = tb + (uint32_t)((k & 1) * NP);
        bool acc = false;
#pragma unroll 1
        for (int dz = 0; dz < 3; ++dz) {
          const int zp = z + dz - 1;
          if (zp < 0 || zp >= d.nz) continue;
          const uint64_t ad = tc_sdesc(sp_a + (uint32_t)((sfirst + zp - zfirst) % RING) * T::p_bytes, kPlaneC * 16,
                                       kHXc * 16);
          const uint64_t bd = tc_sdesc(sw_a + (uint32_t)(dz * 9 * KC * NP * 16), NP * 16, 128);
          const uint32_t alo = (uint32_t)ad, ahi = (uint32_t)(ad >> 32), blo = (uint32_t)bd, bhi = (uint32_t)(bd >> 32);
#pragma unroll
          for (int tap = 0; tap < 9; ++tap)
#pragma unroll
            for (int ks = 0; ks < CIN / 16; ++ks) {
              tc_mma_bf16_lo(dt, alo + (uint32_t)(2 * ks * kPlaneC + tap / 3 * kHXc + tap % 3), ahi,
                             blo + (uint32_t)((tap * KC + 2 * ks) * NP), bhi, idesc, acc, leader);
              acc = true;
            }
        }
        // planes used for the last time by this tile
        if (leader) {
          if (z > 0) tc_commit(&empty[(sfirst + z - 1 - zfirst) % RING]);
          if (z == d.nz - 1) tc_commit(&empty[(sfirst + z - zfirst) % RING]);
          tc_commit(&tfull[k & 1]);
        }
        __syncwarp();
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue: warp reads lanes 32 (warp mod 4) .. + 31, columns of part (warp - 2) / 4
    const int row = 32 * (warp & 3) + lane;
    const int cx = row & 7, cy = row >> 3;
    const int cb = (warp - 2) / 4 * NH;
    pdl_wait_next();
    float bv[NH];
#pragma unroll
    for (int c = 0; c < NH; ++c) bv[c] = (MODE == CM_BWD || cb + c >= COUT || (COUT == 8 && cb + c >= 3)) ? 0.f : __ldg(&p.bias[cb + c]);
    float db[NH] = {};
    double lsum = 0.0;
    const long plane = (long)d.ny * d.nx * 8;
    // (the walk's divisions once per column: they would be a third of the epilogue's instructions)
    int z = walk.t0 % d.nz, b, y0, x0;
    column(walk.t0 / d.nz, b, y0, x0);
    for (int t = walk.t0; t < walk.t1; ++t, ++z) {
      const int k = t - walk.t0;
      if (z == d.nz) {
        z = 0;
        column(t / d.nz, b, y0, x0);
      }
      // (the vote also brings the warp together for the tensor-memory loads)
      if (!__all_sync(0xffffffffu, role_wait(&tfull[k & 1], (uint32_t)(k / 2) & 1u, p.flag))) break;
      tc_fence_after_sync();
      float v[NH];
#pragma unroll
      for (int q = 0; q < NH / 8; ++q) {
        float t8[8];
        tmem_ld8(tb + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((k & 1) * NP + cb + 8 * q), t8);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[8 * q + i] = t8[i];
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[k & 1]);  // the accumulator may be overwritten
      const int gx = x0 + cx, gy = y0 + cy;
      if (gx >= d.nx || gy >= d.ny) continue;
      const long bz = (long)b * d.nz + z;
      if (MODE == CM_HIDDEN || MODE == CM_BWD) {
        // eight channels per 16-byte store
        const long at0 = (bz * (COUT / 8) + cb / 8) * plane + cell_at(d, gy, gx) * 8;
#pragma unroll
        for (int c = 0; c < NH; c += 8) {
          const long at = at0 + c / 8 * plane;
          uint32_t o[4];
          if (MODE == CM_HIDDEN) {
            uint32_t yp[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float v0 = v[c + 2 * j] + bv[c + 2 * j], v1 = v[c + 2 * j + 1] + bv[c + 2 * j + 1];
              yp[j] = pack2(v0, v1);
              o[j] = pack2(gelu_f(v0), gelu_f(v1));
            }
            if (p.ypre) *(uint4*)(p.ypre + at) = make_uint4(yp[0], yp[1], yp[2], yp[3]);
          } else {
            const uint4 y4 = *(const uint4*)(p.ypre + at);
            const uint32_t yw[4] = {y4.x, y4.y, y4.z, y4.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float y0f = bf2f((bf16_t)(yw[j] & 0xffff)), y1f = bf2f((bf16_t)(yw[j] >> 16));
              o[j] = pack2(v[c + 2 * j] * gelu_grad(y0f), v[c + 2 * j + 1] * gelu_grad(y1f));
              db[c + 2 * j] += bf2f((bf16_t)(o[j] & 0xffff));
              db[c + 2 * j + 1] += bf2f((bf16_t)(o[j] >> 16));
            }
          }
          *(uint4*)(p.out + at) = make_uint4(o[0], o[1], o[2], o[3]);
        }
      } else if (cb == 0) {
        const long cell = bz * ((long)d.nx * d.ny) + (long)gy * d.nx + gx;
        const float q[3] = {v[0] + bv[0], v[1] + bv[1], v[2] + bv[2]};
        if (MODE == CM_OUT) {
          p.field[cell] = make_float4(q[0] * p.sd.x + p.mean.x, q[1] * p.sd.y + p.mean.y, q[2] * p.sd.z + p.mean.z, 0.f);
        } else {
          // SmoothL1 (beta 1) against the normalised target
          const float4 tg = p.target[cell];
          const float e[3] = {q[0] - (tg.x - p.mean.x) * p.sd.x, q[1] - (tg.y - p.mean.y) * p.sd.y,
                              q[2] - (tg.z - p.mean.z) * p.sd.z};
          float g[3], l = 0.f;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float a = fabsf(e[c]);
            l += a < 1.f ? 0.5f * e[c] * e[c] : a - 0.5f;
            g[c] = fminf(fmaxf(e[c], -1.f), 1.f) * p.inv_count;
          }
          lsum += (double)l;
          const uint32_t o0 = pack2(g[0], g[1]), o1 = pack2(g[2], 0.f);
          db[0] += bf2f((bf16_t)(o0 & 0xffff));
          db[1] += bf2f((bf16_t)(o0 >> 16));
          db[2] += bf2f((bf16_t)(o1 & 0xffff));
          // (channels 8..15 of the padded sixteen stay at zero)
          *(uint4*)(p.out + bz * 2 * plane + cell_at(d, gy, gx) * 8) = make_uint4(o0, o1, 0u, 0u);
        }
      }
    }
    if (MODE == CM_BWD || MODE == CM_LOSS) {
      constexpr int ND = MODE == CM_LOSS ? 3 : NH;
#pragma unroll
      for (int c = 0; c < ND; ++c) {
        float v = db[c];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0 && (MODE == CM_BWD || cb == 0)) atomicAdd(&p.db[cb + c], v);
      }
      if (MODE == CM_LOSS) {
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, o);
        if (lane == 0 && cb == 0) atomicAdd(p.loss, (float)(lsum * (double)p.inv_count));
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tb, T::TCOLS);
  }
}

// ---------------------------------------------------------------------------
// Weight gradient of one layer: the correlation
//   G[dz, dy][(s, cs)][cr] = sum_cells S[cell + (0, 0, s - 1)][cs] R[cell + (dz - 1, dy - 1, 0)][cr]
// of a "stacked" operand S (CS channels) and a "ring" operand R (CR channels).  With
// S = dY and R = x, G = dW[dz][dy][2 - s]; with S = x and R = dY (the layer whose
// output is wider), G = dW[2 - dz][2 - dy][s].  The three x-shifts of S are three
// copies of its tile in shared memory, so that they fill the M = 128 rows of one
// MMA (3 CS of them; the rest is whatever follows in shared memory, and its
// result is never read), and one MMA serves three taps: a tap per MMA reads the
// same 4 KB of A for a third of the use.  N = CR, K = 16 cells of a row; one
// accumulator of CR columns per dy in tensor memory: a CTA owns one dz and a range of
// 16 x 8 tiles (a chain), in the order x, y, z, sample; two CTAs share an SM.
// Tensor-core accumulation cuts each sum off below the accumulator's last place, so
// its error grows with the number of MMAs a sum goes through: a chain is as many
// tiles as six chains per SM and (dz, dy) make (81 at 64 samples of 64x64x4).
// The middle dz, whose planes of R are all inside the grid, goes first: its blocks
// are the longest.
// Both operands are MN-major (channels contiguous, one 16-byte row of 8 channels
// per cell, core matrices adjacent along K 128 B apart, 8-channel groups SBO
// apart): boxes of the planes.  Planes of R outside the grid are left out.
// The chains are added in FP32 in ws[(dz 3 + dy) CR + cr][(s, cs)], lanes next to
// each other.  Bound: the MMAs' operand reads (6 KB per MMA at N = 64) and L2.
// Measured at 64 samples of 64x64x4, with the kernel before in brackets (a (dz, dy)
// per block, a tap per MMA, copies and MMAs in turn): 64 -> 32 and 32 -> 64 110 us
// each (863, 600), 3 -> 32 and 32 -> 3 88 each (315, 452).  A CTA per SM with five or
// four of the nine (dz, dy), planes of R kept in a ring: 131 and 101.
// ---------------------------------------------------------------------------
constexpr int kTX = 16, kTY = 8;  // tile (cells)
template <int CS, int CR> struct WgradTc {
  static constexpr uint32_t S_SBO = kTX * kTY * 16, R_SBO = kTX * (kTY + 2) * 16;  // slabs of 8 channels
  static constexpr uint32_t s_bytes = 3 * (CS / 8) * S_SBO, r_bytes = (CR / 8) * R_SBO, stage = s_bytes + r_bytes;
  static constexpr int ST = (int)(113 * 1024 / stage) < 4 ? (int)(113 * 1024 / stage) : 4;  // stages
  static_assert(ST >= 2, "wgrad stages");
  // the 16 row groups of an MMA starting in the last stage stay inside
  static constexpr uint32_t reach = (ST - 1) * stage + 16 * S_SBO + kTX * kTY * 16;
  static constexpr size_t smem = ST * stage > reach ? ST * stage : reach;
  static constexpr uint32_t TCOLS = 3 * CR <= 128 ? 128 : 256;
  static_assert(3 * CS <= 128 && 3 * CR <= 256 && CR % 16 == 0, "wgrad shape");
};

template <int CS, int CR>
__global__ void __launch_bounds__(192, 2)
    wgrad_tc_kernel(const __grid_constant__ CUtensorMap S, const __grid_constant__ CUtensorMap R,
                    float* __restrict__ ws, ConvDims d, int chain, int* flag) {
  typedef WgradTc<CS, CR> W;
  constexpr int ST = W::ST;
  extern __shared__ __align__(128) unsigned char smraw[];
  __shared__ __align__(8) uint64_t full[ST], empty[ST], done;
  __shared__ uint32_t tbase, started_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chains = (int)gridDim.x / 3, third = (int)blockIdx.x / chains;
  const int dz = third == 0 ? 1 : third == 1 ? 0 : 2;
  if (tid == 0) {
    for (int q = 0; q < ST; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], 1);
    }
    mbar_init(&done, 2);  // the MMAs' completion, and the thread that issued them
  }
  if (warp == 1) tmem_alloc(&tbase, W::TCOLS);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tb = tbase;
  const int tiles_x = (d.nx + kTX - 1) / kTX, tiles_y = (d.ny + kTY - 1) / kTY;
  const long ntiles = (long)tiles_x * tiles_y * d.nz * d.batch;
  const long t0 = (long)((int)blockIdx.x % chains) * chain, t1 = t0 + chain < ntiles ? t0 + chain : ntiles;
  // tile t: its plane's index b nz + z; whether R's plane is inside the grid
  auto inside = [&](long t, int& bz) {
    bz = (int)(t / (tiles_x * tiles_y));
    const int zp = bz % d.nz + dz - 1;
    return zp >= 0 && zp < d.nz;
  };
  pdl_wait_next();
  if (warp == 0) {
    if (lane == 0) {
      int k = 0;
      bool ok = true;
      for (long t = t0; t < t1; ++t) {
        int bz;
        if (!inside(t, bz)) continue;
        if (k >= ST) ok = role_wait(&empty[k % ST], (uint32_t)(k / ST - 1) & 1u, flag);
        if (!ok) break;
        const int x0 = (int)(t % tiles_x) * kTX, y0 = (int)(t / tiles_x % tiles_y) * kTY;
        uint64_t* bar = &full[k % ST];
        unsigned char* st = smraw + (k % ST) * W::stage;
        mbar_arrive_expect_tx(bar, W::stage);
        // S: three copies shifted by -1, 0, +1 in x (zeros outside the grid)
        for (int sh = 0; sh < 3; ++sh)
          tensor_load3(st + sh * (W::s_bytes / 3), &S, (x0 + sh - 1) * 8, y0, bz * (CS / 8), bar);
        tensor_load3(st + W::s_bytes, &R, x0 * 8, y0 - 1, (bz + dz - 1) * (CR / 8), bar);
        ++k;
      }
      // no copy is in flight when the block ends
      for (int q = max(0, k - ST); q < k; ++q) mbar_wait(&full[q % ST], (uint32_t)(q / ST) & 1u);
    }
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t leader = tc_elect();
    constexpr uint32_t idesc = tc_idesc_bf16(128, CR) | (1u << 15) | (1u << 16);  // A and B MN-major
    const uint32_t s_a = smem_u32(smraw);
    int k = 0;
    bool ok = true;
    for (long t = t0; t < t1; ++t) {
      int bz;
      if (!inside(t, bz)) continue;
      ok = __all_sync(0xffffffffu, role_wait(&full[k % ST], (uint32_t)(k / ST) & 1u, flag));
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t sa = s_a + (uint32_t)(k % ST) * W::stage;
      const uint64_t ad = tc_sdesc(sa, 128, W::S_SBO), bd = tc_sdesc(sa + W::s_bytes, 128, W::R_SBO);
#pragma unroll
      for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int cy = 0; cy < kTY; ++cy)
          tc_mma_bf16_lo(tb + dy * CR, (uint32_t)ad + cy * kTX, (uint32_t)(ad >> 32), (uint32_t)bd + (cy + dy) * kTX,
                         (uint32_t)(bd >> 32), idesc, cy > 0 || k > 0, leader);
      if (leader) tc_commit(&empty[k % ST]);
      __syncwarp();
      ++k;
    }
    if (leader) {
      started_s = ok && k > 0 ? 1u : 0u;
      // (the completion of MMAs does not order this thread's stores; its own arrival does)
      mbar_arrive(&done);
      tc_commit(&done);
    }
    __syncwarp();
    role_wait(&done, 0, flag);  // no MMA is in flight when the block ends
  } else {
    // ---- the chain's sums: lane = row (s, cs) of quarter warp mod 4
    const int row = 32 * (warp & 3) + lane;
    const bool ok = __all_sync(0xffffffffu, role_wait(&done, 0, flag));
    tc_fence_after_sync();
    if (ok && started_s && 32 * (warp & 3) < 3 * CS) {
#pragma unroll 1
      for (int c = 0; c < 3 * CR; c += 8) {
        float v[8];
        tmem_ld8(tb + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c, v);
        if (row < 3 * CS) {
#pragma unroll
          for (int i = 0; i < 8; ++i) atomicAdd(&ws[(long)(dz * 3 * CR + c + i) * (3 * CS) + row], v[i]);
        }
        __syncwarp();
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tb, W::TCOLS);
  }
}

// ws of all four layers -> the gradient's weights (parameter order [co][ci][27])
struct WgradOut {
  long ws, dw;       // offsets
  int cs, cr, cin, cout, sx;  // sx: S is x (else dY)
};
struct WgradOuts {
  WgradOut l[4];
};
__global__ void wgrad_finish_kernel(const float* ws, float* __restrict__ grad, WgradOuts o) {
  const WgradOut l = o.l[blockIdx.y];
  pdl_wait_next();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= l.cout * l.cin * 27) return;
  const int tap = e % 27, ci = e / 27 % l.cin, co = e / 27 / l.cin;
  const int dz = tap / 9, dy = tap / 3 % 3, dx = tap % 3;
  const int j = l.sx ? (2 - dz) * 3 + 2 - dy : dz * 3 + dy, s = l.sx ? dx : 2 - dx;
  const int cs = l.sx ? ci : co, cr = l.sx ? co : ci;
  grad[l.dw + e] = ws[l.ws + (long)(j * l.cr + cr) * (3 * l.cs) + s * l.cs + cs];
}

// input normalisation: m float4 -> the first eight channels of the padded input
__global__ void normalize_in_kernel(const float4* m, bf16_t* __restrict__ x0, ConvDims d, long ncells,
                                    float3 mean, float3 inv_std) {
  const long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait_next();
  if (c >= ncells) return;
  const float4 v = m[c];
  const int x = (int)(c % d.nx), y = (int)(c / d.nx % d.ny);
  const long bz = c / ((long)d.nx * d.ny);
  uint4 o;
  o.x = pack2((v.x - mean.x) * inv_std.x, (v.y - mean.y) * inv_std.y);
  o.y = pack2((v.z - mean.z) * inv_std.z, 0.f);
  o.z = o.w = 0u;
  *(uint4*)(x0 + (bz * 2 * d.ny * d.nx + cell_at(d, y, x)) * 8) = o;
}

// FP32 master weights -> bf16 [27][CIN_PAD/8][COUT_PAD][8] (forward) and the
// flipped, transposed copy [27][CIN_PAD'/8][COUT_PAD'][8] for the backward pass.
__global__ void pack_weights_kernel(const float* __restrict__ W, int cin, int cout, bf16_t* __restrict__ fwd,
                                    int cin_pad, int cout_pad, bf16_t* __restrict__ bwd, int bwd_in_pad,
                                    int bwd_out_pad) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int nf = 27 * cout_pad * cin_pad;
  if (e < nf) {
    const int co = e / 8 % cout_pad, ci = e / 8 / cout_pad % (cin_pad / 8) * 8 + e % 8, tap = e / (cin_pad * cout_pad);
    const float v = (ci < cin && co < cout) ? W[((long)co * cin + ci) * 27 + tap] : 0.f;
    fwd[e] = f2bf(v);
  }
  if (bwd) {
    const int nb = 27 * bwd_out_pad * bwd_in_pad;
    if (e < nb) {
      // backward conv: input channels = this layer's cout, output channels = cin
      const int ci = e / 8 % bwd_out_pad, co = e / 8 / bwd_out_pad % (bwd_in_pad / 8) * 8 + e % 8;
      const int tap = 26 - e / (bwd_in_pad * bwd_out_pad);
      const float v = (ci < cin && co < cout) ? W[((long)co * cin + ci) * 27 + tap] : 0.f;
      bwd[e] = f2bf(v);
    }
  }
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, long n, float lr, float wd, float b1, float b2, float c1, float c2,
                            float eps) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i] + wd * p[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

mx_status adam_update(float* p, const float* g, float* m, float* v, long n, double lr, double wd, int t,
                      cudaStream_t st) {
  const double b1 = 0.9, b2 = 0.999;
  const double c1 = 1.0 - pow(b1, t), c2 = 1.0 - pow(b2, t);
  adam_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p, g, m, v, n, (float)lr, (float)wd, (float)b1,
                                                           (float)b2, (float)c1, (float)c2, 1e-8f);
  return launch_check("adam_kernel");
}

}  // namespace mx

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
using mx::bf16_t;

struct mx_cnn {
  int nx, ny, nz, max_batch;
  long cells;
  float* params = nullptr;  // FP32 masters, oracle order (W1, b1, ..., W4, b4)
  float* grad = nullptr;
  float* am = nullptr;
  float* av = nullptr;
  int adam_t = 0;
  bf16_t* wf[4] = {nullptr, nullptr, nullptr, nullptr};
  bf16_t* wb[4] = {nullptr, nullptr, nullptr, nullptr};
  bf16_t *x0 = nullptr, *a1 = nullptr, *y1 = nullptr, *a2 = nullptr, *y2 = nullptr, *a3 = nullptr, *y3 = nullptr;
  bf16_t *dy4 = nullptr, *dy3 = nullptr, *dy2 = nullptr, *dy1 = nullptr;
  // the activations as tensors [b z C/8][ny][nx 8] with the boxes of the
  // convolutions' input planes and of the weight gradients' S and R tiles
  CUtensorMap c_x0, c_a1, c_a2, c_a3, c_dy4, c_dy3, c_dy2;
  CUtensorMap s_x0, s_a1, s_dy3, s_dy4, r_dy1, r_dy2, r_a2, r_a3;
  float* ws = nullptr;      // weight-gradient sums of the four layers, in their kernels' order
  float* loss = nullptr;
  int* flag = nullptr;  // device status bits (kFlagTimeout), read by mx_cnn_sync / mx_sync
  float stats[12] = {0, 0, 0, 1, 1, 1, 0, 0, 0, 1, 1, 1};
};

namespace mx {

static long layer_w_off(int l) {
  long o = 0;
  for (int q = 0; q < l; ++q) o += (long)kCh[q] * kCh[q + 1] * 27 + kCh[q + 1];
  return o;
}
static long num_params_total() { return layer_w_off(4); }

static ConvDims conv_dims(const mx_cnn* n, int batch) {
  ConvDims d;
  d.nx = n->nx;
  d.ny = n->ny;
  d.nz = n->nz;
  d.batch = batch;
  return d;
}
// elements of an activation of C channels
static size_t act_elems(const mx_cnn* n, int C, int batch) { return (size_t)batch * n->cells * C; }

// Tensor map of an activation of C channels, box bx cells x by rows x all C / 8 planes of a layer.
static mx_status make_map(const mx_cnn* n, CUtensorMap* map, bf16_t* base, int C, int bx, int by) {
  typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode encode = []() -> Encode {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      fn = nullptr;
    }
    return (Encode)fn;
  }();
  if (!encode) {
    set_error("mx_cnn_create: the driver has no cuTensorMapEncodeTiled");
    return MX_ERR_CUDA;
  }
  const cuuint64_t dims[3] = {(cuuint64_t)n->nx * 8, (cuuint64_t)n->ny, (cuuint64_t)n->max_batch * n->nz * (C / 8)};
  const cuuint64_t strides[2] = {(cuuint64_t)n->nx * 16, (cuuint64_t)n->nx * 16 * n->ny};
  const cuuint32_t box[3] = {(cuuint32_t)bx * 8, (cuuint32_t)by, (cuuint32_t)(C / 8)}, one[3] = {1, 1, 1};
  if (encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
    set_error("mx_cnn_create: tensor map not encoded");
    return MX_ERR_CUDA;
  }
  return MX_OK;
}
static mx_status make_maps(mx_cnn* n) {
  auto c = [&](CUtensorMap* m, bf16_t* b, int C) { return make_map(n, m, b, C, kHXc, kHYc); };
  auto s = [&](CUtensorMap* m, bf16_t* b, int C) { return make_map(n, m, b, C, kTX, kTY); };
  auto r = [&](CUtensorMap* m, bf16_t* b, int C) { return make_map(n, m, b, C, kTX, kTY + 2); };
  MX_TRY(c(&n->c_x0, n->x0, 16));
  MX_TRY(c(&n->c_a1, n->a1, 32));
  MX_TRY(c(&n->c_a2, n->a2, 64));
  MX_TRY(c(&n->c_a3, n->a3, 32));
  MX_TRY(c(&n->c_dy4, n->dy4, 16));
  MX_TRY(c(&n->c_dy3, n->dy3, 32));
  MX_TRY(c(&n->c_dy2, n->dy2, 64));
  MX_TRY(s(&n->s_x0, n->x0, 16));
  MX_TRY(s(&n->s_a1, n->a1, 32));
  MX_TRY(s(&n->s_dy3, n->dy3, 32));
  MX_TRY(s(&n->s_dy4, n->dy4, 16));
  MX_TRY(r(&n->r_dy1, n->dy1, 32));
  MX_TRY(r(&n->r_dy2, n->dy2, 64));
  MX_TRY(r(&n->r_a2, n->a2, 64));
  return r(&n->r_a3, n->a3, 32);
}

static int num_sms() {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0)
    v = 1;
  return v;
}

template <int CIN, int COUT, int MODE>
static mx_status conv_run(const CUtensorMap& in, const ConvArgs& p, cudaStream_t st, bool setup = false) {
  typedef ConvTc<CIN, COUT> T;
  auto k = conv_tc_kernel<CIN, COUT, MODE>;
  if (setup) {
    MX_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::smem));
    return MX_OK;
  }
  const ConvDims& d = p.d;
  const long ntiles = (long)((d.nx + kTXc - 1) / kTXc) * ((d.ny + kTYc - 1) / kTYc) * d.nz * d.batch;
  const int sms = num_sms();
  launch_pdl(k, dim3((unsigned)(ntiles < sms ? ntiles : sms)), dim3(T::threads), T::smem, st, in, p);
  return launch_check("conv_tc_kernel");
}

template <int CS, int CR>
static mx_status wgrad_run(const CUtensorMap& S, const CUtensorMap& R, float* ws, const ConvDims& d, int* flag, cudaStream_t st,
                           bool setup = false) {
  typedef WgradTc<CS, CR> W;
  auto k = wgrad_tc_kernel<CS, CR>;
  if (setup) {
    MX_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W::smem));
    return MX_OK;
  }
  const long ntiles = (long)((d.nx + kTX - 1) / kTX) * ((d.ny + kTY - 1) / kTY) * d.nz * d.batch;
  const long six = 6L * num_sms();
  const int chain = (int)((ntiles * 9 + six - 1) / six);
  const long chains = (ntiles + chain - 1) / chain;
  launch_pdl(k, dim3((unsigned)(3 * chains)), dim3(192), W::smem, st, S, R, ws, d, chain, flag);
  return launch_check("wgrad_tc_kernel");
}

// Where each layer's sums lie in ws and go in the gradient.
static WgradOuts wgrad_outs(long* total) {
  // layers 1 and 2 stack x (16, 32 channels), layers 3 and 4 stack dY (32, 16)
  static const int cs[4] = {16, 32, 32, 16}, cr[4] = {32, 64, 64, 32}, sx[4] = {1, 1, 0, 0};
  WgradOuts o;
  long at = 0;
  for (int l = 0; l < 4; ++l) {
    o.l[l] = WgradOut{at, layer_w_off(l), cs[l], cr[l], kCh[l], kCh[l + 1], sx[l]};
    at += 27L * cs[l] * cr[l];
  }
  *total = at;
  return o;
}

static mx_status cnn_setup() {
  const ConvArgs none{};
  const ConvDims nd{};
  const CUtensorMap nm{};
  MX_TRY((conv_run<16, 32, CM_HIDDEN>(nm, none, nullptr, true)));
  MX_TRY((conv_run<32, 64, CM_HIDDEN>(nm, none, nullptr, true)));
  MX_TRY((conv_run<64, 32, CM_HIDDEN>(nm, none, nullptr, true)));
  MX_TRY((conv_run<32, 8, CM_OUT>(nm, none, nullptr, true)));
  MX_TRY((conv_run<32, 8, CM_LOSS>(nm, none, nullptr, true)));
  MX_TRY((conv_run<16, 32, CM_BWD>(nm, none, nullptr, true)));
  MX_TRY((conv_run<32, 64, CM_BWD>(nm, none, nullptr, true)));
  MX_TRY((conv_run<64, 32, CM_BWD>(nm, none, nullptr, true)));
  MX_TRY((wgrad_run<16, 32>(nm, nm, nullptr, nd, nullptr, nullptr, true)));
  return wgrad_run<32, 64>(nm, nm, nullptr, nd, nullptr, nullptr, true);
}

static mx_status pack_all(mx_cnn* n, cudaStream_t st) {
  // forward packs [27][coutpad][cinpad]; backward packs for layers 2..4
  const int bw_in[4] = {0, 64, 32, 16};   // backward conv input channels (this layer's cout, padded)
  const int bw_out[4] = {0, 32, 64, 32};  // backward conv output channels (this layer's cin)
  for (int l = 0; l < 4; ++l) {
    const int cin = kCh[l], cout = kCh[l + 1];
    const int nf = 27 * kCoutPad[l] * kCinPad[l];
    const int nb = l > 0 ? 27 * bw_in[l] * bw_out[l] : 0;
    const int ne = nf > nb ? nf : nb;
    pack_weights_kernel<<<(ne + 255) / 256, 256, 0, st>>>(n->params + layer_w_off(l), cin, cout, n->wf[l], kCinPad[l],
                                                          kCoutPad[l], l > 0 ? n->wb[l] : nullptr, bw_in[l], bw_out[l]);
    MX_TRY(launch_check("pack_weights_kernel"));
  }
  return MX_OK;
}

// The three hidden layers: m -> a3 (and, for training, the pre-activations).
static mx_status cnn_hidden(mx_cnn* n, const float4* m, int batch, bool train, cudaStream_t st) {
  const long nc = n->cells * batch;
  const float* s = n->stats;
  const ConvDims d = conv_dims(n, batch);
  launch_pdl(normalize_in_kernel, dim3((unsigned)((nc + 255) / 256)), dim3(256), 0, st, m, n->x0, d, nc,
             make_float3(s[0], s[1], s[2]), make_float3(1.f / s[3], 1.f / s[4], 1.f / s[5]));
  MX_TRY(launch_check("normalize_in_kernel"));
  const float* P = n->params;
  ConvArgs a{};
  a.d = d;
  a.flag = n->flag;
  a.wk = n->wf[0], a.bias = P + layer_w_off(0) + 32 * 3 * 27, a.out = n->a1;
  a.ypre = train ? n->y1 : nullptr;
  MX_TRY((conv_run<16, 32, CM_HIDDEN>(n->c_x0, a, st)));
  a.wk = n->wf[1], a.bias = P + layer_w_off(1) + 64 * 32 * 27, a.out = n->a2;
  a.ypre = train ? n->y2 : nullptr;
  MX_TRY((conv_run<32, 64, CM_HIDDEN>(n->c_a1, a, st)));
  a.wk = n->wf[2], a.bias = P + layer_w_off(2) + 32 * 64 * 27, a.out = n->a3;
  a.ypre = train ? n->y3 : nullptr;
  return conv_run<64, 32, CM_HIDDEN>(n->c_a2, a, st);
}

static mx_status cnn_forward(mx_cnn* n, const float4* m, float4* h, int batch, cudaStream_t st) {
  MX_TRY(cnn_hidden(n, m, batch, false, st));
  const float* s = n->stats;
  ConvArgs a{};
  a.d = conv_dims(n, batch);
  a.flag = n->flag;
  a.wk = n->wf[3], a.bias = n->params + layer_w_off(3) + 3 * 32 * 27, a.field = h;
  a.mean = make_float3(s[6], s[7], s[8]), a.sd = make_float3(s[9], s[10], s[11]);
  return conv_run<32, 8, CM_OUT>(n->c_a3, a, st);
}

bool cnn_matches(const mx_cnn* n, const Grid& g) { return n->nx == g.nx && n->ny == g.ny && n->nz == g.nz; }

mx_status cnn_demag(mx_cnn* n, const float4* m, float4* h, cudaStream_t st) { return cnn_forward(n, m, h, 1, st); }

// Reads and clears the net's device status flag (synchronises `stream`).
mx_status cnn_take_flag(mx_cnn* n, cudaStream_t st, int* flag_out) {
  int f = 0;
  MX_CUDA_TRY(cudaMemcpyAsync(&f, n->flag, sizeof(int), cudaMemcpyDeviceToHost, st));
  MX_CUDA_TRY(cudaStreamSynchronize(st));
  if (f) {
    MX_CUDA_TRY(cudaMemsetAsync(n->flag, 0, sizeof(int), st));
    MX_CUDA_TRY(cudaStreamSynchronize(st));
  }
  *flag_out = f;
  return MX_OK;
}

}  // namespace mx

using namespace mx;

extern "C" {

int mx_cnn_num_params(void) { return (int)num_params_total(); }

mx_status mx_cnn_destroy(mx_cnn* n) {
  if (!n) return MX_OK;
  void* ptrs[] = {n->params, n->grad, n->am, n->av, n->wf[0], n->wf[1], n->wf[2], n->wf[3], n->wb[1], n->wb[2],
                  n->wb[3], n->x0, n->a1, n->y1, n->a2, n->y2, n->a3, n->y3, n->dy4, n->dy3, n->dy2, n->dy1,
                  n->ws, n->loss, n->flag};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete n;
  return MX_OK;
}

mx_status mx_cnn_create(mx_cnn** out, int nx, int ny, int nz, int max_batch) {
  clear_error();
  if (!out || nx < 1 || ny < 1 || nz < 1 || max_batch < 1) {
    set_error("mx_cnn_create: need out != NULL and nx, ny, nz, max_batch >= 1");
    return MX_ERR_INVALID_ARG;
  }
  *out = nullptr;
  mx_cnn* n = new mx_cnn();
  n->nx = nx;
  n->ny = ny;
  n->nz = nz;
  n->max_batch = max_batch;
  n->cells = (long)nx * ny * nz;
  const long np = num_params_total();
  long nws = 0;
  wgrad_outs(&nws);
  bool ok = true;
  auto alloc = [&](void** p, size_t bytes, bool zero) {
    if (ok && cudaMalloc(p, bytes) != cudaSuccess) {
      cudaGetLastError();
      ok = false;
    }
    if (ok && zero && cudaMemset(*p, 0, bytes) != cudaSuccess) ok = false;
  };
  alloc((void**)&n->params, sizeof(float) * np, true);
  alloc((void**)&n->grad, sizeof(float) * np, false);
  alloc((void**)&n->am, sizeof(float) * np, true);
  alloc((void**)&n->av, sizeof(float) * np, true);
  const int bw_in[4] = {0, 64, 32, 16}, bw_out[4] = {0, 32, 64, 32};
  for (int l = 0; l < 4; ++l) {
    alloc((void**)&n->wf[l], sizeof(bf16_t) * 27 * kCoutPad[l] * kCinPad[l], true);
    if (l > 0) alloc((void**)&n->wb[l], sizeof(bf16_t) * 27 * bw_in[l] * bw_out[l], true);
  }
  // zero once: the channels that padding adds to the sixteen of x0 and dy4 are never written
  bf16_t** act[] = {&n->x0, &n->a1, &n->y1, &n->a2, &n->y2, &n->a3, &n->y3, &n->dy4, &n->dy3, &n->dy2, &n->dy1};
  const int ch[] = {16, 32, 32, 64, 64, 32, 32, 16, 32, 64, 32};
  for (int q = 0; q < 11; ++q) alloc((void**)act[q], sizeof(bf16_t) * act_elems(n, ch[q], max_batch), ch[q] == 16);
  alloc((void**)&n->ws, sizeof(float) * nws, false);
  alloc((void**)&n->loss, sizeof(float), false);
  alloc((void**)&n->flag, sizeof(int), true);
  if (!ok) {
    mx_cnn_destroy(n);
    set_error("mx_cnn_create: device allocation failed");
    return MX_ERR_OOM;
  }
  mx_status st = cnn_setup();
  if (st == MX_OK) st = make_maps(n);
  if (st != MX_OK || cudaDeviceSynchronize() != cudaSuccess) {
    mx_cnn_destroy(n);
    if (st == MX_OK) set_error("mx_cnn_create: set-up failed");
    return st != MX_OK ? st : MX_ERR_CUDA;
  }
  *out = n;
  return MX_OK;
}

mx_status mx_cnn_sync(mx_cnn* n, mx_stream_t stream) {
  clear_error();
  if (!n) {
    set_error("mx_cnn_sync: NULL net");
    return MX_ERR_INVALID_ARG;
  }
  int f = 0;
  MX_TRY(cnn_take_flag(n, (cudaStream_t)stream, &f));
  if (f & kFlagTimeout) {
    set_error("mx_cnn_sync: a bounded wait for the tensor cores ran out");
    return MX_ERR_TIMEOUT;
  }
  return MX_OK;
}

mx_status mx_cnn_set_params(mx_cnn* n, const float* params, mx_stream_t stream) {
  if (!n || !params) {
    set_error("mx_cnn_set_params: NULL argument");
    return MX_ERR_INVALID_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  MX_CUDA_TRY(cudaMemcpyAsync(n->params, params, sizeof(float) * num_params_total(), cudaMemcpyDeviceToDevice, st));
  MX_CUDA_TRY(cudaMemsetAsync(n->am, 0, sizeof(float) * num_params_total(), st));
  MX_CUDA_TRY(cudaMemsetAsync(n->av, 0, sizeof(float) * num_params_total(), st));
  n->adam_t = 0;
  return pack_all(n, st);
}

mx_status mx_cnn_get_params(const mx_cnn* n, float* params, mx_stream_t stream) {
  if (!n || !params) {
    set_error("mx_cnn_get_params: NULL argument");
    return MX_ERR_INVALID_ARG;
  }
  MX_CUDA_TRY(cudaMemcpyAsync(params, n->params, sizeof(float) * num_params_total(), cudaMemcpyDeviceToDevice,
                              (cudaStream_t)stream));
  return MX_OK;
}

mx_status mx_cnn_set_normalizer(mx_cnn* n, const double stats[12]) {
  if (!n || !stats) {
    set_error("mx_cnn_set_normalizer: NULL argument");
    return MX_ERR_INVALID_ARG;
  }
  for (int q = 0; q < 12; ++q) {
    if (!isfinite(stats[q]) || ((q % 6) >= 3 && !(stats[q] > 0))) {
      set_error("mx_cnn_set_normalizer: standard deviations must be > 0 and every entry finite");
      return MX_ERR_INVALID_ARG;
    }
    n->stats[q] = (float)stats[q];
  }
  return MX_OK;
}

static mx_status check_batch(const mx_cnn* n, const float* m, int batch, const char* what) {
  if (!n || !m || batch < 1 || batch > n->max_batch || (((uintptr_t)m) & 15)) {
    set_error(std::string(what) + ": bad network, pointer or batch (1..max_batch)");
    return MX_ERR_INVALID_ARG;
  }
  return MX_OK;
}

mx_status mx_cnn_forward(mx_cnn* n, const float* m, float* h, int batch, mx_stream_t stream) {
  MX_TRY(check_batch(n, m, batch, "mx_cnn_forward"));
  if (!h || (((uintptr_t)h) & 15)) {
    set_error("mx_cnn_forward: h must be a 16-byte aligned device pointer");
    return MX_ERR_INVALID_ARG;
  }
  return cnn_forward(n, (const float4*)m, (float4*)h, batch, (cudaStream_t)stream);
}

mx_status mx_cnn_loss_grad(mx_cnn* n, const float* m, const float* h_target, int batch, float* loss_out,
                           float* grad_out, mx_stream_t stream) {
  MX_TRY(check_batch(n, m, batch, "mx_cnn_loss_grad"));
  if (!h_target || (((uintptr_t)h_target) & 15)) {
    set_error("mx_cnn_loss_grad: h_target must be a 16-byte aligned device pointer");
    return MX_ERR_INVALID_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const long np = num_params_total();
  long nws = 0;
  const WgradOuts wo = wgrad_outs(&nws);
  float *G = n->grad, *ws = n->ws;
  const float *P = n->params, *s = n->stats;
  // (biases and weight sums are added to; the weights' gradient is then written whole)
  MX_CUDA_TRY(cudaMemsetAsync(n->loss, 0, sizeof(float), st));
  MX_CUDA_TRY(cudaMemsetAsync(G, 0, sizeof(float) * np, st));
  MX_CUDA_TRY(cudaMemsetAsync(ws, 0, sizeof(float) * nws, st));
  MX_TRY(cnn_hidden(n, (const float4*)m, batch, true, st));
  const ConvDims d = conv_dims(n, batch);
  auto bias = [&](float* base, int l) { return base + layer_w_off(l) + (long)kCh[l] * kCh[l + 1] * 27; };
  ConvArgs a{};
  a.d = d;
  a.flag = n->flag;
  // last layer with the loss and its gradient
  a.wk = n->wf[3], a.bias = bias((float*)P, 3), a.out = n->dy4, a.target = (const float4*)h_target;
  a.mean = make_float3(s[6], s[7], s[8]), a.sd = make_float3(1.f / s[9], 1.f / s[10], 1.f / s[11]);
  a.inv_count = 1.f / (3.f * (float)(n->cells * batch)), a.loss = n->loss, a.db = bias(G, 3);
  MX_TRY((conv_run<32, 8, CM_LOSS>(n->c_a3, a, st)));
  // per layer: dY of the layer below (with its bias gradient), then the weight gradient
  a.wk = n->wb[3], a.out = n->dy3, a.ypre = n->y3, a.db = bias(G, 2);
  MX_TRY((conv_run<16, 32, CM_BWD>(n->c_dy4, a, st)));
  MX_TRY((wgrad_run<16, 32>(n->s_dy4, n->r_a3, ws + wo.l[3].ws, d, n->flag, st)));
  a.wk = n->wb[2], a.out = n->dy2, a.ypre = n->y2, a.db = bias(G, 1);
  MX_TRY((conv_run<32, 64, CM_BWD>(n->c_dy3, a, st)));
  MX_TRY((wgrad_run<32, 64>(n->s_dy3, n->r_a2, ws + wo.l[2].ws, d, n->flag, st)));
  a.wk = n->wb[1], a.out = n->dy1, a.ypre = n->y1, a.db = bias(G, 0);
  MX_TRY((conv_run<64, 32, CM_BWD>(n->c_dy2, a, st)));
  MX_TRY((wgrad_run<32, 64>(n->s_a1, n->r_dy2, ws + wo.l[1].ws, d, n->flag, st)));
  MX_TRY((wgrad_run<16, 32>(n->s_x0, n->r_dy1, ws + wo.l[0].ws, d, n->flag, st)));
  launch_pdl(wgrad_finish_kernel, dim3((64 * 32 * 27 + 255) / 256, 4), dim3(256), 0, st, n->ws, G, wo);
  MX_TRY(launch_check("wgrad_finish_kernel"));
  if (loss_out) MX_CUDA_TRY(cudaMemcpyAsync(loss_out, n->loss, sizeof(float), cudaMemcpyDeviceToDevice, st));
  if (grad_out) MX_CUDA_TRY(cudaMemcpyAsync(grad_out, n->grad, sizeof(float) * np, cudaMemcpyDeviceToDevice, st));
  return MX_OK;
}

mx_status mx_cnn_adam_step(mx_cnn* n, double lr, double weight_decay, mx_stream_t stream) {
  if (!n || !(lr > 0) || !(weight_decay >= 0)) {
    set_error("mx_cnn_adam_step: need a network, lr > 0 and weight_decay >= 0");
    return MX_ERR_INVALID_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  n->adam_t += 1;
  MX_TRY(adam_update(n->params, n->grad, n->am, n->av, num_params_total(), lr, weight_decay, n->adam_t, st));
  return pack_all(n, st);
}

}  // extern "C"
