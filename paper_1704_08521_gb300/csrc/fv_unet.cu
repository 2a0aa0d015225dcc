// Learned initial guess of the pressure correction (no counterpart in the
// paper; an optional first pass of the SIMPLE-like loop of Section 3).
//
// A 3-D convolutional U-Net of 4 levels (16/32/48/64 channels, two 3x3x3
// convolutions + ReLU per level, 2x2x2 mean pooling, nearest upsampling,
// skip concatenation, a 1x1x1 float32 output layer) maps the float32
// right-hand side r = D w of the pressure equation plus three metric
// channels (log of the local cell widths) to a guess of phi.  Weights and
// activations are BF16, every contraction accumulates in float32.
//
// Kernels:
//   k_conv3   3x3x3 convolution, zero padding, as an implicit GEMM on the
//             BF16 tensor cores (mma.sync m16n8k16): rows = cells, columns =
//             output channels, reduction = 27 taps x input channels, operands
//             staged in shared memory by halo tiles; bias + ReLU fused.  The
//             decoder input (upsampled coarse output ++ skip) is gathered
//             while staging.  The same kernel computes the data gradient with
//             flipped, channel-transposed weights and the ReLU mask.
//   k_wgrad   weight gradients, dW_tap = dY^T X_tap of all taps of a tile,
//             also on the BF16 tensor cores; float32 atomics per block.
//   the rest  pooling, gradients of pooling / upsampling, output layer, the
//             mean-free mean-square loss and Adam are element-wise kernels.
// Layout: activations channel-last ([cell][channel], cells x fastest), every
// channel count a multiple of 16 (the 4 input channels are zero-padded to 16).
// Parameters (float32 master copy, BF16 mirror): per convolution c the
// weights W_c[27][cout][cin] (tap t = 9 (dz+1) + 3 (dy+1) + (dx+1)) then the
// bias b_c[cout]; finally the output layer's 16 weights and 1 bias.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <vector>

#include "fv_internal.cuh"

namespace fv {
namespace unet {

typedef __nv_bfloat16 bf16;

struct Dims {
  int nx, ny, nz;
};

// convolution layers: (level, cin, cout); level 0 is the finest
struct ConvSpec {
  int level, cin, cout;
};
constexpr int kNConv = 14;
constexpr ConvSpec kConvs[kNConv] = {
    {0, 16, 16},  {0, 16, 16},    // encoder level 0
    {1, 16, 32},  {1, 32, 32},    // encoder level 1
    {2, 32, 48},  {2, 48, 48},    // encoder level 2
    {3, 48, 64},  {3, 64, 64},    // bottom
    {2, 112, 48}, {2, 48, 48},    // decoder level 2: up(64) ++ skip(48)
    {1, 80, 32},  {1, 32, 32},    // decoder level 1: up(48) ++ skip(32)
    {0, 48, 16},  {0, 16, 16},    // decoder level 0: up(32) ++ skip(16)
};

__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// ------------------------------------------------------------ conv tiles --
// Both contraction kernels work on spatial tiles of 8 x 4 x 4 cells (level
// dims are 8, 4, 2, 1 times any integer, so the tiles of level 0 are whole in
// x and y) staged once, with a one-cell halo, in shared memory as
// [halo cell][channel] rows.  A row is padded by 16 bytes: with channel counts
// that are multiples of 16 the row stride is then 16 modulo 32 bytes, so the
// eight 16-byte rows of an ldmatrix tile fall in different bank groups.
constexpr int kTX = 8, kTY = 4, kTZ = 4;
constexpr int kTile = kTX * kTY * kTZ;                              // 128 cells
constexpr int kHX = kTX + 2, kHY = kTY + 2, kHZ = kTZ + 2;
constexpr int kHalo = kHX * kHY * kHZ;                              // 360 cells

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// 16 bytes global -> shared, zeros when !valid (src is not read then)
__device__ __forceinline__ void cpa16z(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cpa_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

// the input of a convolution: X [cell][xc] alone, or (low != null) the decoder
// input, channels [0, lowc) from the next coarser level (nearest upsampling),
// the xc others from the skip X
struct ConvIn {
  const bf16* X;
  int xc;
  const bf16* low;
  int lowc;
};

// first cell of spatial tile b of the level
__device__ __forceinline__ void tile_origin(int b, const Dims& d, int& i, int& j, int& k) {
  const int tx = (d.nx + kTX - 1) / kTX, ty = (d.ny + kTY - 1) / kTY;
  i = (b % tx) * kTX;
  j = (b / tx % ty) * kTY;
  k = b / (tx * ty) * kTZ;
}

// channels [c0, c0 + NCH) of the halo of the tile at (i0, j0, k0) -> xs
// (row pitch NCH + 8 elements); zeros outside the box.  The source of a
// 16-byte run does not change within it: lowc, xc, c0 are multiples of 8.
template <int NCH, int NTHR>
__device__ __forceinline__ void stage_halo(bf16* xs, const ConvIn& in, int c0, int i0, int j0, int k0,
                                           const Dims& d, int tid) {
  constexpr int runs = NCH / 8, pitch = NCH + 8;
#pragma unroll 4
  for (int e = tid; e < kHalo * runs; e += NTHR) {
    const int h = e / runs, c = c0 + 8 * (e - h * runs);
    const int i = i0 + h % kHX - 1, j = j0 + h / kHX % kHY - 1, k = k0 + h / (kHX * kHY) - 1;
    const bool ok = (unsigned)i < (unsigned)d.nx && (unsigned)j < (unsigned)d.ny && (unsigned)k < (unsigned)d.nz;
    const bf16* src = in.X;
    if (ok) {
      if (c < in.lowc) {
        const size_t cc = ((size_t)(k >> 1) * (d.ny >> 1) + (j >> 1)) * (d.nx >> 1) + (i >> 1);
        src = in.low + cc * in.lowc + c;
      } else {
        const size_t cc = ((size_t)k * d.ny + j) * d.nx + i;
        src = in.X + cc * in.xc + (c - in.lowc);
      }
    }
    cpa16z(xs + h * pitch + (c - c0), src, ok);
  }
}

// Y[cell][co] = act(bias[co] + sum_{t, ci} X[nb(cell, t)][ci] W[t][co][ci]),
// zero padding; Y has row stride ny_ch.  A block computes 16 output channels
// (blockIdx.y) of one tile: the halo of X and the 27 x 16 x cin weights are
// staged once, each of the 4 warps accumulates two 16-cell rows of MMA tiles.
//   DGRAD: the data gradient with the same kernel: X is the output gradient,
//   W[t][co][ci] the layer's weights taken as W[26 - t], co the reduction
//   index; the [co][ci] rows are read transposed by ldmatrix.trans, so no
//   flipped copy is made.  mask (optional): Y is zeroed where mask <= 0 (the
//   ReLU of the layer that produced this input).
// mma.sync rather than tcgen05: a choice, not a bound.  Taps and channel chunks
// could be issued to a tensor-memory accumulator in this order as well; its sums
// would round differently inside a step of 16 channels, and with the last bit of a
// float32 sum stored BF16 values and ReLU decisions downstream flip.
// Bound by launch latency at the coarse levels (8^3..16^3 cells) and by shared
// memory at level 0 (3 KB of fragments per 16 KFLOP).  Measured 33 us for
// 16 -> 16 at 64^3 and 10 us for 64 -> 64 at 8^3; the version that read its
// fragments from global memory took 111 us and 183 us (8 blocks).
//   CIN is a template argument so that the staging's index arithmetic and the
//   channel loop are constants.
//   MT: 16-cell MMA rows per warp (2: 4 warps; 1: 8 warps, for the levels
//   whose few blocks leave SMs idle and whose time is one block's chain).
template <int CIN, bool DGRAD, int MT>
__global__ void __launch_bounds__(256 / MT) k_conv3(ConvIn in, const bf16* __restrict__ W,
                                               const float* __restrict__ bias, bf16* __restrict__ Y,
                                               int cout, const bf16* __restrict__ mask, Dims d) {
  extern __shared__ __align__(16) unsigned char sm[];
  constexpr int pitch = CIN + 8, NTHR = 256 / MT;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  bf16* xs = reinterpret_cast<bf16*>(sm);
  bf16* ws = xs + kHalo * pitch;
  const int n0 = blockIdx.y * 16;
  int i0, j0, k0;
  tile_origin(blockIdx.x, d, i0, j0, k0);
  stage_halo<CIN, NTHR>(xs, in, 0, i0, j0, k0, d, tid);
  if (DGRAD) {        // rows (t, reduction index), 16 outputs each, pitch 24
#pragma unroll 4
    for (int e = tid; e < 27 * CIN * 2; e += NTHR) {
      const int r = e >> 1, h = e & 1;
      cpa16z(ws + r * 24 + 8 * h, W + (size_t)r * cout + n0 + 8 * h, true);
    }
  } else {            // rows (t, output), CIN each
    constexpr int runs = CIN / 8;
#pragma unroll 4
    for (int e = tid; e < 27 * 16 * runs; e += NTHR) {
      const int r = e / runs, q = e - r * runs;
      cpa16z(ws + r * pitch + 8 * q, W + ((size_t)(r >> 4) * cout + n0 + (r & 15)) * CIN + 8 * q, true);
    }
  }
  cpa_wait_all();
  __syncthreads();
  float acc[MT][2][4];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[m][n][q] = 0.f;
  // ldmatrix source rows of this lane: A, cell row (lane & 15), channel half
  // lane >> 4; B, see below
  uint32_t abase[MT];
#pragma unroll
  for (int m = 0; m < MT; ++m) {
    const int c = (MT * warp + m) * 16 + (lane & 15);
    const int x = c % kTX, y = c / kTX % kTY, z = c / (kTX * kTY);
    abase[m] = smem_u32(xs + ((z * kHY + y) * kHX + x) * pitch + (lane >> 4) * 8);
  }
  const uint32_t bbase = DGRAD
      ? smem_u32(ws + ((lane & 7) + ((lane >> 3) & 1) * 8) * 24 + (lane >> 4) * 8)
      : smem_u32(ws + ((lane & 7) + (lane >> 4) * 8) * pitch + ((lane >> 3) & 1) * 8);
  for (int tz = 0; tz < 3; ++tz) {
#pragma unroll
    for (int ty = 0; ty < 3; ++ty) {
#pragma unroll
      for (int tx = 0; tx < 3; ++tx) {
        const uint32_t aoff = (uint32_t)(((tz * kHY + ty) * kHX + tx) * pitch) * 2;
        const int t = 9 * tz + 3 * ty + tx;
        const uint32_t boff = DGRAD ? (uint32_t)((26 - t) * CIN * 24) * 2 : (uint32_t)(t * 16 * pitch) * 2;
#pragma unroll
        for (int kc = 0; kc < CIN; kc += 16) {
          uint32_t a[MT][4], b[4];
#pragma unroll
          for (int m = 0; m < MT; ++m) ldsm4(a[m], abase[m] + aoff + kc * 2);
          if (DGRAD) ldsm4t(b, bbase + boff + kc * 48);
          else ldsm4(b, bbase + boff + kc * 2);
          const uint32_t b0[2] = {b[0], b[1]}, b1[2] = {b[2], b[3]};
#pragma unroll
          for (int m = 0; m < MT; ++m) {
            mma_bf16(acc[m][0], a[m], b0);
            mma_bf16(acc[m][1], a[m], b1);
          }
        }
      }
    }
  }
  // accumulator q: row g + 8 (q >> 1), column 2 t4 + (q & 1)
  const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int c = (MT * warp + m) * 16 + g + 8 * hh;
      const int i = i0 + c % kTX, j = j0 + c / kTX % kTY, k = k0 + c / (kTX * kTY);
      if (i >= d.nx || j >= d.ny || k >= d.nz) continue;
      const size_t o = (((size_t)k * d.ny + j) * d.nx + i) * cout + n0 + 2 * t4;
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        float v0 = acc[m][n][2 * hh] + (bias ? bias[n0 + n * 8 + 2 * t4] : 0.f);
        float v1 = acc[m][n][2 * hh + 1] + (bias ? bias[n0 + n * 8 + 2 * t4 + 1] : 0.f);
        if (!DGRAD) { v0 = fmaxf(v0, 0.f); v1 = fmaxf(v1, 0.f); }   // ReLU
        if (mask) {
          const __nv_bfloat162 y = *reinterpret_cast<const __nv_bfloat162*>(mask + o + n * 8);
          if (!(__bfloat162float(y.x) > 0.f)) v0 = 0.f;
          if (!(__bfloat162float(y.y) > 0.f)) v1 = 0.f;
        }
        *reinterpret_cast<uint32_t*>(Y + o + n * 8) = pack2(__float2bfloat16(v0), __float2bfloat16(v1));
      }
    }
}

inline size_t conv_smem(int cin, bool dgrad) {
  return sizeof(bf16) * ((size_t)kHalo * (cin + 8) + (dgrad ? (size_t)27 * cin * 24 : (size_t)27 * 16 * (cin + 8)));
}

// dW[t][co][ci] += sum over cells dY[cell][co] X[nb(cell, t)][ci], db[co] +=
// sum dY[cell][co].  blockIdx.y = (16-channel tile of co, 16 NCI channels of
// ci); the block walks over tiles blockIdx.x, + gridDim.x, ..., stages dY and
// the halo of X, and each of its 9 warps keeps the accumulators of 3 taps in
// registers over all of them (M = 16 co, N = 16 NCI ci, K = cells; dY and X
// are read through ldmatrix.trans), so a weight is added to global memory
// once per block.  Per 16 cells a warp reads 0.5 KB of dY and 1.5 NCI KB of X
// for 6 NCI MMAs.  The version with one warp per (tap, 16 x 16) tile gathered
// 2-byte elements from global memory: 375 us per 16 -> 16 layer at 64^3, 28 us here.
template <int NCI>
__global__ void __launch_bounds__(288) k_wgrad(const bf16* __restrict__ dY, int cout, ConvIn in,
                                               int cin, float* __restrict__ dW,
                                               float* __restrict__ db, Dims d, int ntile) {
  constexpr int CI = 16 * NCI, XP = CI + 8, YP = 24;
  __shared__ __align__(16) bf16 xs[kHalo * XP];
  __shared__ __align__(16) bf16 ys[kTile * YP];
  __shared__ float sb[16];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ncc = cin / CI;
  const int co0 = (blockIdx.y / ncc) * 16, ci0 = (blockIdx.y % ncc) * CI;
  const bool do_bias = ci0 == 0;
  float acc[3][2 * NCI][4];
#pragma unroll
  for (int t = 0; t < 3; ++t)
#pragma unroll
    for (int n = 0; n < 2 * NCI; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[t][n][q] = 0.f;
  float bsum = 0.f;
  if (tid < 16) sb[tid] = 0.f;
  // A = dY^T from [cell][co] rows, B = X from [cell][ci] rows, both transposed
  const uint32_t abase = smem_u32(ys + ((lane & 7) + (lane >> 4) * 8) * YP + ((lane >> 3) & 1) * 8);
  const int kr = (lane & 7) + ((lane >> 3) & 1) * 8;   // cell row of the 16 this lane addresses for B
  uint32_t toff[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int t = 3 * warp + q;
    toff[q] = (uint32_t)((((t / 9) * kHY + (t / 3) % 3) * kHX + t % 3) * XP) * 2;
  }
  for (int b = blockIdx.x; b < ntile; b += gridDim.x) {
    int i0, j0, k0;
    tile_origin(b, d, i0, j0, k0);
    __syncthreads();                          // the previous tile is consumed
    stage_halo<CI, 288>(xs, in, ci0, i0, j0, k0, d, tid);
    if (tid < 2 * kTile) {
      const int c = tid >> 1, h = tid & 1;
      const int i = i0 + c % kTX, j = j0 + c / kTX % kTY, k = k0 + c / (kTX * kTY);
      const bool ok = i < d.nx && j < d.ny && k < d.nz;
      const size_t o = ok ? (((size_t)k * d.ny + j) * d.nx + i) * cout + co0 + 8 * h : 0;
      cpa16z(ys + c * YP + 8 * h, dY + o, ok);
    }
    cpa_wait_all();
    __syncthreads();
    if (do_bias && tid < 256) {
#pragma unroll
      for (int q = 0; q < kTile / 16; ++q) bsum += __bfloat162float(ys[(q * 16 + (tid >> 4)) * YP + (tid & 15)]);
    }
#pragma unroll 2
    for (int s = 0; s < kTile / 16; ++s) {
      uint32_t a[4];
      ldsm4t(a, abase + s * 16 * YP * 2);
      const int c = s * 16 + kr;
      const int x = c % kTX, y = c / kTX % kTY, z = c / (kTX * kTY);
      const uint32_t bb = smem_u32(xs + ((z * kHY + y) * kHX + x) * XP + (lane >> 4) * 8);
#pragma unroll
      for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int n = 0; n < NCI; ++n) {
          uint32_t r[4];
          ldsm4t(r, bb + toff[q] + n * 32);
          const uint32_t b0[2] = {r[0], r[1]}, b1[2] = {r[2], r[3]};
          mma_bf16(acc[q][2 * n], a, b0);
          mma_bf16(acc[q][2 * n + 1], a, b1);
        }
    }
  }
  const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int n = 0; n < 2 * NCI; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int co = co0 + g + 8 * (e >> 1);
        const int c = ci0 + n * 8 + 2 * t4 + (e & 1);
        atomicAdd(dW + ((size_t)(3 * warp + q) * cout + co) * cin + c, acc[q][n][e]);
      }
  if (do_bias) {
    if (tid < 256) {                          // lanes l and l + 16 hold the same channel
      bsum += __shfl_xor_sync(0xffffffffu, bsum, 16);
      if (lane < 16) atomicAdd(&sb[lane], bsum);
    }
    __syncthreads();
    if (tid < 16) atomicAdd(db + co0 + tid, sb[tid]);
  }
}

// eight BF16 channels of a 16-byte run
struct Run8 {
  float v[8];
};
__device__ __forceinline__ Run8 load8(const bf16* p) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
  Run8 r;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    r.v[2 * q] = __uint_as_float(w[q] << 16);
    r.v[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u);
  }
  return r;
}
__device__ __forceinline__ void store8(bf16* p, const Run8& r) {
  uint32_t w[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) w[q] = pack2(__float2bfloat16(r.v[2 * q]), __float2bfloat16(r.v[2 * q + 1]));
  *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}
// zero r where the ReLU output at y is not positive
__device__ __forceinline__ void mask8(Run8& r, const bf16* y) {
  const Run8 m = load8(y);
#pragma unroll
  for (int q = 0; q < 8; ++q)
    if (!(m.v[q] > 0.f)) r.v[q] = 0.f;
}

// 2x2x2 mean pooling of X (fine dims d, ch channels) into Y (coarse); one
// thread per cell and 8 channels, as in the two kernels below
__global__ void k_pool(const bf16* __restrict__ X, bf16* __restrict__ Y, int ch, Dims d) {
  const int cx = d.nx / 2, cy = d.ny / 2, cz = d.nz / 2, runs = ch >> 3;
  const int64_t n = (int64_t)cx * cy * cz * runs;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(e / runs), k = 8 * (int)(e - (int64_t)c * runs);
    const int i = c % cx, j = (c / cx) % cy, l = c / (cx * cy);
    Run8 s = {};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int f = ((2 * l + (q >> 2)) * d.ny + 2 * j + ((q >> 1) & 1)) * d.nx + 2 * i + (q & 1);
      const Run8 x = load8(X + (size_t)f * ch + k);
#pragma unroll
      for (int o = 0; o < 8; ++o) s.v[o] += x.v[o];
    }
#pragma unroll
    for (int o = 0; o < 8; ++o) s.v[o] *= 0.125f;
    store8(Y + (size_t)c * ch + k, s);
  }
}

// gradient of an encoder output that feeds the pooling (dY, coarse) and the
// skip (dS): dX[f] = dS[f] + dY[coarse(f)] / 8, zero where act <= 0
__global__ void k_pool_back(const bf16* __restrict__ dY, const bf16* __restrict__ dS,
                            const bf16* __restrict__ act, bf16* __restrict__ dX, int ch, Dims d) {
  const int cx = d.nx / 2, cy = d.ny / 2, runs = ch >> 3;
  const int64_t n = (int64_t)d.nx * d.ny * d.nz * runs;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int f = (int)(e / runs), k = 8 * (int)(e - (int64_t)f * runs);
    const int i = f % d.nx, j = (f / d.nx) % d.ny, l = f / (d.nx * d.ny);
    const int c = ((l / 2) * cy + j / 2) * cx + i / 2;
    Run8 s = load8(dS + (size_t)f * ch + k);
    const Run8 y = load8(dY + (size_t)c * ch + k);
#pragma unroll
    for (int o = 0; o < 8; ++o) s.v[o] += 0.125f * y.v[o];
    mask8(s, act + (size_t)f * ch + k);
    store8(dX + (size_t)f * ch + k, s);
  }
}

// gradient of a decoder input [low (upsampled, lowc ch), skip]: dXl[c] = sum
// of the 8 fine gradients, zero where the low output actl <= 0; dS[f] = the
// remaining channels
__global__ void k_up_cat_back(const bf16* __restrict__ dY, int lowc, int skipc,
                              const bf16* __restrict__ actl, bf16* __restrict__ dXl,
                              bf16* __restrict__ dS, Dims d) {
  const int ch = lowc + skipc, lr = lowc >> 3, sr = skipc >> 3;
  const int cx = d.nx / 2, cy = d.ny / 2, cz = d.nz / 2;
  const int64_t nc = (int64_t)cx * cy * cz * lr;
  const int64_t nf = (int64_t)d.nx * d.ny * d.nz * sr;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nc + nf; e += (int64_t)gridDim.x * blockDim.x) {
    if (e < nc) {
      const int c = (int)(e / lr), k = 8 * (int)(e - (int64_t)c * lr);
      const int i = c % cx, j = (c / cx) % cy, l = c / (cx * cy);
      Run8 s = {};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int f = ((2 * l + (q >> 2)) * d.ny + 2 * j + ((q >> 1) & 1)) * d.nx + 2 * i + (q & 1);
        const Run8 y = load8(dY + (size_t)f * ch + k);
#pragma unroll
        for (int o = 0; o < 8; ++o) s.v[o] += y.v[o];
      }
      mask8(s, actl + (size_t)c * lowc + k);
      store8(dXl + (size_t)c * lowc + k, s);
    } else {
      const int64_t e2 = e - nc;
      const int f = (int)(e2 / sr), k = 8 * (int)(e2 - (int64_t)f * sr);
      *reinterpret_cast<uint4*>(dS + (size_t)f * skipc + k) =
          *reinterpret_cast<const uint4*>(dY + (size_t)f * ch + lowc + k);
    }
  }
}

// raw input planes in[4][ncell] (float32) -> X[ncell][16] (channels 4..15 zero)
__global__ void k_pack_planes(const float* __restrict__ in, bf16* __restrict__ X, int ncell) {
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
    Run8 r = {};
#pragma unroll
    for (int k = 0; k < 4; ++k) r.v[k] = in[(size_t)k * ncell + c];
    store8(X + (size_t)c * 16, r);
    store8(X + (size_t)c * 16 + 8, Run8{});
  }
}

// max |r| (non-negative floats order like their bit patterns)
__global__ void k_absmax(const float* __restrict__ r, int64_t n, unsigned* out) {
  float m = 0.f;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    m = fmaxf(m, fabsf(r[e]));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

// local cell scale h_c^2 = (dx_i dy_j dz_k)^(2/3): r h^2 is the right-hand
// side of the pressure equation in index units (unit spacing)
__device__ __forceinline__ float cell_h2(int c, int nx, int ny, const float* idx0, const float* idx1,
                                         const float* idx2) {
  const int i = c % nx, j = (c / nx) % ny, k = c / (nx * ny);
  return cbrtf(1.f / (idx0[i] * idx1[j] * idx2[k]));
}

// red[2] += sum (r h^2)^2
__global__ void k_rhs_sumsq(const float* __restrict__ r, int nx, int ny, int nz,
                            const float* __restrict__ idx0, const float* __restrict__ idx1,
                            const float* __restrict__ idx2, double* red) {
  const int ncell = nx * ny * nz;
  double s = 0.0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
    const float hh = cell_h2(c, nx, ny, idx0, idx1, idx2);
    const double q = (double)r[c] * (double)(hh * hh);
    s += q * q;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(red + 2, s);
}

// solver input: X[c] = [q_c / S, log(n_x dx_i), log(n_y dy_j), log(n_z dz_k), 0...],
// q = r h^2, S = rms(q) (written to *scale; 0 when r = 0)
__global__ void k_pack_rhs(const float* __restrict__ r, const double* __restrict__ red, int nx,
                           int ny, int nz, const float* __restrict__ idx0,
                           const float* __restrict__ idx1, const float* __restrict__ idx2,
                           bf16* __restrict__ X, float* __restrict__ scale) {
  const int ncell = nx * ny * nz;
  const float S = (float)sqrt(red[2] / ncell);
  const float inv = S > 0.f ? 1.f / S : 0.f;
  if (blockIdx.x == 0 && threadIdx.x == 0) *scale = S;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
    const int i = c % nx, j = (c / nx) % ny, k = c / (nx * ny);
    const float hh = cell_h2(c, nx, ny, idx0, idx1, idx2);
    bf16* o = X + (size_t)c * 16;
    o[0] = __float2bfloat16(r[c] * (hh * hh) * inv);
    o[1] = __float2bfloat16(logf(nx / idx0[i]));
    o[2] = __float2bfloat16(logf(ny / idx1[j]));
    o[3] = __float2bfloat16(logf(nz / idx2[k]));
#pragma unroll
    for (int q = 4; q < 16; ++q) o[q] = __float2bfloat16(0.f);
  }
}

// phi[c] = out[c] * S  (undo the normalisation of input and target)
__global__ void k_unscale(const float* __restrict__ out, const float* __restrict__ scale,
                          float* __restrict__ phi, int n) {
  const float m = *scale;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) phi[c] = out[c] * m;
}

// normalised training target t[c] = phi[c] / S
__global__ void k_scale_target(const double* __restrict__ phi, const float* __restrict__ scale,
                               float* __restrict__ t, int n) {
  const float m = *scale;
  const float s = m > 0.f ? 1.f / m : 0.f;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x)
    t[c] = (float)phi[c] * s;
}

__global__ void k_to_f32(const double* __restrict__ a, float* __restrict__ b, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    b[e] = (float)a[e];
}

// output layer: out[c] = b + sum_k w[k] H[c][k]
__global__ void k_head(const bf16* __restrict__ H, const float* __restrict__ w,
                       const float* __restrict__ b, float* __restrict__ out, int ncell) {
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
    float s = b[0];
#pragma unroll
    for (int k = 0; k < 16; ++k) s += w[k] * __bfloat162float(H[(size_t)c * 16 + k]);
    out[c] = s;
  }
}

// red[0] += sum (out - t)
__global__ void k_err_sum(const float* __restrict__ out, const float* __restrict__ t, int n,
                          double* red) {
  double s = 0.0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x)
    s += (double)out[c] - (double)t[c];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(red, s);
}

// mean-free square loss L = mean (e - mean e)^2, e = out - t.  red[1] += L,
// dH = dL/dout * w (BF16; zero where the ReLU output H <= 0), dw[k] += sum
// dL/dout H[k], db += sum dL/dout.  The 17 sums are reduced over the warp
// before they reach shared memory (one atomic per warp and sum).
__global__ void k_head_back(const bf16* __restrict__ H, const float* __restrict__ w,
                            const float* __restrict__ out, const float* __restrict__ t, int n,
                            double* red, bf16* __restrict__ dH, float* __restrict__ dw,
                            float* __restrict__ db) {
  __shared__ float sg[17];
  if (threadIdx.x < 17) sg[threadIdx.x] = 0.f;
  __syncthreads();
  const double ebar = red[0] / n;
  double l = 0.0;
  float gw[17];
#pragma unroll
  for (int k = 0; k < 17; ++k) gw[k] = 0.f;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
    const double e = (double)out[c] - (double)t[c] - ebar;
    l += e * e / n;
    const float go = (float)(2.0 * e / n);
    gw[16] += go;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const Run8 x = load8(H + (size_t)c * 16 + 8 * h);
      Run8 y;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        gw[8 * h + k] += go * x.v[k];
        y.v[k] = x.v[k] > 0.f ? go * w[8 * h + k] : 0.f;
      }
      store8(dH + (size_t)c * 16 + 8 * h, y);
    }
  }
#pragma unroll
  for (int k = 0; k < 17; ++k) {
    for (int o = 16; o > 0; o >>= 1) gw[k] += __shfl_xor_sync(0xffffffffu, gw[k], o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&sg[k], gw[k]);
  }
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(red + 1, l);
  __syncthreads();
  if (threadIdx.x < 16) atomicAdd(dw + threadIdx.x, sg[threadIdx.x]);
  if (threadIdx.x == 16) atomicAdd(db, sg[16]);
}

// Adam (Kingma & Ba 2015) on the float32 parameters; refreshes the BF16 mirror
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ gr, float* __restrict__ m,
                       float* __restrict__ v, bf16* __restrict__ pb, int n, float lr, float b1,
                       float b2, float c1, float c2) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const float g = gr[e];
    const float mm = b1 * m[e] + (1.f - b1) * g;
    const float vv = b2 * v[e] + (1.f - b2) * g * g;
    m[e] = mm;
    v[e] = vv;
    const float q = p[e] - lr * (mm / c1) / (sqrtf(vv / c2) + 1e-8f);
    p[e] = q;
    pb[e] = __float2bfloat16(q);
  }
}

__global__ void k_mirror(const float* __restrict__ a, bf16* __restrict__ b, int n) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x)
    b[e] = __float2bfloat16(a[e]);
}

inline unsigned blocks_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  b = std::min<int64_t>(b, 152 * 16);
  return (unsigned)std::max<int64_t>(b, 1);
}

}  // namespace unet
}  // namespace fv

struct fv_unet {
  cudaStream_t stream = nullptr;
  int nparam = 0;
  int woff[fv::unet::kNConv] = {}, boff[fv::unet::kNConv] = {};
  int head_w = 0, head_b = 0;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;   // params, grads, Adam moments
  fv::unet::bf16* pb = nullptr;   // BF16 mirror of the parameters
  int step = 0;
  // activation workspace, sized for cap cells at level 0 (level l: cap / 8^l)
  int64_t cap = 0, gcap = 0;
  int n[4][3] = {};
  int64_t ncell[4] = {};
  bool have_fwd = false;          // a forward pass at the current dims is in the buffers
  fv::unet::bf16* in16 = nullptr;
  fv::unet::bf16* act[fv::unet::kNConv] = {};
  fv::unet::bf16* pool[3] = {};   // pooled encoder outputs (inputs of levels 1..3)
  float* out = nullptr;           // network output [cells]
  float* tgt = nullptr;           // normalised target [cells]
  double* red = nullptr;          // reductions: loss (0, 1), right-hand side (2)
  float* scale = nullptr;         // normalisation S of the last packed right-hand side
  // gradient workspace (allocated by the first backward pass)
  fv::unet::bf16 *gA = nullptr, *gB = nullptr, *gC = nullptr;
  fv::unet::bf16* gS[3] = {};
};

namespace fv {
namespace unet {

static fv_status dalloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    *p = nullptr;
    set_error("unet: device allocation failed");
    return FV_ENOMEM;
  }
  return FV_OK;
}

static void dfree(void* p) {
  if (p) cudaFree(p);
}

static void free_ws(fv_unet* u) {
  dfree(u->in16);
  for (auto& a : u->act) { dfree(a); a = nullptr; }
  for (auto& p : u->pool) { dfree(p); p = nullptr; }
  dfree(u->out); dfree(u->tgt);
  u->in16 = nullptr; u->out = u->tgt = nullptr;
  u->cap = 0;
  u->have_fwd = false;
}

static void free_grad(fv_unet* u) {
  dfree(u->gA); dfree(u->gB); dfree(u->gC);
  u->gA = u->gB = u->gC = nullptr;
  for (auto& s : u->gS) { dfree(s); s = nullptr; }
  u->gcap = 0;
}

static bool dims_ok(int nx, int ny, int nz) {
  auto ok = [](int v) { return v >= 8 && v <= 1024 && v % 8 == 0; };
  return ok(nx) && ok(ny) && ok(nz) && (int64_t)nx * ny * nz <= (int64_t)1 << 27;
}

// set the level dims and make sure the activation buffers hold them
static fv_status ensure_ws(fv_unet* u, int nx, int ny, int nz) {
  if (!dims_ok(nx, ny, nz)) {
    set_error("unet: every dimension must be a multiple of 8 in [8, 1024], at most 2^27 cells");
    return FV_EINVAL;
  }
  const int64_t nc = (int64_t)nx * ny * nz;
  if (nc > u->cap) {
    free_ws(u);
    free_grad(u);
    fv_status s = FV_OK;
    auto A = [&](void** p, size_t b) { if (s == FV_OK) s = dalloc(p, b); };
    A((void**)&u->in16, (size_t)nc * 16 * sizeof(bf16));
    for (int c = 0; c < kNConv; ++c)
      A((void**)&u->act[c], (size_t)(nc >> (3 * kConvs[c].level)) * kConvs[c].cout * sizeof(bf16));
    for (int q = 0; q < 3; ++q)
      A((void**)&u->pool[q], (size_t)(nc >> (3 * (q + 1))) * kConvs[2 * q + 1].cout * sizeof(bf16));
    A((void**)&u->out, (size_t)nc * sizeof(float));
    A((void**)&u->tgt, (size_t)nc * sizeof(float));
    if (s != FV_OK) { free_ws(u); return s; }
    u->cap = nc;
  }
  const int d[3] = {nx, ny, nz};
  bool same = true;
  for (int a = 0; a < 3; ++a) same = same && u->n[0][a] == d[a];
  for (int l = 0; l < 4; ++l) {
    for (int a = 0; a < 3; ++a) u->n[l][a] = d[a] >> l;
    u->ncell[l] = nc >> (3 * l);
  }
  if (!same) u->have_fwd = false;
  return FV_OK;
}

// Gradient buffers: gA/gB hold one layer's output gradient (at most 16
// channels at level 0; a level l >= 1 holds at most 112 channels on 1/8^l
// of the cells), gC the decoder-input gradient (at most 48 channels at
// level 0), gS[l] the skip gradient of encoder level l.
static fv_status ensure_grad(fv_unet* u) {
  const int64_t nc = u->cap;
  if (u->gcap >= nc) return FV_OK;
  free_grad(u);
  fv_status s = FV_OK;
  auto A = [&](void** p, size_t b) { if (s == FV_OK) s = dalloc(p, b); };
  A((void**)&u->gA, (size_t)nc * 16 * sizeof(bf16));
  A((void**)&u->gB, (size_t)nc * 16 * sizeof(bf16));
  A((void**)&u->gC, (size_t)nc * 48 * sizeof(bf16));
  for (int l = 0; l < 3; ++l) A((void**)&u->gS[l], (size_t)(nc >> (3 * l)) * kConvs[2 * l + 1].cout * sizeof(bf16));
  if (s != FV_OK) { free_grad(u); return s; }
  u->gcap = nc;
  return FV_OK;
}

#define UNET_LAUNCH(...)   \
  do {                     \
    ::fv::count_launch();  \
    __VA_ARGS__;           \
    FV_CHECK_LAUNCH();     \
  } while (0)

inline int tiles(const int n[3]) {
  return ((n[0] + kTX - 1) / kTX) * ((n[1] + kTY - 1) / kTY) * ((n[2] + kTZ - 1) / kTZ);
}

template <int CIN, bool DGRAD>
static fv_status conv_t(cudaStream_t st, const ConvIn& in, const bf16* W, const float* bias, bf16* Y,
                        int cout, const bf16* mask, const int n[3]) {
  const Dims d{n[0], n[1], n[2]};
  const dim3 grid(tiles(n), cout / 16);
  const size_t smem = conv_smem(CIN, DGRAD);
  // at least one block per SM: throughput counts, two MMA rows share a weight
  // fragment; fewer: one block's chain of taps counts, half as long with one
  if ((int64_t)grid.x * grid.y >= 152)
    UNET_LAUNCH((k_conv3<CIN, DGRAD, 2><<<grid, 128, smem, st>>>(in, W, bias, Y, cout, mask, d)));
  else
    UNET_LAUNCH((k_conv3<CIN, DGRAD, 1><<<grid, 256, smem, st>>>(in, W, bias, Y, cout, mask, d)));
  return FV_OK;
}

template <bool DGRAD>
static fv_status conv_any(cudaStream_t st, const ConvIn& in, int cin, const bf16* W, const float* bias,
                          bf16* Y, int cout, const bf16* mask, const int n[3]) {
  switch (cin) {
    case 16: return conv_t<16, DGRAD>(st, in, W, bias, Y, cout, mask, n);
    case 32: return conv_t<32, DGRAD>(st, in, W, bias, Y, cout, mask, n);
    case 48: return conv_t<48, DGRAD>(st, in, W, bias, Y, cout, mask, n);
    case 64: return conv_t<64, DGRAD>(st, in, W, bias, Y, cout, mask, n);
  }
  if constexpr (!DGRAD) {
    if (cin == 80) return conv_t<80, false>(st, in, W, bias, Y, cout, mask, n);
    if (cin == 112) return conv_t<112, false>(st, in, W, bias, Y, cout, mask, n);
  }
  set_error("unet: unsupported channel count");
  return FV_EINVAL;
}

template <int CIN, bool DGRAD>
static fv_status conv_attr() {
  const int b = (int)conv_smem(CIN, DGRAD);
  FV_CUDA(cudaFuncSetAttribute(k_conv3<CIN, DGRAD, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
  FV_CUDA(cudaFuncSetAttribute(k_conv3<CIN, DGRAD, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
  return FV_OK;
}

// up to 190 KB of shared memory (112 input channels)
static fv_status set_conv_attributes() {
  FV_TRY((conv_attr<16, false>()));
  FV_TRY((conv_attr<32, false>()));
  FV_TRY((conv_attr<48, false>()));
  FV_TRY((conv_attr<64, false>()));
  FV_TRY((conv_attr<80, false>()));
  FV_TRY((conv_attr<112, false>()));
  FV_TRY((conv_attr<16, true>()));
  FV_TRY((conv_attr<32, true>()));
  FV_TRY((conv_attr<48, true>()));
  FV_TRY((conv_attr<64, true>()));
  return FV_OK;
}

// activations of layer c from its input
static fv_status conv(fv_unet* u, int c, const ConvIn& in) {
  const ConvSpec& s = kConvs[c];
  return conv_any<false>(u->stream, in, s.cin, u->pb + u->woff[c], u->p + u->boff[c], u->act[c], s.cout,
                         nullptr, u->n[s.level]);
}

// input of the first convolution of decoder level q: [up(low), skip]
static ConvIn decoder_in(const fv_unet* u, int q) {
  const int l = 2 - q, lowl = q > 0 ? 9 + 2 * (q - 1) : 7;
  return {u->act[2 * l + 1], kConvs[2 * l + 1].cout, u->act[lowl], kConvs[lowl].cout};
}

static ConvIn plain_in(const bf16* X, int c) { return {X, kConvs[c].cin, nullptr, 0}; }

// forward pass from u->in16 to u->out
static fv_status forward(fv_unet* u) {
  cudaStream_t st = u->stream;
  const bf16* X = u->in16;
  for (int l = 0; l < 4; ++l) {
    const int c1 = 2 * l, c2 = 2 * l + 1;
    FV_TRY(conv(u, c1, plain_in(X, c1)));
    FV_TRY(conv(u, c2, plain_in(u->act[c1], c2)));
    if (l < 3) {
      const Dims d{u->n[l][0], u->n[l][1], u->n[l][2]};
      UNET_LAUNCH((k_pool<<<blocks_for(u->ncell[l + 1] * kConvs[c2].cout / 8), 256, 0, st>>>(
          u->act[c2], u->pool[l], kConvs[c2].cout, d)));
      X = u->pool[l];
    }
  }
  for (int q = 0; q < 3; ++q) {
    const int c1 = 8 + 2 * q, c2 = 9 + 2 * q;
    FV_TRY(conv(u, c1, decoder_in(u, q)));
    FV_TRY(conv(u, c2, plain_in(u->act[c1], c2)));
  }
  UNET_LAUNCH((k_head<<<blocks_for(u->ncell[0]), 256, 0, st>>>(u->act[13], u->p + u->head_w,
                                                                 u->p + u->head_b, u->out,
                                                                 (int)u->ncell[0])));
  u->have_fwd = true;
  return FV_OK;
}

// parameter gradients of layer c from its pre-activation gradient gy and its
// input.  About two blocks per SM over (tiles x channel pairs): fewer blocks
// leave SMs idle, more only add atomics (27 x 16 x 16 NCI per block).
static fv_status param_grad(fv_unet* u, int c, const bf16* gy, const ConvIn& in) {
  const ConvSpec& s = kConvs[c];
  const int* n = u->n[s.level];
  const Dims d{n[0], n[1], n[2]};
  const int nci = s.cin % 48 == 0 ? 3 : s.cin % 32 == 0 ? 2 : 1;
  const int items = (s.cout / 16) * (s.cin / (16 * nci)), nt = tiles(n);
  const dim3 grid(std::max(1, std::min(nt, 2 * 152 / items)), items);
  float *dw = u->g + u->woff[c], *db = u->g + u->boff[c];
  if (nci == 3) UNET_LAUNCH((k_wgrad<3><<<grid, 288, 0, u->stream>>>(gy, s.cout, in, s.cin, dw, db, d, nt)));
  else if (nci == 2) UNET_LAUNCH((k_wgrad<2><<<grid, 288, 0, u->stream>>>(gy, s.cout, in, s.cin, dw, db, d, nt)));
  else UNET_LAUNCH((k_wgrad<1><<<grid, 288, 0, u->stream>>>(gy, s.cout, in, s.cin, dw, db, d, nt)));
  return FV_OK;
}

// input gradient of layer c from gy (cin channels), zero where mask <= 0
static fv_status data_grad(fv_unet* u, int c, const bf16* gy, bf16* dX, const bf16* mask) {
  const ConvSpec& s = kConvs[c];
  return conv_any<true>(u->stream, {gy, s.cout, nullptr, 0}, s.cout, u->pb + u->woff[c], nullptr, dX, s.cin,
                        mask, u->n[s.level]);
}

// loss of the last forward pass against u->tgt and all parameter gradients
static fv_status backward(fv_unet* u, double* loss) {
  if (!u->have_fwd) { set_error("unet: backward needs a forward pass at the same dims"); return FV_EINVAL; }
  FV_TRY(ensure_grad(u));
  cudaStream_t st = u->stream;
  const int n0 = (int)u->ncell[0];
  FV_CUDA(cudaMemsetAsync(u->g, 0, u->nparam * sizeof(float), st));
  FV_CUDA(cudaMemsetAsync(u->red, 0, 2 * sizeof(double), st));
  UNET_LAUNCH((k_err_sum<<<blocks_for(n0), 256, 0, st>>>(u->out, u->tgt, n0, u->red)));
  UNET_LAUNCH((k_head_back<<<blocks_for(n0), 256, 0, st>>>(u->act[13], u->p + u->head_w, u->out, u->tgt,
                                                           n0, u->red, u->gA, u->g + u->head_w,
                                                           u->g + u->head_b)));
  // g: the pre-activation gradient of the current layer's output (the ReLU
  // masks are applied by the kernels that write it)
  bf16* g = u->gA;
  bf16* h = u->gB;
  for (int q = 2; q >= 0; --q) {
    const int l = 2 - q, c1 = 8 + 2 * q, c2 = 9 + 2 * q;
    const ConvIn in = decoder_in(u, q);
    FV_TRY(param_grad(u, c2, g, plain_in(u->act[c1], c2)));
    FV_TRY(data_grad(u, c2, g, h, u->act[c1]));
    std::swap(g, h);
    FV_TRY(param_grad(u, c1, g, in));
    FV_TRY(data_grad(u, c1, g, u->gC, nullptr));
    const Dims d{u->n[l][0], u->n[l][1], u->n[l][2]};
    UNET_LAUNCH((k_up_cat_back<<<blocks_for((u->ncell[l + 1] * in.lowc + u->ncell[l] * in.xc) / 8), 256, 0, st>>>(
        u->gC, in.lowc, in.xc, in.low, g, u->gS[l], d)));
  }
  for (int l = 3; l >= 0; --l) {
    const int c1 = 2 * l, c2 = 2 * l + 1;
    if (l < 3) {
      // act[c2] feeds the pooling (gradient g, coarse) and the skip (gS[l])
      const Dims d{u->n[l][0], u->n[l][1], u->n[l][2]};
      const int ch = kConvs[c2].cout;
      UNET_LAUNCH((k_pool_back<<<blocks_for(u->ncell[l] * ch / 8), 256, 0, st>>>(g, u->gS[l], u->act[c2], h,
                                                                                ch, d)));
      std::swap(g, h);
    }
    const bf16* X = l == 0 ? u->in16 : u->pool[l - 1];
    FV_TRY(param_grad(u, c2, g, plain_in(u->act[c1], c2)));
    FV_TRY(data_grad(u, c2, g, h, u->act[c1]));
    std::swap(g, h);
    FV_TRY(param_grad(u, c1, g, plain_in(X, c1)));
    if (l > 0) {
      FV_TRY(data_grad(u, c1, g, h, nullptr));
      std::swap(g, h);
    }
  }
  if (loss) {
    double hr[2];
    FV_CUDA(cudaMemcpyAsync(hr, u->red, sizeof(hr), cudaMemcpyDeviceToHost, st));
    FV_CUDA(cudaStreamSynchronize(st));
    *loss = hr[1];
  }
  return FV_OK;
}

static fv_status adam(fv_unet* u, float lr) {
  u->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)u->step), c2 = 1.f - std::pow(b2, (float)u->step);
  UNET_LAUNCH((k_adam<<<blocks_for(u->nparam), 256, 0, u->stream>>>(u->p, u->g, u->m, u->v, u->pb,
                                                                     u->nparam, lr, b1, b2, c1, c2)));
  return FV_OK;
}

// normalised input of the float32 right-hand side r on grid g into u->in16
// (and its scale S into u->scale)
static fv_status pack_rhs(fv_unet* u, const fv_grid* g, const float* r) {
  cudaStream_t st = u->stream;
  const float* const* idx = g->met_f.idx;
  FV_CUDA(cudaMemsetAsync(u->red + 2, 0, sizeof(double), st));
  UNET_LAUNCH((k_rhs_sumsq<<<blocks_for(g->ncell), 256, 0, st>>>(r, g->n[0], g->n[1], g->n[2], idx[0],
                                                                 idx[1], idx[2], u->red)));
  UNET_LAUNCH((k_pack_rhs<<<blocks_for(g->ncell), 256, 0, st>>>(r, u->red, g->n[0], g->n[1], g->n[2],
                                                                idx[0], idx[1], idx[2], u->in16,
                                                                u->scale)));
  return FV_OK;
}

static fv_status guess_body(fv_unet* u, const fv_grid* g, const float* r, float* phi) {
  FV_TRY(ensure_ws(u, g->n[0], g->n[1], g->n[2]));
  FV_TRY(pack_rhs(u, g, r));
  FV_TRY(forward(u));
  UNET_LAUNCH((k_unscale<<<blocks_for(g->ncell), 256, 0, u->stream>>>(u->out, u->scale, phi,
                                                                      (int)g->ncell)));
  return FV_OK;
}

static fv_status train_body(fv_unet* u, const fv_grid* g, const double* r, const double* phi,
                            float lr, double* loss) {
  FV_TRY(ensure_ws(u, g->n[0], g->n[1], g->n[2]));
  cudaStream_t st = u->stream;
  UNET_LAUNCH((k_to_f32<<<blocks_for(g->ncell), 256, 0, st>>>(r, u->out, g->ncell)));
  FV_TRY(pack_rhs(u, g, u->out));
  UNET_LAUNCH((k_scale_target<<<blocks_for(g->ncell), 256, 0, st>>>(phi, u->scale, u->tgt,
                                                                      (int)g->ncell)));
  FV_TRY(forward(u));
  FV_TRY(backward(u, loss));
  return adam(u, lr);
}

}  // namespace unet

// Guess of phi (float32, device) for the float32 right-hand side r on grid g,
// on the grid's stream (the learned first pass of the SIMPLE loop).  r and
// phi may alias: r is read in full before phi is written.
fv_status unet_guess_f32(fv_unet* u, const fv_grid* g, const float* r, float* phi) {
  cudaStream_t keep = u->stream;
  u->stream = g->stream;
  fv_status s = unet::guess_body(u, g, r, phi);
  u->stream = keep;
  return s;
}

fv_status absmax_f32_host(const fv_grid* g, const float* x, int64_t n, double* out) {
  // one unsigned slot at the end of the grid's scalar area
  unsigned* slot = reinterpret_cast<unsigned*>(g->d_scal + kScalars - 1);
  FV_CUDA(cudaMemsetAsync(slot, 0, sizeof(unsigned), g->stream));
  count_launch();
  unet::k_absmax<<<unet::blocks_for(n), 256, 0, g->stream>>>(x, n, slot);
  FV_CHECK_LAUNCH();
  unsigned bits = 0;
  FV_CUDA(cudaMemcpyAsync(&bits, slot, sizeof(unsigned), cudaMemcpyDeviceToHost, g->stream));
  FV_CUDA(cudaStreamSynchronize(g->stream));
  float f;
  std::memcpy(&f, &bits, sizeof(f));
  *out = f;
  return FV_OK;
}

}  // namespace fv

using namespace fv::unet;
using fv::set_error;
using fv::cuda_fail;

extern "C" {

void fv_unet_destroy(fv_unet* u) {
  if (!u) return;
  free_ws(u);
  free_grad(u);
  dfree(u->p); dfree(u->g); dfree(u->m); dfree(u->v); dfree(u->pb);
  dfree(u->red); dfree(u->scale);
  delete u;
}

fv_status fv_unet_create(uint64_t seed, void* cuda_stream, fv_unet** out) {
  if (!out) { set_error("fv_unet_create: out is NULL"); return FV_EINVAL; }
  *out = nullptr;
  fv_unet* u = new fv_unet();
  u->stream = (cudaStream_t)cuda_stream;
  if (set_conv_attributes() != FV_OK) { delete u; return FV_ECUDA; }
  int off = 0;
  for (int c = 0; c < kNConv; ++c) {
    u->woff[c] = off;
    off += 27 * kConvs[c].cin * kConvs[c].cout;
    u->boff[c] = off;
    off += kConvs[c].cout;
  }
  u->head_w = off;
  off += 16;
  u->head_b = off;
  off += 1;
  u->nparam = off;
  fv_status s = FV_OK;
  auto A = [&](void** p, size_t b) { if (s == FV_OK) s = dalloc(p, b); };
  A((void**)&u->p, off * sizeof(float));
  A((void**)&u->g, off * sizeof(float));
  A((void**)&u->m, off * sizeof(float));
  A((void**)&u->v, off * sizeof(float));
  A((void**)&u->pb, off * sizeof(bf16));
  A((void**)&u->red, 4 * sizeof(double));
  A((void**)&u->scale, sizeof(float));
  if (s != FV_OK) { fv_unet_destroy(u); return s; }
  // He-normal weights (seeded), zero biases
  std::vector<float> h(off, 0.f);
  std::mt19937_64 rng(seed);
  std::normal_distribution<float> nd(0.f, 1.f);
  for (int c = 0; c < kNConv; ++c) {
    const float sd = std::sqrt(2.f / (27.f * kConvs[c].cin));
    for (int e = 0; e < 27 * kConvs[c].cin * kConvs[c].cout; ++e) h[u->woff[c] + e] = sd * nd(rng);
  }
  for (int k = 0; k < 16; ++k) h[u->head_w + k] = 0.25f * nd(rng);
  cudaError_t e = cudaMemcpy(u->p, h.data(), off * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(u->g, 0, off * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(u->m, 0, off * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(u->v, 0, off * sizeof(float));
  if (e == cudaSuccess) {
    fv::count_launch();
    k_mirror<<<blocks_for(off), 256, 0, u->stream>>>(u->p, u->pb, off);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(u->stream);
  if (e != cudaSuccess) {
    fv_status r = cuda_fail(e, "fv_unet_create", __FILE__, __LINE__);
    fv_unet_destroy(u);
    return r;
  }
  *out = u;
  return FV_OK;
}

int fv_unet_param_count(const fv_unet* u) { return u ? u->nparam : 0; }

fv_status fv_unet_set_stream(fv_unet* u, void* cuda_stream) {
  if (!u) { set_error("fv_unet_set_stream: NULL network"); return FV_EINVAL; }
  u->stream = (cudaStream_t)cuda_stream;
  return FV_OK;
}

fv_status fv_unet_set_params(fv_unet* u, const float* params) {
  if (!u || !params) { set_error("fv_unet_set_params: NULL argument"); return FV_EINVAL; }
  FV_CUDA(cudaMemcpyAsync(u->p, params, u->nparam * sizeof(float), cudaMemcpyDeviceToDevice, u->stream));
  UNET_LAUNCH((k_mirror<<<blocks_for(u->nparam), 256, 0, u->stream>>>(u->p, u->pb, u->nparam)));
  FV_CUDA(cudaMemsetAsync(u->m, 0, u->nparam * sizeof(float), u->stream));
  FV_CUDA(cudaMemsetAsync(u->v, 0, u->nparam * sizeof(float), u->stream));
  u->step = 0;
  return FV_OK;
}

fv_status fv_unet_get_params(const fv_unet* u, float* params, float* grads) {
  if (!u) { set_error("fv_unet_get_params: NULL network"); return FV_EINVAL; }
  if (params)
    FV_CUDA(cudaMemcpyAsync(params, u->p, u->nparam * sizeof(float), cudaMemcpyDeviceToDevice, u->stream));
  if (grads)
    FV_CUDA(cudaMemcpyAsync(grads, u->g, u->nparam * sizeof(float), cudaMemcpyDeviceToDevice, u->stream));
  return FV_OK;
}

fv_status fv_unet_forward(fv_unet* u, int nx, int ny, int nz, const float* in, float* out) {
  if (!u || !in || !out) { set_error("fv_unet_forward: NULL argument"); return FV_EINVAL; }
  FV_TRY(ensure_ws(u, nx, ny, nz));
  UNET_LAUNCH((k_pack_planes<<<blocks_for(u->ncell[0]), 256, 0, u->stream>>>(in, u->in16, (int)u->ncell[0])));
  FV_TRY(forward(u));
  FV_CUDA(cudaMemcpyAsync(out, u->out, u->ncell[0] * sizeof(float), cudaMemcpyDeviceToDevice, u->stream));
  return FV_OK;
}

fv_status fv_unet_backward(fv_unet* u, const float* target, double* loss) {
  if (!u || !target) { set_error("fv_unet_backward: NULL argument"); return FV_EINVAL; }
  if (!u->have_fwd) { set_error("fv_unet_backward: no forward pass to differentiate"); return FV_EINVAL; }
  FV_CUDA(cudaMemcpyAsync(u->tgt, target, u->ncell[0] * sizeof(float), cudaMemcpyDeviceToDevice, u->stream));
  return backward(u, loss);
}

fv_status fv_unet_adam(fv_unet* u, float lr) {
  if (!u || !(lr > 0.f)) { set_error("fv_unet_adam: NULL network or lr <= 0"); return FV_EINVAL; }
  return adam(u, lr);
}

fv_status fv_unet_guess(fv_unet* u, const fv_grid* g, const double* r, double* phi) {
  if (!u || !g || !r || !phi) { set_error("fv_unet_guess: NULL argument"); return FV_EINVAL; }
  cudaStream_t keep = u->stream;
  u->stream = g->stream;
  auto body = [&]() -> fv_status {
    FV_TRY(ensure_ws(u, g->n[0], g->n[1], g->n[2]));
    // float32 copy of r and the guess share the target buffer
    UNET_LAUNCH((k_to_f32<<<blocks_for(g->ncell), 256, 0, u->stream>>>(r, u->tgt, g->ncell)));
    FV_TRY(guess_body(u, g, u->tgt, u->tgt));
    return fv::launch_widen_f32(g, u->tgt, phi, g->ncell);
  };
  fv_status s = body();
  u->stream = keep;
  return s;
}

fv_status fv_unet_train_step(fv_unet* u, const fv_grid* g, const double* r, const double* phi,
                             float lr, double* loss) {
  if (!u || !g || !r || !phi || !(lr > 0.f)) {
    set_error("fv_unet_train_step: NULL argument or lr <= 0");
    return FV_EINVAL;
  }
  cudaStream_t keep = u->stream;
  u->stream = g->stream;
  fv_status s = train_body(u, g, r, phi, lr, loss);
  u->stream = keep;
  return s;
}

}  // extern "C"
