// Float64 tensor-product transforms on the tensor cores.
//
// GB300 multiplies float64 at about 1 TFLOP/s, so the six dense transforms of
// a float64 pressure solve (2 n^4 flop each on n^3 cells) are by far the
// longest part of the float64 form.  Here each transform
//   out[v][p] = sum_k M[p][k] in[v][k]
// is computed exactly enough in integers that the BF16 tensor cores multiply
// without rounding (the splitting of Ozaki, Ogita, Oishi & Rump 2012, Numer.
// Algorithms 59): every row of M and every K-vector of the field is scaled by
// a power of two and rounded to a 60-bit integer X, which is written as eight
// signed base-256 digits d_0 .. d_7 (|d| <= 128, |d_0| <= 16: exact in BF16).
// The product of two such numbers is the sum over pairs of digits (i, j) of
// d_i d_j 256^(14 - i - j); the pairs with i + j <= 8 are kept, the others are
// below 2^-60 of the product of the two maxima.  A pair's sum over k is one
// BF16 tensor-core product accumulated in float32, an integer below 2^24 for
// K <= 128 in every group i + j = s <= 5 (at most (2 16 128 + 4 128^2) 128 =
// 8.9e6), so these sums are exact, as is the joint sum of the groups 0 and 1
// (256 16^2 128 + 2 16 128 128 < 2^24); the groups 6 .. 8 share an accumulator
// that rounds at about 2^-62 of the product of the maxima.  The sums are
// joined in 96-bit integers and rounded once to float64.  The maxima matter:
// on the strongly stretched axes the terms that make up a result can be 60
// times smaller than the largest entries of row and vector, so a version that
// cut at 2^-54 of their product (36 products, groups 5 .. 7 joined) was up to
// four times less accurate than float64 sums; this one is no less accurate
// (tests/test_gpu_oz.py against extended precision).  What a vector holds more than
// 2^-60 below its largest entry is lost, where float64 keeps every entry relative
// to itself; in a solve this shows nowhere: right-hand sides of single cells, wall
// layers and entries over 18 orders of magnitude came out 3 to 7 times more accurate
// than with the float64 kernels, in the largest error, the mean square and
// component by component (median and 99 %).
//
// One block: N K-vectors of the field, all n <= 128 rows of M.  The field is
// split once into its digits (N x K x 8 BF16, the B operands, resident); the
// digits of M stream through a two-stage ring of 16-column chunks (bulk
// copies), 43 products of 128 x N x 16 per chunk.  Six accumulators of N
// columns in tensor memory: N = 80 (64 for K > 112, whose digits would not
// fit), one block per SM.  Sixteen warps split the field and later join the
// sums, a seventeenth issues the products chunk by chunk as their digits
// become ready.  Measured at 100^3: 27 us a transform (125 blocks; the tensor
// pipe is busy for about a quarter of that, the rest is splitting, joining and
// latency) against 342 us for the float64 kernels, 44 us with eight warps that
// did all of it in turn; a float64 evaluation of 8^3 .. 128^3 cells takes 245 ..
// 1512 us against 337 .. 7149 us, so the kernel serves every axis it covers.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fv_internal.cuh"
#include "fv_tc5.cuh"

namespace fv {

namespace {

typedef uint16_t bf16b;                // BF16 bit pattern

constexpr int kDig = 8;                // digits per number
constexpr int kAcc = 6;                // accumulators: groups {0, 1}, 2, 3, 4, 5, {6, 7, 8}
constexpr int kOzMax = 128;            // rows of M (= n) at most
constexpr int kWorkers = 16;           // warps that split the field and read the sums
constexpr int kOzThreads = 32 * kWorkers + 32;   // and one that issues the products
constexpr int kChunkBytes = kDig * 128 * 16 * 2;   // one 16-column chunk of M's digits
constexpr int kOzLimit = 1 << 22;      // polls of an mbarrier before the block gives up

__host__ __device__ inline int up16(int n) { return (n + 15) & ~15; }
__host__ __device__ inline int tile_n(int n) { return up16(n) > 112 ? 64 : 80; }
inline size_t oz_smem(int n) {
  return 2 * (size_t)kChunkBytes + (size_t)kDig * tile_n(n) * up16(n) * 2;
}

// digits 256^(7 - i) of X (|X| < 2^60) as bytes, each plus 128
__host__ __device__ inline uint64_t digit_bytes(int64_t X) {
  return ((uint64_t)X + 0x0080808080808080ull) ^ 0x8000000000000000ull;
}

// x 2^(60 - e) rounded to an integer, 2^e the power of two above the largest
// value of the vector (b = its biased exponent, >= 1)
__host__ __device__ inline int64_t to_fixed(uint64_t bits, int b) {
  const int ex = (int)((bits >> 52) & 0x7ff);
  uint64_t m = bits & 0xfffffffffffffull;
  if (ex) m |= 1ull << 52;
  const int sh = (ex ? ex : 1) - b + 7;
  uint64_t u = 0;
  if (sh >= 0) u = m << sh;
  else if (sh > -60) u = (m + (1ull << (-sh - 1))) >> -sh;
  return (bits >> 63) ? -(int64_t)u : (int64_t)u;
}

// float bits of digit i times 2^(-8 i) (exact in eight bits, so BF16 is their
// upper half): the float 2^(23 - 8 i) + byte 2^(-8 i), less what the bytes are
// biased by
template <int I>
__device__ __forceinline__ uint32_t digit_float(uint64_t bytes) {
  constexpr uint32_t magic = (uint32_t)(150 - 8 * I) << 23;
  const uint32_t word = I < 4 ? (uint32_t)(bytes >> 32) : (uint32_t)bytes;
  const float f = __uint_as_float(__byte_perm(word, magic, 0x7650 | (3 - I % 4)));
  return __float_as_uint(f - __uint_as_float(magic | 0x80u));
}

// 16-byte runs (8 entries of one vector) of the digits I .. 7
template <int I>
__device__ __forceinline__ void put_digits(unsigned char* dst, int slice, const uint64_t (&d)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    w[q] = __byte_perm(digit_float<I>(d[2 * q]), digit_float<I>(d[2 * q + 1]), 0x7632);
  *reinterpret_cast<uint4*>(dst + I * slice) = make_uint4(w[0], w[1], w[2], w[3]);
  if constexpr (I + 1 < kDig) put_digits<I + 1>(dst, slice, d);
}

// accumulator of the pairs with i + j = s
__host__ __device__ constexpr int acc_of(int s) { return s < 2 ? 0 : s < 6 ? s - 1 : kAcc - 1; }

// s1 2^32 + s0 (|s1| < 2^41, |s0| < 2^50), times 2^sc, rounded to float64
__device__ __forceinline__ double join96(int64_t s1, int64_t s0, int sc) {
  int64_t hi = s1 + (s0 >> 32);
  uint32_t lo = (uint32_t)s0;
  const bool neg = hi < 0;
  if (neg) {
    lo = 0u - lo;
    hi = ~hi + (lo == 0u ? 1 : 0);
  }
  uint64_t m;
  int z;
  if (hi != 0) {                   // hi < 2^42: z >= 22
    z = __clzll(hi);
    m = ((uint64_t)hi << z) | (((uint64_t)lo << 32) >> (64 - z));
  } else {
    if (lo == 0u) return 0.0;
    z = __clz((int)lo);
    m = (uint64_t)lo << (32 + z);
    z += 64;
  }
  const uint64_t mant = (m >> 11) + ((m >> 10) & 1);    // 2^52 .. 2^53
  const int ef = 1023 + 95 - z + sc;                    // biased exponent
  if (ef >= 1 && ef <= 2045) {
    const uint64_t bits = ((uint64_t)(ef - 1) << 52) + mant;
    return __longlong_as_double((long long)(neg ? bits | (1ull << 63) : bits));
  }
  const double o = scalbn((double)mant, 43 - z + sc);   // overflow or subnormal
  return neg ? -o : o;
}

struct OzArgs {
  const double* in;
  double* out;
  const bf16b* mat;        // [K / 16][digit][128 x 16 canonical]
  const int* rexp;         // biased exponent of each row's largest entry
  OzScale sc;              // SCALE: factors of the results
  int n;                   // rows of M = entries of a vector
  int64_t nvec, Q;         // vectors; entry k of vector v is at (v / Q) n Q + k Q + v % Q
  unsigned* fault;
};

// SCALE: 0 none, 1 a factor per cell, 2 one per entry and index along another axis
template <bool RIGHT, int SCALE>
__global__ void __launch_bounds__(kOzThreads) k_oz(OzArgs A) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t full[2], empty[2], ready[kOzMax / 16], done;
  __shared__ uint32_t tslot;
  __shared__ int bad;
  __shared__ int vexp[80];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = A.n, K = up16(n), N = tile_n(n), nk = K >> 4;
  const int64_t v0 = (int64_t)blockIdx.x * N;
  unsigned char* ring = sm;
  unsigned char* B = sm + 2 * kChunkBytes;      // [digit][N x K canonical]
  const int slice = N * K * 2;
  // The field in tasks of one warp: NV vectors x NR runs of 8 entries.  LEFT:
  // 16 vectors (consecutive in memory) x 2 runs, one 16-column chunk; RIGHT
  // (the entries of a vector are consecutive): 8 vectors x 4 runs, so that a
  // run is two sectors and the eight lanes of a 16-byte store phase hit the
  // eight rows of a core matrix.  Chunks in order, so that the products of the
  // first ones overlap the splitting of the others.
  constexpr int NV = RIGHT ? 8 : 16, NR = 32 / NV, NT = 3;
  const int runs = K >> 3, nvb = N / NV;
  const int ntask = nvb * ((runs + NR - 1) / NR);   // <= 40
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      tc5::mbar_init(&full[s], 1);
      tc5::mbar_init(&empty[s], 1);
    }
    for (int c = 0; c < nk; ++c) tc5::mbar_init(&ready[c], nvb);   // one arrival per task of the chunk
    tc5::mbar_init(&done, 1);
    bad = 0;
    tc5::fence_proxy_async();
    const int first = nk < 2 ? nk : 2;
    for (int c = 0; c < first; ++c)
      tc5::bulk_load(ring + c * kChunkBytes, (const unsigned char*)A.mat + (size_t)c * kChunkBytes,
                     kChunkBytes, &full[c]);
  }
  if (tid < 80) vexp[tid] = 1;
  // everything above uses constants only; the field is the predecessor's output
  tc5::pdl_wait();
  // The block takes all of the SM's tensor memory: only after the wait, and the
  // successor is let in only once every block has it, so that no block waits
  // for columns held by a kernel that waits for this one.
  if (warp == 0) tc5::tmem_alloc(&tslot, 512);
  __syncthreads();
  tc5::pdl_trigger();
  double x[NT][8];
  if (warp < kWorkers) {
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      const int t = warp + kWorkers * i;
      const int vl = (t % nvb) * NV + lane % NV, r = (t / nvb) * NR + lane / NV;
      const int64_t v = v0 + vl;
      const bool ok = t < ntask && r < runs && v < A.nvec;
      int64_t base = 0;
      if (ok) base = RIGHT ? v * n : (v / A.Q) * n * A.Q + v % A.Q;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int k = 8 * r + q;
        x[i][q] = (ok && k < n) ? __ldg(A.in + base + (RIGHT ? (int64_t)k : k * A.Q)) : 0.0;
      }
    }
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      const int t = warp + kWorkers * i;
      const int vl = (t % nvb) * NV + lane % NV;
      int b = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) b = max(b, (__double2hiint(x[i][q]) & 0x7fffffff) >> 20);
      if (b > 1) atomicMax(&vexp[vl], b);
    }
  }
  tc5::fence_before_sync();
  __syncthreads();
  tc5::fence_after_sync();
  const uint32_t tmem = tslot;
  if (warp < kWorkers) {
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      const int t = warp + kWorkers * i;
      const int vl = (t % nvb) * NV + lane % NV, r = (t / nvb) * NR + lane / NV;
      if (t >= ntask) break;
      if (r < runs) {
        const int b = vexp[vl];
        uint64_t d[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) d[q] = digit_bytes(to_fixed((uint64_t)__double_as_longlong(x[i][q]), b));
        put_digits<0>(B + tc5::canon_offset16(vl, 8 * r, K), slice, d);
      }
      tc5::fence_proxy_async();
      __syncwarp();
      // this task's chunks: lane 0 (and, RIGHT, lane 16 for the second one)
      if (lane == 0 || (RIGHT && lane == 16 && r < runs)) tc5::mbar_arrive(&ready[r >> 1]);
    }
  } else if (lane == 0) {
    bool ok = true;
    const uint32_t idesc = tc5::idesc_bf16(128, N);
    const uint32_t ra = tc5::smem_u32(ring), rb = tc5::smem_u32(B), sbo = (uint32_t)(K / 8) * 128;
    for (int c = 0; c < nk; ++c) {
      const int st = c & 1;
      ok = tc5::mbar_wait(&full[st], (uint32_t)(c >> 1) & 1u, kOzLimit) && ok;
      ok = tc5::mbar_wait(&ready[c], 0, kOzLimit) && ok;
      tc5::fence_after_sync();
#pragma unroll
      for (int i = 0; i < kDig; ++i)
#pragma unroll
        for (int j = 0; j < kDig; ++j) {
          if (i + j > kDig) continue;
          const int g = acc_of(i + j);
          const bool first = c == 0 && i == 0 && (j == 0 || g != acc_of(j - 1));
          tc5::mma_f16(tmem + (uint32_t)(g * N),
                       tc5::sdesc(ra + st * kChunkBytes + i * (128 * 32), 128, 256),
                       tc5::sdesc(rb + j * slice + c * 256, 128, sbo), idesc, first ? 0u : 1u);
        }
      tc5::commit(&empty[st]);
      // while these products run: the other stage's are done, refill it
      if (c >= 1 && c + 1 < nk) {
        ok = tc5::mbar_wait(&empty[st ^ 1], (uint32_t)((c - 1) >> 1) & 1u, kOzLimit) && ok;
        tc5::bulk_load(ring + (st ^ 1) * kChunkBytes,
                       (const unsigned char*)A.mat + (size_t)(c + 1) * kChunkBytes, kChunkBytes,
                       &full[st ^ 1]);
      }
    }
    tc5::commit(&done);
    ok = tc5::mbar_wait(&done, 0, kOzLimit) && ok;
    if (!ok) {
      bad = 1;
      atomicOr(A.fault, 1u);   // reported as FV_ETIMEOUT
    }
  }
  __syncthreads();
  tc5::fence_after_sync();
  if (warp < kWorkers) {
    const bool failed = bad != 0;
    const int p = 32 * (warp & 3) + lane;
    const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    const int per = N / 4, c_begin = (warp >> 2) * per;    // 20 or 16 columns per warp
    const int ea = p < n ? __ldg(A.rexp + p) : 1;
    for (int c = c_begin; c < c_begin + per; c += 4) {
      uint32_t a[kAcc][4];
      __syncwarp();   // tcgen05.ld is warp-collective
#pragma unroll
      for (int g = 0; g < kAcc; ++g) tc5::ld4_nowait(trow + (uint32_t)(g * N + c), a[g]);
      tc5::ld_wait();
      const int64_t v = v0 + c;
      if (p < n && v < A.nvec) {
        double o[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          // group sums: integers times 2^(-8 s), but for the last
          const int g01 = __float2int_rn(__uint_as_float(a[0][q]) * 0x1p8f);
          const int g2 = __float2int_rn(__uint_as_float(a[1][q]) * 0x1p16f);
          const int g3 = __float2int_rn(__uint_as_float(a[2][q]) * 0x1p24f);
          const int g4 = __float2int_rn(__uint_as_float(a[3][q]) * 0x1p32f);
          const int g5 = __float2int_rn(__uint_as_float(a[4][q]) * 0x1p40f);
          const float t = __uint_as_float(a[5][q]) * 0x1p48f;
          const int ti = __float2int_rn(t);
          const int tf = __float2int_rn((t - (float)ti) * 256.f);
          const int64_t s1 = ((int64_t)g01 << 16) + ((int64_t)g2 << 8) + g3;
          const int64_t s0 = ((int64_t)g4 << 24) + ((int64_t)g5 << 16) + ((int64_t)ti << 8) + tf;
          const int eb = vexp[c + q];
          // unit 2^56 of X_a X_b = a b 2^(120 - e_a - e_b), e = biased exponent - 1022
          o[q] = join96(s1, s0, ea + eb - 2108);
          if (eb == 2047 || failed) o[q] = __longlong_as_double(0x7ff8000000000000ll);
        }
        if (SCALE == 2) {
          const unsigned t = (unsigned)v / (unsigned)A.sc.da;   // index along the other axis: t % na
          int r = (int)((unsigned)v - t * A.sc.da), i = (int)(t % (unsigned)A.sc.na);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            o[q] *= __ldg(A.sc.inv + i * n + p);
            if (++r == A.sc.da) {
              r = 0;
              if (++i == A.sc.na) i = 0;
            }
          }
        }
        const int64_t e = RIGHT ? v * n + p : (v / A.Q) * n * A.Q + (int64_t)p * A.Q + v % A.Q;
        if (!RIGHT && (A.Q & 3) == 0) {      // four vectors of one row: two 16-byte stores
          if (SCALE == 1) {
            const double2 i0 = __ldg(reinterpret_cast<const double2*>(A.sc.inv + e));
            const double2 i1 = __ldg(reinterpret_cast<const double2*>(A.sc.inv + e) + 1);
            o[0] *= i0.x; o[1] *= i0.y; o[2] *= i1.x; o[3] *= i1.y;
          }
          *reinterpret_cast<double2*>(A.out + e) = make_double2(o[0], o[1]);
          *(reinterpret_cast<double2*>(A.out + e) + 1) = make_double2(o[2], o[3]);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int64_t w = v + q;
            if (w < A.nvec) {
              const int64_t f = RIGHT ? w * n + p : (w / A.Q) * n * A.Q + (int64_t)p * A.Q + w % A.Q;
              A.out[f] = SCALE == 1 ? o[q] * __ldg(A.sc.inv + f) : o[q];
            }
          }
        }
      }
    }
  }
  tc5::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc5::tmem_dealloc(tmem, 512);
}

// digits of the n x n row-major matrix M in the order the kernel streams them
// (out starts as zeros)
void lay_out(const std::vector<double>& M, int n, bf16b* out, int* rexp) {
  struct Table {                         // BF16 bits of (byte - 128) 2^(-8 i)
    bf16b v[kDig][256];
    Table() {
      for (int i = 0; i < kDig; ++i)
        for (int b = 0; b < 256; ++b) {
          const float f = std::ldexp((float)(b - 128), -8 * i);
          uint32_t u;
          std::memcpy(&u, &f, 4);
          v[i][b] = (bf16b)(u >> 16);
        }
    }
  };
  static const Table tab;
  for (int p = 0; p < n; ++p) {
    const double* row = &M[(size_t)p * n];
    int b = 1;
    for (int k = 0; k < n; ++k) {
      uint64_t u;
      std::memcpy(&u, row + k, 8);
      b = std::max(b, (int)((u >> 52) & 0x7ff));
    }
    rexp[p] = b;
    for (int k0 = 0; k0 < n; k0 += 8) {  // one 16-byte run per digit
      bf16b* dst = out + ((size_t)(k0 >> 4) * kChunkBytes + tc5::canon_offset16(p, k0 & 15, 16)) / 2;
      for (int q = 0; q < 8 && k0 + q < n; ++q) {
        uint64_t u;
        std::memcpy(&u, row + k0 + q, 8);
        const uint64_t bytes = digit_bytes(to_fixed(u, b));
        for (int i = 0; i < kDig; ++i) dst[i * 128 * 16 + q] = tab.v[i][(bytes >> (56 - 8 * i)) & 0xff];
      }
    }
  }
}

__global__ void k_inv_lam(TpfDev<double> tp, double* __restrict__ inv, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % tp.n[0]), j = (int)(e / tp.n[0] % tp.n[1]), k = (int)(e / ((int64_t)tp.n[0] * tp.n[1]));
    const bool null = i == tp.null_index[0] && j == tp.null_index[1] && k == tp.null_index[2];
    inv[e] = null ? 0.0 : 1.0 / (tp.lam[2][k] + tp.lam[1][j] + tp.lam[0][i]);
  }
}

}  // namespace

bool oz_ok(const fv_grid* g, int axis) { return g->oz.mat[axis][0] != nullptr; }

fv_status build_oz(fv_grid* g) {
  // operands of the axes the kernel covers; the float64 kernels serve the others
  size_t bytes = 0;
  int same[3];                           // the first axis with the same cells
  for (int d = 0; d < 3; ++d) {
    same[d] = d;
    for (int e = d - 1; e >= 0; --e)
      if (g->n[e] == g->n[d]) same[d] = e;
    if (g->n[d] <= kOzMax && same[d] == d) bytes += 2 * ((size_t)(up16(g->n[d]) / 16) * kChunkBytes + 512);
  }
  if (!bytes) return FV_OK;
  std::vector<unsigned char> h(bytes);
  size_t off[3][2], o = 0;
  for (int d = 0; d < 3; ++d) {
    if (g->n[d] > kOzMax) continue;
    const size_t one = (size_t)(up16(g->n[d]) / 16) * kChunkBytes + 512;
    for (int q = 0; q < 2; ++q) {
      if (same[d] != d) { off[d][q] = off[same[d]][q]; continue; }
      off[d][q] = o;
      lay_out(q == 0 ? g->basis[d].Einv : g->basis[d].E, g->n[d], (bf16b*)(h.data() + o),
              (int*)(h.data() + o + one - 512));
      o += one;
    }
  }
  const bool all = g->n[0] <= kOzMax && g->n[1] <= kOzMax && g->n[2] <= kOzMax;
  const size_t need = bytes + (all ? (size_t)g->ncell * sizeof(double) : 0);
  if (cudaMalloc(&g->d_oz, need) != cudaSuccess) {
    (void)cudaGetLastError();
    g->d_oz = nullptr;
    set_error("cudaMalloc of the float64 tensor-core operands failed");
    return FV_ENOMEM;
  }
  g->ws_bytes += (int64_t)need;
  FV_CUDA(cudaMemcpy(g->d_oz, h.data(), bytes, cudaMemcpyHostToDevice));
  for (int d = 0; d < 3; ++d) {
    if (g->n[d] > kOzMax) continue;
    const size_t one = (size_t)(up16(g->n[d]) / 16) * kChunkBytes + 512;
    for (int q = 0; q < 2; ++q) {
      g->oz.mat[d][q] = (const char*)g->d_oz + off[d][q];
      g->oz.rexp[d][q] = (const int*)((const char*)g->d_oz + off[d][q] + one - 512);
    }
  }
  if (all) g->oz.inv = (double*)((char*)g->d_oz + bytes);
  const int cap = (int)std::max(oz_smem(112), oz_smem(kOzMax));
  FV_CUDA(cudaFuncSetAttribute(k_oz<true, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  FV_CUDA(cudaFuncSetAttribute(k_oz<false, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  FV_CUDA(cudaFuncSetAttribute(k_oz<false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  FV_CUDA(cudaFuncSetAttribute(k_oz<false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  return FV_OK;
}

fv_status fill_oz_factors(fv_grid* g) {
  if (!g->oz.inv) return FV_OK;
  k_inv_lam<<<(unsigned)std::min<int64_t>((g->ncell + 255) / 256, 152 * 16), 256, 0, g->stream>>>(
      g->tpf_d, g->oz.inv, g->ncell);
  FV_CHECK_LAUNCH();
  return FV_OK;
}

fv_status oz_transform(const fv_grid* g, int axis, int inverse, OzScale scale, const double* in, double* out) {
  OzArgs A;
  A.in = in;
  A.out = out;
  A.mat = (const bf16b*)g->oz.mat[axis][inverse];
  A.rexp = g->oz.rexp[axis][inverse];
  A.sc = scale;
  A.n = g->n[axis];
  A.nvec = g->ncell / A.n;
  A.Q = axis == 0 ? 1 : axis == 1 ? g->n[0] : (int64_t)g->n[0] * g->n[1];
  A.fault = g->d_fault;
  const int N = tile_n(A.n);
  const dim3 grid((unsigned)((A.nvec + N - 1) / N));
  LaunchScope ls_(g, axis == 0 ? FV_K_TPF_X : FV_K_TPF_YZ);
  auto* kern = axis == 0 ? k_oz<true, 0> : !scale.inv ? k_oz<false, 0> : scale.na ? k_oz<false, 2> : k_oz<false, 1>;
  FV_CUDA(tc5::launch_pdl(kern, grid, dim3(kOzThreads), oz_smem(A.n), g->stream, A));
  return FV_OK;
}

}  // namespace fv
