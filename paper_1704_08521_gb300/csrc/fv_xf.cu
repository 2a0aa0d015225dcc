// Float32 tensor-product transforms of long axes on the tensor cores.
//
// The fused kernels of fv_poisson.cu hold a whole plane in shared memory and
// end at about 112 cells per axis.  Beyond that each transform
//   out[v][p] = sum_k M[p][k] in[v][k]
// is one GEMM here, accurate to float32: every operand is written as the sum
// of three BF16 numbers (x = h + m + l, each the rounding of what is left: 24
// bits) and the six products h h, h m, m h, h l, m m, l h are accumulated in
// float32 in tensor memory (tcgen05 kind::f16); the three others are below
// 2^-24 of the product.  Six BF16 products cost what three TF32 ones do, carry
// two more bits and need 6 instead of 8 bytes of shared memory per element.
//
// The tensor core cuts off what a sum has beyond float32 (an FP32 FMA rounds), so
// every addition to an accumulator takes up to an ulp of it away: 6 n / 16 of
// them, all in one accumulator, made the solution 3e-6 .. 5e-6 of its largest
// value wrong (sine map, 150^3), five times what the FP32 kernel's sums of n
// terms did.  So h h, which carries the value, has an accumulator of its own
// (n / 16 additions), cut in two halves of K where tensor memory has room for
// three, and the five small products share another, whose cuts are 2^-8 of
// that; the epilogue adds them.  Error of the first correction against float64,
// relative to the FP32 kernels' (113 .. 520 cells, cosine and sine map): 0.15 ..
// 0.7 in the mean square, 0.15 .. 1.2 in the largest.
//
// One block: 128 K-vectors of the field (the M side, one tensor-memory lane
// each) and a chunk of the rows of M (the N side, the columns).  K streams
// through a ring of 16-entry chunks: the chunk of the pre-split matrix by a bulk
// copy, the chunk of the field through registers (loaded two turns ahead, split
// and stored by two sets of eight warps in turn).  One more warp issues the
// products, another the copies.  Chunks of up to 128 rows let two blocks share
// an SM, so that one's epilogue overlaps the other's products; from 161 to 256
// rows one chunk, one block per SM, since splitting the field twice costs more
// (256^3 3860 us against 3980, 192^3 2255 against 2331; 150^3 1033 us with two
// chunks of 80 rows against 1048 with one).  A float-float evaluation at 150^3 takes
// 1033 us and at 256^3 3864 us, 1606 and 7730 with the FP32 kernels this replaces; with
// all products in one accumulator it took 924 and 3631.
#include <algorithm>
#include <cstring>
#include <vector>

#include <cuda_bf16.h>

#include "fv_internal.cuh"
#include "fv_tc5.cuh"

namespace fv {

namespace {

constexpr int kXGroups = 2;            // sets of eight warps that take the chunks in turn
constexpr int kXWorkers = 8 * kXGroups;
constexpr int kXThreads = 32 * (kXWorkers + 2);
constexpr int kXStages = 4;
constexpr int kXABytes = 3 * 128 * 16 * 2;
constexpr int kXLimit = 1 << 22;       // polls of an mbarrier before the block gives up

__host__ __device__ inline int up16(int n) { return (n + 15) & ~15; }
// rows of M per block at most, chunks of them, rows of a chunk (a multiple of 16, all equal)
__host__ __device__ inline int max_rows(int n) { return up16(n) > 160 && up16(n) <= 256 ? 256 : 128; }
__host__ __device__ inline int chunks_of(int n) { return (up16(n) + max_rows(n) - 1) / max_rows(n); }
__host__ __device__ inline int chunk_rows(int n) { return up16((n + chunks_of(n) - 1) / chunks_of(n)); }
// accumulators of N columns: three where two blocks of an SM still fit its 512
__host__ __device__ inline int accs(int N) { return 3 * N <= 256 ? 3 : 2; }
inline size_t xf_smem(int n) { return (size_t)kXStages * (kXABytes + 96 * chunk_rows(n)); }

struct XfArgs {
  const float* in;
  float* out;
  const unsigned char* mat;   // [chunk of rows][K / 16][3][rows x 16 canonical]
  const float *lx, *ly, *lz;  // SCALE: eigenvalues
  int n, nx, null_x, null_y, null_z;
  int64_t nvec, Q;            // vectors; entry k of vector v is at (v / Q) n Q + k Q + v % Q
  uint32_t tcols;
  unsigned* fault;
  const int* skip;            // nothing to do once nonzero
};

// two floats -> BF16 pair (lo in the lower half); the floats become the rests
__device__ __forceinline__ uint32_t split2(float& a, float& b) {
  uint32_t w;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(b), "f"(a));
  a -= __uint_as_float(w << 16);
  b -= __uint_as_float(w & 0xffff0000u);
  return w;
}

template <bool RIGHT, bool SCALE>
__global__ void __launch_bounds__(kXThreads, 2) k_xf(XfArgs A) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t full[kXStages], ready[kXStages], empty[kXStages], done;
  __shared__ uint32_t tslot;
  __shared__ int bad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = A.n, nk = (n + 15) >> 4, N = chunk_rows(n), nch = chunks_of(n);
  const int chunk = (int)(blockIdx.x % (unsigned)nch), p0 = chunk * N;
  const int nkh = accs(N) == 3 ? (nk + 1) / 2 : nk;   // chunks whose h h goes to the first accumulator
  const int bbytes = 96 * N, sbytes = kXABytes + bbytes;
  const int64_t v0 = (int64_t)(blockIdx.x / (unsigned)nch) * 128;
  const unsigned char* mat = A.mat + (size_t)chunk * nk * bbytes;
  if (tid == 0) {
    for (int s = 0; s < kXStages; ++s) {
      tc5::mbar_init(&full[s], 1);
      tc5::mbar_init(&ready[s], 8);
      tc5::mbar_init(&empty[s], 1);
    }
    tc5::mbar_init(&done, 1);
    bad = 0;
    tc5::fence_proxy_async();
    for (int c = 0; c < kXStages && c < nk; ++c)
      tc5::bulk_load(sm + c * sbytes + kXABytes, mat + (size_t)c * bbytes, bbytes, &full[c]);
  }
  // everything above uses constants only; the field is the predecessor's
  // output.  Tensor memory is taken after the wait and the successor let in
  // after that, so that no block waits for columns held by a kernel that waits
  // for this one.
  tc5::pdl_wait();
  if (A.skip && *A.skip != 0) {          // the loop ended before this pass
    if (tid == 0)                        // no copy may outlive the block
      for (int c = 0; c < kXStages && c < nk; ++c) tc5::mbar_wait(&full[c], 0, kXLimit);
    return;
  }
  if (warp == 0) tc5::tmem_alloc(&tslot, A.tcols);
  tc5::fence_before_sync();
  __syncthreads();
  tc5::fence_after_sync();
  tc5::pdl_trigger();
  const uint32_t tmem = tslot;
  if (warp < kXWorkers) {
    // this thread's vector and its 8-entry run of every chunk.  LEFT: a warp
    // reads 32 consecutive vectors; RIGHT: 16 vectors x 2 runs (64 contiguous
    // bytes each).  Eight consecutive lanes fill a core matrix either way.
    const int w8 = warp & 7, grp = warp >> 3;
    const int vl = RIGHT ? 16 * w8 + (lane & 15) : 32 * (w8 & 3) + lane;
    const int run = RIGHT ? lane >> 4 : w8 >> 2;
    const int64_t v = v0 + vl;
    const bool ok = v < A.nvec;
    const float* src = A.in;
    if (ok) src += RIGHT ? v * n : (v / A.Q) * n * A.Q + v % A.Q;
    const int64_t sk = RIGHT ? 1 : A.Q;
    const bool vec = RIGHT && (n & 3) == 0 && ((uintptr_t)A.in & 15) == 0;
    unsigned char* dst = sm + tc5::canon_offset16(vl, 8 * run, 16);
    float x[2][8];
    auto load = [&](int c, float (&y)[8]) {
      const int k = 16 * c + 8 * run;
      if (vec && ok && k + 8 <= n) {
        const float4 f0 = __ldg(reinterpret_cast<const float4*>(src + k));
        const float4 f1 = __ldg(reinterpret_cast<const float4*>(src + k) + 1);
        y[0] = f0.x; y[1] = f0.y; y[2] = f0.z; y[3] = f0.w;
        y[4] = f1.x; y[5] = f1.y; y[6] = f1.z; y[7] = f1.w;
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) y[q] = (ok && k + q < n) ? __ldg(src + (k + q) * sk) : 0.f;
      }
    };
    if (grp < nk) load(grp, x[0]);
    if (grp + kXGroups < nk) load(grp + kXGroups, x[1]);
    bool live = true;
    auto step = [&](int c, float (&y)[8]) {
      uint32_t w[3][4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float a = y[2 * q], b = y[2 * q + 1];
        w[0][q] = split2(a, b);
        w[1][q] = split2(a, b);
        w[2][q] = split2(a, b);
      }
      if (c + 2 * kXGroups < nk) load(c + 2 * kXGroups, y);
      const int st = c % kXStages, use = c / kXStages;
      // the products that read this stage before are done
      if (use > 0) live = tc5::mbar_wait(&empty[st], (uint32_t)(use - 1) & 1u, kXLimit) && live;
      unsigned char* d = dst + st * sbytes;
#pragma unroll
      for (int s = 0; s < 3; ++s)
        *reinterpret_cast<uint4*>(d + s * 4096) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
      tc5::fence_proxy_async();
      __syncwarp();
      if (lane == 0) tc5::mbar_arrive(&ready[st]);
    };
    for (int c = grp; c < nk; c += 2 * kXGroups) {
      step(c, x[0]);
      if (c + kXGroups < nk) step(c + kXGroups, x[1]);
    }
    if (!live) bad = 1;
  } else if (warp == kXWorkers && lane == 0) {
    bool ok = true;
    const uint32_t idesc = tc5::idesc_bf16(128, N);
    const uint32_t base = tc5::smem_u32(sm);
    for (int c = 0; c < nk; ++c) {
      const int st = c % kXStages;
      const uint32_t ph = (uint32_t)(c / kXStages) & 1u;
      ok = tc5::mbar_wait(&full[st], ph, kXLimit) && ok;
      ok = tc5::mbar_wait(&ready[st], ph, kXLimit) && ok;
      tc5::fence_after_sync();
      const uint32_t a = base + st * sbytes, b = a + kXABytes;
      const bool first = c == 0 || c == nkh;   // of a main accumulator
#pragma unroll
      for (int s = 2; s >= 0; --s)             // small products first
#pragma unroll
        for (int i = 0; i <= s; ++i)
          tc5::mma_f16(tmem + (uint32_t)(s ? N : c < nkh ? 0 : 2 * N), tc5::sdesc(a + i * 4096, 128, 256),
                       tc5::sdesc(b + (s - i) * 32 * N, 128, 256), idesc,
                       (s == 0 ? first : s == 2 && i == 0 && c == 0) ? 0u : 1u);
      tc5::commit(&empty[st]);
    }
    tc5::commit(&done);
    ok = tc5::mbar_wait(&done, 0, kXLimit) && ok;
    if (!ok) bad = 1;
  } else if (warp == kXWorkers + 1 && lane == 0) {
    bool ok = true;
    for (int c = kXStages; c < nk; ++c) {
      const int st = c % kXStages;
      ok = tc5::mbar_wait(&empty[st], (uint32_t)(c / kXStages - 1) & 1u, kXLimit) && ok;
      tc5::bulk_load(sm + st * sbytes + kXABytes, mat + (size_t)c * bbytes, bbytes, &full[st]);
    }
    if (!ok) bad = 1;
  }
  __syncthreads();
  tc5::fence_after_sync();
  const bool failed = bad != 0;
  if (tid == 0 && failed) atomicOr(A.fault, 1u);   // reported as FV_ETIMEOUT
  if (warp < kXWorkers) {
    const int64_t v = v0 + 32 * (warp & 3) + lane;
    const bool ok = v < A.nvec;
    const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    const int per = (N / 8 + kXWorkers / 4 - 1) / (kXWorkers / 4) * 8;
    const int c_begin = min(N, (warp >> 2) * per), c_end = min(N, c_begin + per);
    float* o = A.out;
    if (ok) o += RIGHT ? v * n : (v / A.Q) * n * A.Q + v % A.Q;
    float lq = 0.f;
    bool nullq = false;
    if (SCALE && ok) {
      const int i = (int)(v % A.nx), j = (int)(v / A.nx);
      lq = __ldg(A.lx + i) + __ldg(A.ly + j);
      nullq = i == A.null_x && j == A.null_y;
    }
    const bool vec4 = RIGHT && (n & 3) == 0 && ((uintptr_t)A.out & 15) == 0;
    const bool vec2 = RIGHT && (n & 1) == 0 && ((uintptr_t)A.out & 7) == 0;
    for (int c = c_begin; c < c_end; c += 8) {
      float y[8], z[8];
      __syncwarp();   // tcgen05.ld is warp-collective
      tc5::ld8(trow + (uint32_t)c, y);
      tc5::ld8(trow + (uint32_t)(N + c), z);
      if (nkh < nk) {
        float y2[8];
        tc5::ld8(trow + (uint32_t)(2 * N + c), y2);
#pragma unroll
        for (int q = 0; q < 8; ++q) y[q] += y2[q];
      }
      const int p = p0 + c;
      if (!ok || p >= n) continue;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        y[q] += z[q];
        if (SCALE) {
          const float l = p + q < n ? __ldg(A.lz + p + q) : 1.f;
          y[q] = (nullq && p + q == A.null_z) ? 0.f : y[q] / (l + lq);
        }
        if (failed) y[q] = __int_as_float(0x7fc00000);
      }
      if (vec4 && p + 8 <= n) {
        *reinterpret_cast<float4*>(o + p) = make_float4(y[0], y[1], y[2], y[3]);
        *reinterpret_cast<float4*>(o + p + 4) = make_float4(y[4], y[5], y[6], y[7]);
      } else if (vec2) {
#pragma unroll
        for (int q = 0; q < 8; q += 2)
          if (p + q < n) *reinterpret_cast<float2*>(o + p + q) = make_float2(y[q], y[q + 1]);
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (p + q < n) o[RIGHT ? (int64_t)(p + q) : (p + q) * A.Q] = y[q];
      }
    }
  }
  tc5::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc5::tmem_dealloc(tmem, A.tcols);
}

uint16_t bf16_host(float x) {        // round to nearest even (finite x)
  uint32_t u;
  std::memcpy(&u, &x, 4);
  return (uint16_t)((u + 0x7fffu + ((u >> 16) & 1u)) >> 16);
}

// the n x n row-major matrix M in three BF16 parts, in the order the kernel
// streams them
size_t mat_bytes(int n) { return (size_t)chunks_of(n) * up16(n) / 16 * 96 * chunk_rows(n); }

void lay_out(const std::vector<double>& M, int n, unsigned char* out) {
  const int N = chunk_rows(n), nk = up16(n) / 16;
  std::memset(out, 0, mat_bytes(n));
  for (int p = 0; p < n; ++p)
    for (int k = 0; k < n; ++k) {
      double x = M[(size_t)p * n + k];
      unsigned char* blk = out + ((size_t)(p / N) * nk + (k >> 4)) * 96 * N;
      for (int s = 0; s < 3; ++s) {
        const uint16_t b = bf16_host((float)x);
        std::memcpy(blk + s * 32 * N + tc5::canon_offset16(p % N, k & 15, 16), &b, 2);
        const uint32_t u = (uint32_t)b << 16;
        float f;
        std::memcpy(&f, &u, 4);
        x -= (double)f;
      }
    }
}

}  // namespace

fv_status build_xf(fv_grid* g) {
  // where the fused kernels do not serve the grid
  if (g->tc.ready) return FV_OK;
  size_t bytes = 0, off[3][2];
  int same[3];
  for (int d = 0; d < 3; ++d) {
    same[d] = d;
    for (int e = d - 1; e >= 0; --e)
      if (g->n[e] == g->n[d]) same[d] = e;
    for (int q = 0; q < 2; ++q) {
      if (same[d] != d) { off[d][q] = off[same[d]][q]; continue; }
      off[d][q] = bytes;
      bytes += (mat_bytes(g->n[d]) + 255) / 256 * 256;
    }
  }
  std::vector<unsigned char> h(bytes);
  for (int d = 0; d < 3; ++d)
    if (same[d] == d)
      for (int q = 0; q < 2; ++q) lay_out(q == 0 ? g->basis[d].Einv : g->basis[d].E, g->n[d], h.data() + off[d][q]);
  if (cudaMalloc(&g->d_xf, bytes) != cudaSuccess) {
    (void)cudaGetLastError();
    g->d_xf = nullptr;
    set_error("cudaMalloc of the tensor-core operands failed");
    return FV_ENOMEM;
  }
  g->ws_bytes += (int64_t)bytes;
  FV_CUDA(cudaMemcpy(g->d_xf, h.data(), bytes, cudaMemcpyHostToDevice));
  for (int d = 0; d < 3; ++d)
    for (int q = 0; q < 2; ++q) g->xf[d][q] = (const unsigned char*)g->d_xf + off[d][q];
  const int cap = (int)xf_smem(256);
  FV_CUDA(cudaFuncSetAttribute(k_xf<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  FV_CUDA(cudaFuncSetAttribute(k_xf<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  FV_CUDA(cudaFuncSetAttribute(k_xf<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  return FV_OK;
}

static fv_status xf_transform(const fv_grid* g, int axis, int inverse, bool scale, const float* in, float* out,
                              const int* skip) {
  XfArgs A;
  A.in = in;
  A.out = out;
  A.mat = g->xf[axis][inverse];
  A.lx = g->tpf_f.lam[0];
  A.ly = g->tpf_f.lam[1];
  A.lz = g->tpf_f.lam[2];
  A.n = g->n[axis];
  A.nx = g->n[0];
  A.null_x = g->tpf_f.null_index[0];
  A.null_y = g->tpf_f.null_index[1];
  A.null_z = g->tpf_f.null_index[2];
  A.nvec = g->ncell / A.n;
  A.Q = axis == 0 ? 1 : axis == 1 ? g->n[0] : (int64_t)g->n[0] * g->n[1];
  A.tcols = 32;
  while ((int)A.tcols < accs(chunk_rows(A.n)) * chunk_rows(A.n)) A.tcols <<= 1;
  A.fault = g->d_fault;
  A.skip = skip;
  const dim3 grid((unsigned)((A.nvec + 127) / 128 * chunks_of(A.n)));
  const size_t smem = xf_smem(A.n);
  LaunchScope ls_(g, axis == 0 ? FV_K_TPF_X : FV_K_TPF_YZ);
  if (axis == 0) FV_CUDA(tc5::launch_pdl(k_xf<true, false>, grid, dim3(kXThreads), smem, g->stream, A));
  else if (scale) FV_CUDA(tc5::launch_pdl(k_xf<false, true>, grid, dim3(kXThreads), smem, g->stream, A));
  else FV_CUDA(tc5::launch_pdl(k_xf<false, false>, grid, dim3(kXThreads), smem, g->stream, A));
  return FV_OK;
}

bool xf_ok(const fv_grid* g) { return g->d_xf != nullptr; }

fv_status xf_solve(const fv_grid* g, const float* r, float* phi, const int* skip) {
  float* a = (float*)g->tpf_buf[0];
  float* b = (float*)g->tpf_buf[1];
  FV_TRY(xf_transform(g, 0, 0, false, r, a, skip));
  FV_TRY(xf_transform(g, 1, 0, false, a, b, skip));
  FV_TRY(xf_transform(g, 2, 0, true, b, a, skip));
  FV_TRY(xf_transform(g, 2, 1, false, a, b, skip));
  FV_TRY(xf_transform(g, 1, 1, false, b, a, skip));
  return xf_transform(g, 0, 1, false, a, phi, skip);
}

}  // namespace fv
