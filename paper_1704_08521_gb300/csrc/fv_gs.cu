// One Gram-Schmidt step of the Krylov methods (Section 3) as one kernel: the
// new vector w against the first j1 basis vectors by classical Gram-Schmidt
// applied twice in the W-inner product, its norm, and its normalised copy as
// the next basis vector, in float-float arithmetic on the FP32 pipes.
//
// On the small grids where GMRES and Arnoldi take thousands of vectors the
// work of a step is a few microseconds (16^3 cells, 50 vectors: 5 MB from L2),
// yet it took twelve launches: two inner products and their reductions, two
// updates, the norm and its reduction, the Hessenberg column, the scaling.
// Here every block keeps one slice of w in shared memory through the whole
// step and reads its slice of the basis four times; between the phases the
// blocks meet at a barrier in global memory (a cooperative launch: all blocks
// are resident).  Five barriers:
//   partial products (w, v) | one block per v sums them | update, partial
//   products again | sums | update, partial norm | norm, scaling.
// A wait at a barrier is bounded; a block that gives up raises the grid's
// timeout word and still arrives at the barriers that are left.  With the word
// set the coefficients, the norm and the new vector are NaN (of a block that
// gives up at the last barrier only: its slice).
#include <algorithm>

#include "fv_ff.cuh"
#include "fv_internal.cuh"

namespace fv {

namespace {

constexpr int kGsThreads = 512;
constexpr int kGsWarps = kGsThreads / 32;
constexpr int kGsMaxVec = 130;
constexpr int kGsGroup = 4;              // basis vectors a warp takes at a time
constexpr int kGsMaxSlice = 3072;        // entries of w per block at most: see gs_shape
constexpr int kGsPolls = 1 << 20;        // polls of a barrier before a block gives up

__device__ __forceinline__ ff entry(const double* p) { return f64_split_trunc(__ldg(p)); }
__device__ __forceinline__ ff entry(const float2* p) {
  const float2 v = __ldg(p);
  return ff{v.x, v.y};
}

struct GsArgs {
  const void* V;            // basis, columns of ldv entries
  int64_t ldv;
  int j1;                   // vectors in it
  double* w;                // in: the new vector; out: orthogonalised (and scaled: scale_w)
  const float2* W;          // face weights
  int64_t n;
  int slice;                // entries per block
  double* part;             // [kGsMaxVec][blocks]
  double* h;                // [2][kGsMaxVec]: the coefficients of the two passes
  unsigned long long* bar;  // arrivals since the counter was made; whole barriers only
  unsigned* fault;
  double* hcol;             // column of H: j1 coefficients and the norm, ldh apart
  int64_t ldh;
  double* scale;            // 1 / norm (0 for a zero vector); may be null
  float2* colf;             // next basis vector as float-float pairs, or null
  int scale_w;              // w /= norm
  int norm_only;            // write the norm alone into hcol
};

__device__ __forceinline__ ff add(ff a, ff b) {     // TwoSum and one renormalisation, as the other sums
  ff s = two_sum(a.hi, b.hi);
  s.lo += a.lo + b.lo;
  return fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ ff shfl(ff a, int o) {
  return ff{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

// all blocks meet; false once a wait has given up
__device__ bool meet(const GsArgs& A, bool ok) {
  __shared__ int good;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned long long t = atomicAdd(A.bar, 1ull);
    const unsigned long long goal = (t / gridDim.x + 1) * gridDim.x;
    int polls = 0;
    if (ok) {
      unsigned long long now;
      do {
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(now) : "l"(A.bar) : "memory");
      } while (now < goal && ++polls < kGsPolls);
      ok = now >= goal;
      if (!ok) atomicOr(A.fault, 1u);
    }
    __threadfence();
    good = ok;
  }
  __syncthreads();
  return good != 0;
}

// partial[v][block] = sum over the slice of (W w) v.  The entries are cut into
// `seg` runs, 16 / seg warps each; a warp takes kGsGroup vectors at a time
// over its run and adds its lanes so that the first exchange halves the number
// of sums a lane holds.
template <typename VT>
__device__ void dots(const GsArgs& A, const VT* Vs, int cnt, const float2* ww, float2* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int seg = 1;
  while (seg < kGsWarps && cnt > 128 * seg) seg <<= 1;
  const int run = ((cnt + seg - 1) / seg + 31) & ~31;
  const int s = warp % seg, g0 = warp / seg, gs = kGsWarps / seg;
  const int lo = min(cnt, s * run), hi = min(cnt, lo + run);
  for (int v = g0 * kGsGroup; v < A.j1; v += gs * kGsGroup) {
    ff acc[kGsGroup];
    const VT* p[kGsGroup];
#pragma unroll
    for (int q = 0; q < kGsGroup; ++q) {
      acc[q] = ff{0.f, 0.f};
      p[q] = Vs + (int64_t)min(v + q, A.j1 - 1) * A.ldv;
    }
#pragma unroll 2
    for (int e = lo + lane; e < hi; e += 32) {
      const float2 x = ww[e];
      ff b[kGsGroup];
#pragma unroll
      for (int q = 0; q < kGsGroup; ++q) b[q] = entry(p[q] + e);
#pragma unroll
      for (int q = 0; q < kGsGroup; ++q) ff_mad(acc[q], ff{x.x, x.y}, b[q]);
    }
    static_assert(kGsGroup == 4, "two halving exchanges");
    const bool up = lane & 16, uq = lane & 8;
    const ff k0 = up ? acc[2] : acc[0], k1 = up ? acc[3] : acc[1];
    const ff t0 = add(k0, shfl(up ? acc[0] : acc[2], 16)), t1 = add(k1, shfl(up ? acc[1] : acc[3], 16));
    ff t = add(uq ? t1 : t0, shfl(uq ? t0 : t1, 8));
    t = add(t, shfl(t, 4));
    t = add(t, shfl(t, 2));
    t = add(t, shfl(t, 1));
    const int q = (up ? 2 : 0) + (uq ? 1 : 0);
    if ((lane & 7) == 0 && v + q < A.j1) red[s * kGsMaxVec + v + q] = make_float2(t.hi, t.lo);
  }
  __syncthreads();
  for (int v = threadIdx.x; v < A.j1; v += kGsThreads) {
    ff t{red[v].x, red[v].y};
    for (int q = 1; q < seg; ++q) t = add(t, ff{red[q * kGsMaxVec + v].x, red[q * kGsMaxVec + v].y});
    __stcg(A.part + (int64_t)v * gridDim.x + blockIdx.x, (double)t.hi + (double)t.lo);
  }
}

// the blocks' partial sums of vector v, by one warp (every lane gets the sum)
__device__ double gather(const GsArgs& A, int v) {
  double s = 0.0;
  for (int b = threadIdx.x & 31; b < (int)gridDim.x; b += 32) s += __ldcg(A.part + (int64_t)v * gridDim.x + b);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// w -= sum_v h_v v on the slice; ws (w) and ww (W w) are rewritten
template <typename VT>
__device__ void update(const GsArgs& A, const VT* Vs, int cnt, const double* h, int64_t e0, float2* hs,
                       float2* comb, float2* ws, float2* ww) {
  for (int v = threadIdx.x; v < A.j1; v += kGsThreads) {
    const ff x = f64_split_trunc(-__ldcg(h + v));
    hs[v] = make_float2(x.hi, x.lo);
  }
  __syncthreads();
  int E = kGsThreads;                       // threads along the entries; the others share the vectors
  while (E > 32 && E / 2 >= cnt) E >>= 1;
  const int ng = kGsThreads / E, t = threadIdx.x % E, gq = threadIdx.x / E;
  for (int b = 0; b < cnt; b += E) {
    const int e = b + t;
    ff s{0.f, 0.f};
    if (e < cnt) {
      const VT* p = Vs + e;
      int v = gq;
      for (; v + 3 * ng < A.j1; v += 4 * ng) {
        ff a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = entry(p + (int64_t)(v + q * ng) * A.ldv);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 c = hs[v + q * ng];
          ff_mad(s, ff{c.x, c.y}, a[q]);
        }
      }
      for (; v < A.j1; v += ng) {
        const float2 c = hs[v];
        ff_mad(s, ff{c.x, c.y}, entry(p + (int64_t)v * A.ldv));
      }
    }
    if (ng > 1) {
      comb[threadIdx.x] = make_float2(s.hi, s.lo);
      __syncthreads();
    }
    if (gq == 0 && e < cnt) {
      for (int q = 1; q < ng; ++q) s = add(s, ff{comb[q * E + t].x, comb[q * E + t].y});
      const ff x = ff_add(ff{ws[e].x, ws[e].y}, s);
      ws[e] = make_float2(x.hi, x.lo);
      const float2 wt = __ldg(A.W + e0 + e);
      const ff y = ff_mul(ff{wt.x, wt.y}, x);
      ww[e] = make_float2(y.hi, y.lo);
    }
    if (ng > 1) __syncthreads();
  }
  __syncthreads();
}

// What bounds it: at 16^3 the chain of five barriers (about 1 us each) and the
// latency of the loads between them; from about 40^3 the float-float
// multiply-adds (about a dozen FP32 instructions per basis entry and pass).
template <typename VT>
__global__ void __launch_bounds__(kGsThreads) k_cgs2(GsArgs A) {
  extern __shared__ float2 sm[];
  __shared__ float2 hs[kGsMaxVec], comb[kGsThreads], red[kGsWarps * kGsMaxVec];
  float2* ws = sm;
  float2* ww = sm + A.slice;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t e0 = (int64_t)blockIdx.x * A.slice;
  const int cnt = (int)min((int64_t)A.slice, A.n - e0);
  const VT* Vs = (const VT*)A.V + e0;
  for (int e = tid; e < cnt; e += kGsThreads) {
    const ff x = f64_split_trunc(A.w[e0 + e]);
    const float2 wt = __ldg(A.W + e0 + e);
    const ff y = ff_mul(ff{wt.x, wt.y}, x);
    ws[e] = make_float2(x.hi, x.lo);
    ww[e] = make_float2(y.hi, y.lo);
  }
  __syncthreads();
  bool ok = true;
  for (int pass = 0; pass < 2; ++pass) {
    double* h = A.h + pass * kGsMaxVec;
    dots<VT>(A, Vs, cnt, ww, red);
    ok = meet(A, ok);
    for (int v = blockIdx.x + gridDim.x * warp; v < A.j1; v += gridDim.x * kGsWarps) {
      const double s = gather(A, v);
      if (lane == 0) __stcg(h + v, s);
    }
    ok = meet(A, ok);
    update<VT>(A, Vs, cnt, h, e0, hs, comb, ws, ww);
  }
  {                                          // the norm: (W w, w) over the slice
    ff s{0.f, 0.f};
    for (int e = tid; e < cnt; e += kGsThreads) ff_mad(s, ff{ww[e].x, ww[e].y}, ff{ws[e].x, ws[e].y});
    for (int o = 16; o > 0; o >>= 1) s = add(s, shfl(s, o));
    if (lane == 0) red[warp] = make_float2(s.hi, s.lo);
    __syncthreads();
    if (tid == 0) {
      for (int q = 1; q < kGsWarps; ++q) s = add(s, ff{red[q].x, red[q].y});
      __stcg(A.part + blockIdx.x, (double)s.hi + (double)s.lo);
    }
  }
  ok = meet(A, ok);
  __shared__ double norm;
  if (warp == 0) {
    double s = gather(A, 0);
    if (!ok || *reinterpret_cast<const volatile unsigned*>(A.fault)) s = __longlong_as_double(0x7ff8000000000000ll);
    if (lane == 0) norm = s < 0.0 ? 0.0 : sqrt(s);
  }
  __syncthreads();
  const double hn = norm, sc = hn == 0.0 ? 0.0 : 1.0 / hn;
  if (blockIdx.x == 0) {
    if (!A.norm_only)
      for (int v = tid; v < A.j1; v += kGsThreads)
        A.hcol[(int64_t)v * A.ldh] = isnan(hn) ? hn : __ldcg(A.h + v) + __ldcg(A.h + kGsMaxVec + v);
    if (tid == 0) {
      A.hcol[(int64_t)A.j1 * A.ldh] = hn;
      if (A.scale) *A.scale = sc;
    }
  }
  const double m = isnan(hn) || (A.scale_w && hn != 0.0) ? sc : 1.0;
  for (int e = tid; e < cnt; e += kGsThreads) {
    const double x = ff_join(ws[e].x, ws[e].y);
    A.w[e0 + e] = m * x;
    if (A.colf) {
      const ff s = f64_split_trunc(sc * x);
      A.colf[e0 + e] = make_float2(s.hi, s.lo);
    }
  }
}

}  // namespace

// Blocks and entries per block of a step on this grid; false beyond
// kGsMaxSlice.  Leading eigenvalues with m = 40, microseconds per new vector, this
// kernel against the separate ones (runs of the same input repeat to 0.1 %):
// 16^3 127 / 158, 32^3 163 / 191, 40^3 197 / 228, 48^3 252 / 276, 52^3 316 / 324
// (2776 entries per block), 56^3 376 / 350 (3468), 64^3 525 / 441: a basis beyond
// L2 is better streamed by three blocks per SM with asynchronous copies.  Newton
// at 16^3: 449 ms with the separate kernels, 344 with this one.
static bool gs_shape(const fv_grid* g, int* blocks, int* slice) {
  static const int sms = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v;
  }();
  if (sms < 1) return false;
  const int64_t n = g->nvel;
  int64_t per = (n + sms - 1) / sms;
  per = std::max<int64_t>((per + 1) & ~(int64_t)1, 32);
  if (per > kGsMaxSlice) return false;
  *slice = (int)per;
  *blocks = (int)((n + per - 1) / per);
  return true;
}

bool gs_fused_ok(const fv_grid* g, int j1) {
  int b, s;
  return j1 > 0 && j1 <= kGsMaxVec && gs_shape(g, &b, &s);
}

fv_status gs_fused(const fv_grid* g, const void* V, bool pairs, int64_t ldv, int j1, double* w, double* h2,
                   unsigned long long* bar, double* hcol, int64_t ldh, double* scale, float2* colf,
                   bool scale_w, bool norm_only) {
  GsArgs A;
  int blocks;
  if (!gs_shape(g, &blocks, &A.slice)) { set_error("gs_fused: vectors too long"); return FV_EINVAL; }
  A.V = V;
  A.ldv = ldv;
  A.j1 = j1;
  A.w = w;
  A.W = g->wts_ff;
  A.n = g->nvel;
  A.part = g->d_part;
  A.h = h2;
  A.bar = bar;
  A.fault = g->d_fault;
  A.hcol = hcol;
  A.ldh = ldh;
  A.scale = scale;
  A.colf = colf;
  A.scale_w = scale_w ? 1 : 0;
  A.norm_only = norm_only ? 1 : 0;
  const void* f = pairs ? (const void*)k_cgs2<float2> : (const void*)k_cgs2<double>;
  const size_t smem = 2 * (size_t)A.slice * sizeof(float2);
  if (smem > 16 * 1024)
    FV_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 2 * kGsMaxSlice * (int)sizeof(float2)));
  LaunchScope ls_(g, FV_K_DOTS);
  void* args[1] = {&A};
  FV_CUDA(cudaLaunchCooperativeKernel(f, dim3(blocks), dim3(kGsThreads), args, smem, g->stream));
  return FV_OK;
}

}  // namespace fv
