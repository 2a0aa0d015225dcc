// The SIMPLE passes of the evaluation graphs (Section 3, the algorithm after
// Eq. 10), compiled without FMA contraction so that every TwoSum and TwoProd
// keeps its rounding.
//
// A pass takes the new correction phi_m, forms the corrected velocity
// v - omega G phi_m and its divergence r = D v, the right-hand side of the next
// solve, in the order and with every rounding of the host-driven loop
// (k_correct_ff): both give the same bits.  v goes from one float-float buffer
// to the other, so that the next pass removes what this one's roundings left;
// p is summed by k_join, if it is asked for, from the first three corrections
// (three is the usual number), which are kept apart, or by the passes beyond
// the third.  A version that kept only the predictor and the corrections and
// formed v from them in every pass read less, but its float-float roundings were
// not seen by the following solve, and with the lower parts of the sums added in
// plain float32 |D v| came out 2 to 100 times larger.  With full sums it was no
// faster either: 100^3 mixed 225 us an evaluation against 217, 256^3 float-float
// 3990 against 3640.
//
// Every face belongs to two cells: a thread computes the three low faces of
// its cell and gets the high ones from its x and y neighbours through shared
// memory and, along z, from its own next plane (the block marches up a chunk
// of planes; the loads of the next plane are issued before a plane is
// computed).  A thread owns two cells adjacent along x: one address, predicate
// and access then serve both, and half of the x-faces stay in registers.  A
// block has one thread per pair of its TX x TY tile and one more row and
// column.
//
// The last block to finish reduces the block maxima, takes the loop's decision
// and sets the condition of the graph's WHILE node: no separate kernel.
//
// Bound by instruction issue (float-float arithmetic), not by memory (40 to 52 B
// per cell).  An evaluation with these passes takes 217 us at 100^3 mixed and
// 3640 us at 256^3 float-float, against 260 and 4216 us with one cell per thread
// and a kernel of its own for the decision; fetching the low neighbours a plane
// ahead as well cost registers and 20 % of the float-float time.
#include "fv_ff.cuh"
#include "fv_internal.cuh"
#include "fv_tc5.cuh"

namespace fv {

namespace {

__device__ __forceinline__ ff of2(float2 a) { return {a.x, a.y}; }
__device__ __forceinline__ float2 to2(ff a) { return make_float2(a.hi, a.lo); }

constexpr int kPassThreads = 320;

__device__ __forceinline__ float block_max(float v, float* red) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  v = lane < nw ? red[lane] : 0.f;
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;                       // every thread
}

// base value of a face in its stored form
__device__ __forceinline__ ff base_of(float w) { return {w, 0.f}; }
__device__ __forceinline__ ff base_of(float2 w) { return of2(w); }

// v at a face after one correction, a at this cell and b at its low neighbour:
// v - omega (a - b) / dc.  Mixed form: the gradient in float32, as the form's
// contract has it.
__device__ __forceinline__ ff face_mixed(ff v, float a, float b, float idc, float omega) {
  const float g = (a - b) * idc;
  return ff_add_f(v, -omega * g);
}

// Float-float form: the difference of two float32 values is an exact sum of two
// floats; product and subtraction in float-float.
__device__ __forceinline__ ff face_ff(ff v, float a, float b, float2 idc, float omega) {
  ff g = ff_mul(two_sum(a, -b), of2(idc));
  if (omega != 1.f) g = ff_mul_f(g, omega);
  return ff_sub(v, g);
}

// one direction of the divergence
__device__ __forceinline__ ff div_term(ff h, ff l, float2 idx) { return ff_mul(ff_sub(h, l), of2(idx)); }

struct PassArgs {
  MetFF m;
  const float* w32;            // mixed: the predictor
  float2* vff[2];              // v after n passes is in vff[(n + 1) & 1], so is the float-float predictor (n = 0)
  const float* phi[4];
  float2* p;
  float* r;
  const CallBlock* cb;
  LoopState* ls;
  float* part;
  const unsigned* fault;
  cudaGraphConditionalHandle h;
  int set_handle, decide;
  int idx;                     // which of the first three passes, 3: any later one
  int tx, ty, kz;
};

// two adjacent values: one access where VEC (p aligned), else p[0], p[second]
template <bool VEC>
__device__ __forceinline__ void load2(const float* p, int second, float (&v)[2]) {
  if (VEC) {
    const float2 t = __ldg(reinterpret_cast<const float2*>(p));
    v[0] = t.x;
    v[1] = t.y;
  } else {
    v[0] = __ldg(p);
    v[1] = __ldg(p + second);
  }
}
template <bool VEC>
__device__ __forceinline__ void load2(const float2* p, int second, float2 (&v)[2]) {
  if (VEC) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = make_float2(t.x, t.y);
    v[1] = make_float2(t.z, t.w);
  } else {
    v[0] = __ldg(p);
    v[1] = __ldg(p + second);
  }
}

// values of one plane at this thread's two cells
template <typename TB>
struct Plane {
  float f[2];                  // the correction
  TB b[3][2];                  // v
};

// One pass over the tile: v stored as TB -> vout with the correction phi, and
// p_terms corrections, the latest ones, to p (four: the first sum); VEC: nx is
// even, pairs are aligned.  Updates this thread's maxima of |phi| and |D v|.
// Loads are not predicated: indices are clamped to the grid, and what a wall or
// a thread beyond the grid loads that way is not used.
template <bool FF, typename TB, bool VEC>
__device__ __forceinline__ void pass_body(const PassArgs& A, const TB* __restrict__ base,
                                          const float* __restrict__ phi, float2* __restrict__ vout,
                                          int p_terms, float& aphi, float& adiv, float2* sh) {
  const MetFF& m = A.m;
  const int nx = m.n[0], ny = m.n[1], nz = m.n[2], nc = (int)m.ncell, nxy = nx * ny;
  const int LX = A.tx / 2 + 1;
  const int tid = threadIdx.x, li = tid % LX, lj = tid / LX;
  const int i = blockIdx.x * A.tx + 2 * li, j = blockIdx.y * A.ty + lj;
  const int k0 = blockIdx.z * A.kz, k1 = min(k0 + A.kz, nz);
  const bool in = lj <= A.ty && i < nx && j < ny;
  const bool in1 = VEC ? in : in && i + 1 < nx;
  const bool own = in && 2 * li < A.tx && lj < A.ty;
  const float omega = A.cb->omega;
  const int col = in ? j * nx + i : 0;
  const int dx = in && i > 0 ? 1 : 0, dy = in && j > 0 ? nx : 0, d1 = in1 ? 1 : 0;
  auto load = [&](int k, Plane<TB>& P) {
    const int e = min(k, nz - 1) * nxy + col;
    load2<VEC>(phi + e, d1, P.f);
    load2<VEC>(base + 2 * nc + e, d1, P.b[2]);
    if (k < k1) {                             // plane k1: only its low z-faces (the chunk's top)
      load2<VEC>(base + e, d1, P.b[0]);
      load2<VEC>(base + nc + e, d1, P.b[1]);
    }
  };
  float cx[2] = {0.f, 0.f}, cy = 0.f;
  float2 cxf[2] = {}, cyf = make_float2(0.f, 0.f), dxi[2] = {}, dyi = cyf;
  if (in) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (i + q < nx) {
        if (FF) cxf[q] = m.idcf[0][i + q];
        else cx[q] = m.idc[0][i + q];
        dxi[q] = m.idx[0][i + q];
      }
    if (FF) cyf = m.idcf[1][j];
    else cy = m.idc[1][j];
    dyi = m.idx[1][j];
  }
  auto face = [&](TB b, float a, float c, float idc, float2 idcf) -> ff {
    if constexpr (FF) return face_ff(base_of(b), a, c, idcf, omega);
    else return face_mixed(base_of(b), a, c, idc, omega);
  };
  float fz[2];                 // the correction of the plane below
  load2<VEC>(phi + max(k0 - 1, 0) * nxy + col, d1, fz);
  ff px[2] = {}, py[2] = {}, vzp[2] = {};    // of the plane whose z-face above is awaited
  const ff zero = {0.f, 0.f};
  // plane k (in cur; k + 1 is fetched into nxt)
  auto step = [&](int k, Plane<TB>& cur, Plane<TB>& nxt) {
    // the low neighbours of this plane: fetched one plane ago as other threads'
    // own cells, so near; the next plane itself: far, a plane ahead
    float fx, fy[2];
    {
      const int e = min(k, nz - 1) * nxy + col;
      fx = __ldg(phi + (e - dx));
      load2<VEC>(phi + (e - dy), d1, fy);
    }
    if (k < k1) load(k + 1, nxt);
    // low z-faces of plane k, which close plane k - 1
    ff vz[2] = {zero, zero};
    if (k > 0 && k < nz) {
      const float zc = FF ? 0.f : m.idc[2][k];
      const float2 zcf = FF ? m.idcf[2][k] : make_float2(0.f, 0.f);
      vz[0] = face(cur.b[2][0], cur.f[0], fz[0], zc, zcf);
      vz[1] = face(cur.b[2][1], cur.f[1], fz[1], zc, zcf);
    }
    if (k > k0 && own) {
      const float2 dz = m.idx[2][k - 1];
      float d[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        d[q] = ff_add(ff_add(px[q], py[q]), div_term(vz[q], vzp[q], dz)).hi;
        if (VEC || q == 0 || in1) {
          float a2 = fabsf(d[q]);
          if (!(a2 <= 3e38f)) a2 = __int_as_float(0x7f800000);
          adiv = fmaxf(adiv, a2);
        }
      }
      float* o = A.r + (k - 1) * nxy + col;
      if (VEC) {
        *reinterpret_cast<float2*>(o) = make_float2(d[0], d[1]);
      } else {
        o[0] = d[0];
        if (in1) o[1] = d[1];
      }
    }
    if (k == k1) return;
    ff vx[2], vy[2];
    vx[0] = face(cur.b[0][0], cur.f[0], fx, cx[0], cxf[0]);
    if (dx == 0) vx[0] = zero;
    vx[1] = face(cur.b[0][1], cur.f[1], cur.f[0], cx[1], cxf[1]);
    vy[0] = face(cur.b[1][0], cur.f[0], fy[0], cy, cyf);
    vy[1] = face(cur.b[1][1], cur.f[1], fy[1], cy, cyf);
    if (dy == 0) vy[0] = vy[1] = zero;
    float2* sx = sh + (k & 1) * 3 * kPassThreads;
    float4* sy = reinterpret_cast<float4*>(sx + kPassThreads);
    sx[tid] = to2(vx[0]);
    sy[tid] = make_float4(vy[0].hi, vy[0].lo, vy[1].hi, vy[1].lo);
    __syncthreads();
    if (own) {
      const ff x2 = i + 2 < nx ? of2(sx[tid + 1]) : zero;
      const float4 y2 = j + 1 < ny ? sy[tid + LX] : make_float4(0.f, 0.f, 0.f, 0.f);
      px[0] = div_term(VEC || in1 ? vx[1] : zero, vx[0], dxi[0]);
      px[1] = div_term(x2, vx[1], dxi[1]);
      py[0] = div_term({y2.x, y2.y}, vy[0], dyi);
      py[1] = div_term({y2.z, y2.w}, vy[1], dyi);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float u = fabsf(cur.f[q]);           // (beyond an odd row: the first cell again)
        if (!(u <= 3e38f)) u = __int_as_float(0x7f800000);
        aphi = fmaxf(aphi, u);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const ff(&o)[2] = c == 0 ? vx : c == 1 ? vy : vz;
        float2* d = vout + c * nc + k * nxy + col;
        if (VEC) {
          *reinterpret_cast<float4*>(d) = make_float4(o[0].hi, o[0].lo, o[1].hi, o[1].lo);
        } else {
          d[0] = to2(o[0]);
          if (in1) d[1] = to2(o[1]);
        }
      }
      for (int q = 0; q < (p_terms ? in1 ? 2 : 1 : 0); ++q) {
        const int e = k * nxy + col + q;
        ff w = p_terms == 1 ? of2(A.p[e]) : ff{0.f, 0.f};
        for (int s = 4 - p_terms; s < 4; ++s) w = ff_add_f(w, omega * __ldg(A.phi[s] + e));
        A.p[e] = to2(w);
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) vzp[q] = vz[q];
    fz[0] = cur.f[0];
    fz[1] = cur.f[1];
  };
  Plane<TB> P0, P1;
  load(k0, P0);
  for (int k = k0; k <= k1; k += 2) {
    step(k, P0, P1);
    if (k < k1) step(k + 1, P1, P0);
  }
}

// Stop test of the SIMPLE loop (Section 3: until ||phi|| < eps, read as
// ||phi_k||_inf <= eps ||phi_1||_inf; plus the round-off floor and the pass
// cap); sets the condition of the graph's WHILE node.
__device__ void decide(const PassArgs& A, float a, float d) {
  LoopState* ls = A.ls;
  const int pass = ls->pass + 1;
  ls->pass = pass;
  if (pass == 1) ls->phi1 = a;
  const float prev = ls->phi_last;
  ls->phi_prev = prev;
  ls->phi_last = a;
  ls->div_last = d;
  const float phi1 = ls->phi1;
  int go = 1;
  if (*A.fault) { ls->status = 4; go = 0; }   // a pressure transform's wait gave up
  else if (isinf(a) || isinf(d) || isnan(a) || isnan(d)) { ls->nan = 1; ls->status = 3; go = 0; }
  else if (a == 0.f || a <= A.cb->eps * phi1) { ls->status = 1; go = 0; }
  else if (pass >= 3 && a > 0.25f * prev && a <= 1e-9f * phi1) { ls->status = 1; go = 0; }
  else if (pass >= A.cb->max_pass) { ls->status = 2; go = 0; }
  if (A.set_handle) cudaGraphSetConditional(A.h, go ? 1u : 0u);
}

// A loop that ended before the pass leaves it at once.  FIRST: the first pass of
// the mixed form, whose predictor is float32.
template <bool FF, bool FIRST, bool VEC>
__global__ void __launch_bounds__(kPassThreads, 2) k_pass(PassArgs A) {
  __shared__ __align__(16) float2 sh[6 * kPassThreads];
  __shared__ float red[32];
  __shared__ unsigned last;
  tc5::pdl_trigger();   // the pressure transform that follows may start its set-up
  if (A.decide && A.ls->status != 0) return;   // ended before this pass
  float aphi = 0.f, adiv = 0.f;
  const int done = A.idx < 3 ? A.idx : A.ls->pass;
  const float2* vin = A.vff[(done + 1) & 1];
  float2* vout = A.vff[done & 1];
  const int p_terms = A.idx < 3 ? 0 : done == 3 ? 4 : 1;
  if constexpr (FIRST) pass_body<FF, float, VEC>(A, A.w32, A.phi[0], vout, p_terms, aphi, adiv, sh);
  else pass_body<FF, float2, VEC>(A, vin, A.phi[A.idx], vout, p_terms, aphi, adiv, sh);
  aphi = block_max(aphi, red);
  adiv = block_max(adiv, red);
  if (!A.decide) return;
  const int nb = gridDim.x * gridDim.y * gridDim.z;
  const int b = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (threadIdx.x == 0) {
    __stcg(A.part + b, aphi);
    __stcg(A.part + nb + b, adiv);
    __threadfence();
    last = atomicAdd(&A.ls->ticket, 1u);
  }
  __syncthreads();
  if (last != (unsigned)nb - 1) return;
  __threadfence();
  float a = 0.f, d = 0.f;
  for (int q = threadIdx.x; q < nb; q += blockDim.x) {
    a = fmaxf(a, __ldcg(A.part + q));
    d = fmaxf(d, __ldcg(A.part + nb + q));
  }
  a = block_max(a, red);
  d = block_max(d, red);
  if (threadIdx.x == 0) {
    A.ls->ticket = 0;
    decide(A, a, d);
  }
}

struct JoinArgs {
  int n[3];
  const float2* vff[2];
  const float* phi[3];
  const float2* p;
  const CallBlock* cb;
  LoopState* ls;
  int kz;                  // planes per thread
};

// out = v - sigma x, p_out = p (float64): the last v; p from the corrections, or
// from where the fourth and later passes have summed them
__global__ void __launch_bounds__(kCellThreads) k_join(JoinArgs A) {
  const int pass = A.ls->pass;
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && A.ls->status > A.ls->worst)
    A.ls->worst = A.ls->status;
  const double* x = A.cb->x;
  double* out = A.cb->out;
  double* pout = A.cb->p;
  const float sigma = A.cb->sigma, omega = A.cb->omega;
  const int nxy = A.n[0] * A.n[1], nz = A.n[2], nc = nxy * nz;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nxy) return;
  const float2* v = pass & 1 ? A.vff[0] : A.vff[1];
#pragma unroll 1
  for (int k = blockIdx.y * A.kz; k < min(nz, (int)(blockIdx.y + 1) * A.kz); ++k) {
    const int e = k * nxy + t;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ff a = of2(__ldg(v + c * nc + e));
      if (sigma != 0.f) a = ff_sub(a, ff_mul_f(f64_split(__ldg(x + c * nc + e)), sigma));
      out[c * nc + e] = ff_join(a.hi, a.lo);
    }
    if (pout) {
      ff q = {0.f, 0.f};
      if (pass > 3) q = of2(A.p[e]);
#pragma unroll
      for (int s = 0; s < 3; ++s)
        if (s < pass && pass <= 3) q = ff_add_f(q, omega * __ldg(A.phi[s] + e));
      pout[e] = ff_join(q.hi, q.lo);
    }
  }
}

template <bool FF, bool FIRST, bool VEC>
fv_status run_pass_v(const PassArgs& A0, cudaStream_t s) {
  PassArgs A = A0;
  static int per_sm = 0;       // residency of the kernel, the same for every grid
  if (!per_sm) {
    int q = 0;
    FV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, k_pass<FF, FIRST, VEC>, kPassThreads, 0));
    per_sm = q < 1 ? 1 : q;
  }
  // tiles of at most 64 cells along x that split it evenly; rows per tile and
  // planes per chunk such that one wave of resident blocks covers the grid and
  // the busiest SM computes the fewest thread planes (halo row, and the chunk's
  // extra z-face at 0.6 of a plane, included)
  const int* n = A.m.n;
  const int ntx = (n[0] + 63) / 64;
  A.tx = ((n[0] + ntx - 1) / ntx + 1) / 2 * 2;
  const int LX = A.tx / 2 + 1;
  double best = 1e300;
  int nty = 1;
  for (int ty = kPassThreads / LX - 1; ty >= 1; --ty) {
    const int rows = (n[1] + ty - 1) / ty, t = (n[1] + rows - 1) / rows;
    int chunks = 152 * per_sm / (ntx * rows);
    chunks = chunks < 1 ? 1 : chunks > n[2] ? n[2] : chunks;
    const int kz = (n[2] + chunks - 1) / chunks;
    const int64_t blocks = (int64_t)ntx * rows * ((n[2] + kz - 1) / kz);
    const double cost = (double)((blocks + 151) / 152) * (kz + 0.6) * LX * (t + 1);
    if (cost < best) {
      best = cost;
      nty = rows;
      A.ty = t;
      A.kz = kz;
    }
  }
  const dim3 grid(ntx, nty, (n[2] + A.kz - 1) / A.kz);
  const int thr = (LX * (A.ty + 1) + 31) / 32 * 32;
  k_pass<FF, FIRST, VEC><<<grid, thr, 0, s>>>(A);
  FV_CHECK_LAUNCH();
  return FV_OK;
}

template <bool FF, bool FIRST>
fv_status run_pass(const PassArgs& A, cudaStream_t s) {
  return A.m.n[0] % 2 == 0 ? run_pass_v<FF, FIRST, true>(A, s) : run_pass_v<FF, FIRST, false>(A, s);
}

}  // namespace

fv_status launch_pass(const fv_grid* g, int prec, int idx, const CallBlock* cb, LoopState* ls,
                      const cudaGraphConditionalHandle* h, bool decide) {
  PassArgs A = {};
  A.m = g->met_ff;
  A.w32 = g->w32;
  A.vff[0] = g->vff[0];
  A.vff[1] = g->vff[1];
  for (int s = 0; s < 4; ++s) A.phi[s] = g->phis[s];
  A.p = g->pff;
  A.r = g->r32;
  A.cb = cb;
  A.ls = ls;
  A.part = (float*)g->d_part;
  A.fault = g->d_fault;
  if (h) A.h = *h;
  A.set_handle = h ? 1 : 0;
  A.decide = decide ? 1 : 0;
  LaunchScope ls_(g, FV_K_CORRECT);
  A.idx = idx;
  if (prec == FV_FF) return run_pass<true, false>(A, g->stream);
  if (idx == 0) return run_pass<false, true>(A, g->stream);
  return run_pass<false, false>(A, g->stream);
}

fv_status launch_join(const fv_grid* g, const CallBlock* cb, LoopState* ls) {
  JoinArgs A;
  for (int d = 0; d < 3; ++d) {
    A.n[d] = g->n[d];
    A.phi[d] = g->phis[d];
  }
  A.vff[0] = g->vff[0];
  A.vff[1] = g->vff[1];
  A.p = g->pff;
  A.cb = cb;
  A.ls = ls;
  A.kz = cell_planes(g);
  LaunchScope ls_(g, FV_K_VECTOR);
  k_join<<<cell_grid_fit(g), cell_threads(g), 0, g->stream>>>(A);
  FV_CHECK_LAUNCH();
  return FV_OK;
}

}  // namespace fv
