// The SIMPLE passes of the evaluation graphs (Section 3, the algorithm after
// Eq. 10), compiled without FMA contraction so that every TwoSum and TwoProd
// keeps its rounding.
//
// A pass takes the new correction phi_m, forms the corrected velocity
// v = w - omega G (phi_1 + ... + phi_m) and its divergence r = D v, the
// right-hand side of the next solve.  v is not stored between the first three
// passes (three is the usual number): the predictor w and the float32
// corrections phi_1 .. phi_3 hold it exactly, so pass m reads w (12 B per cell
// in float32, 24 B in float-float) and 4 m B of corrections and writes 4 B,
// instead of reading and writing the float-float v and p (72 B).  The result
// is formed once, by k_join, from the same terms in the same order.  Passes
// beyond the third (slow inner solves, under-relaxation) store v: the fourth
// folds w and all four corrections into a float-float buffer, later ones read
// it and write the other.
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
// Bound by instruction issue (float-float arithmetic: about 290 instructions
// per cell in the third float-float pass), not by memory.  Measured (cold
// cache): the three passes at 100^3 mixed 15, 17 and 20 us against 23-27 us
// each for the kernel that stored v and p; at 256^3 float-float 171, 240 and
// 242 us against 355 us.  One cell per thread took 390 instructions and 18 us
// for the second mixed pass at 100^3 (14 us with two); fetching the low
// neighbours a plane ahead as well cost registers and 20 % of the float-float
// time.
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

// v at a face: base - omega sum_s (a_s - b_s) / dc, the corrections a (this
// cell) and b (low neighbour) in order.
// Mixed form: each gradient in float32, as the form's contract has it.
template <int NS>
__device__ __forceinline__ ff face_mixed(ff v, const float (&a)[NS], const float (&b)[NS], float idc,
                                         float omega) {
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const float g = (a[s] - b[s]) * idc;
    v = ff_add_f(v, -omega * g);
  }
  return v;
}

// Float-float form: the differences of float32 values are exact sums of two
// floats; they are added (|phi| falls by ~1e-6 per pass, so one TwoSum per
// step keeps ~2^-48 of the first), then one product with omega / dc and one
// subtraction: with the full TwoSum of both parts where v is returned, stored
// or decides the last correction (ACC), else with the lower parts added in
// float32.
template <int NS, bool ACC>
__device__ __forceinline__ ff face_ff(ff v, const float (&a)[NS], const float (&b)[NS], float2 idc) {
  ff d = two_sum(a[0], -b[0]);
#pragma unroll
  for (int s = 1; s < NS; ++s) {
    const ff t = two_sum(a[s], -b[s]);
    const ff u = two_sum(d.hi, t.hi);
    d = {u.hi, u.lo + (d.lo + t.lo)};
  }
  ff g;
  g.hi = d.hi * idc.x;
  g.lo = fma_f(d.hi, idc.x, -g.hi);
  g.lo = fma_f(d.hi, idc.y, g.lo);
  g.lo = fma_f(d.lo, idc.x, g.lo);
  if (ACC) return ff_sub(v, fast_two_sum(g.hi, g.lo));
  const ff u = two_sum(v.hi, -g.hi);
  return {u.hi, u.lo + (v.lo - g.lo)};     // |lo| may exceed half an ulp of hi
}

// one direction of the divergence: (hi - lo) / dx as an unevaluated sum
template <bool ACC>
__device__ __forceinline__ ff div_term(ff h, ff l, float2 idx) {
  if (ACC) return ff_mul(ff_sub(h, l), of2(idx));
  const ff d = two_sum(h.hi, -l.hi);
  const float e = d.lo + (h.lo - l.lo);
  ff p;
  p.hi = d.hi * idx.x;
  p.lo = fma_f(d.hi, idx.x, -p.hi);
  p.lo = fma_f(d.hi, idx.y, p.lo);
  p.lo = fma_f(e, idx.x, p.lo);
  return p;
}

// the three directions added and rounded to float32
template <bool ACC>
__device__ __forceinline__ float div_sum(ff x, ff y, ff z) {
  if (ACC) return ff_add(ff_add(x, y), z).hi;
  const ff u = two_sum(x.hi, y.hi), w = two_sum(u.hi, z.hi);
  return w.hi + (w.lo + u.lo + (x.lo + y.lo + z.lo));
}

struct PassArgs {
  MetFF m;
  const float* w32;            // mixed: the predictor
  float2* vff[2];              // float-float: the predictor in vff[1]; folded states
  const float* phi[4];
  float2* p;
  float* r;
  const CallBlock* cb;
  LoopState* ls;
  float* part;
  const unsigned* fault;
  cudaGraphConditionalHandle h;
  int set_handle, decide;
  int tx, ty, kz;
};

// omega / dc of the float-float form
__device__ __forceinline__ float2 scaled(float2 idc, float omega) {
  return omega == 1.f ? idc : to2(ff_mul_f(of2(idc), omega));
}

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
template <int NS, typename TB>
struct Plane {
  float f[NS][2];
  TB b[3][2];
};

// One pass over the tile: base stored as TB, NS corrections (the last one
// new); FOLD: v goes to vout and p to m.p; VEC: nx is even, pairs are aligned.
// Updates this thread's maxima of |phi| (new) and |D v|.  Loads are not
// predicated: indices are clamped to the grid, and what a wall or a thread
// beyond the grid loads that way is not used.
template <bool FF, int NS, typename TB, bool FOLD, bool VEC>
__device__ __forceinline__ void pass_body(const PassArgs& A, const TB* __restrict__ base,
                                          const float* const (&phi)[NS], float2* __restrict__ vout,
                                          bool p_first, float& aphi, float& adiv, float2* sh) {
  // The right-hand side of the usual last solve (the second pass's, or any after
  // the third) limits how divergence-free the float-float result is: it is
  // summed in full; the first one's rounding is removed by the next pass.
  constexpr bool ACC = FF && (NS == 2 || FOLD);
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
  auto load = [&](int k, Plane<NS, TB>& P) {
    const int e = min(k, nz - 1) * nxy + col;
#pragma unroll
    for (int s = 0; s < NS; ++s) load2<VEC>(phi[s] + e, d1, P.f[s]);
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
        if (FF) cxf[q] = scaled(m.idcf[0][i + q], omega);
        else cx[q] = m.idc[0][i + q];
        dxi[q] = m.idx[0][i + q];
      }
    if (FF) cyf = scaled(m.idcf[1][j], omega);
    else cy = m.idc[1][j];
    dyi = m.idx[1][j];
  }
  auto face = [&](ff b, const float (&a)[NS], const float (&c)[NS], float idc, float2 idcf) -> ff {
    if constexpr (FF) return face_ff<NS, ACC>(b, a, c, idcf);
    else return face_mixed<NS>(b, a, c, idc, omega);
  };
  float fz[NS][2];             // the corrections of the plane below
#pragma unroll
  for (int s = 0; s < NS; ++s) load2<VEC>(phi[s] + max(k0 - 1, 0) * nxy + col, d1, fz[s]);
  ff px[2] = {}, py[2] = {}, vzp[2] = {};    // of the plane whose z-face above is awaited
  const ff zero = {0.f, 0.f};
  // plane k (in cur; k + 1 is fetched into nxt)
  auto step = [&](int k, Plane<NS, TB>& cur, Plane<NS, TB>& nxt) {
    // the low neighbours of this plane: fetched one plane ago as other threads'
    // own cells, so near; the next plane itself: far, a plane ahead
    float fx[NS], fy[NS][2];
    {
      const int e = min(k, nz - 1) * nxy + col;
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        fx[s] = __ldg(phi[s] + (e - dx));
        load2<VEC>(phi[s] + (e - dy), d1, fy[s]);
      }
    }
    if (k < k1) load(k + 1, nxt);
    float a0[NS], a1[NS], c0[NS], c1[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) { a0[s] = cur.f[s][0]; a1[s] = cur.f[s][1]; }
    // low z-faces of plane k, which close plane k - 1
    ff vz[2] = {zero, zero};
    if (k > 0 && k < nz) {
#pragma unroll
      for (int s = 0; s < NS; ++s) { c0[s] = fz[s][0]; c1[s] = fz[s][1]; }
      const float zc = FF ? 0.f : m.idc[2][k];
      const float2 zcf = FF ? scaled(m.idcf[2][k], omega) : make_float2(0.f, 0.f);
      vz[0] = face(base_of(cur.b[2][0]), a0, c0, zc, zcf);
      vz[1] = face(base_of(cur.b[2][1]), a1, c1, zc, zcf);
    }
    if (k > k0 && own) {
      const float2 dz = m.idx[2][k - 1];
      float d[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        d[q] = div_sum<ACC>(px[q], py[q], div_term<ACC>(vz[q], vzp[q], dz));
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
#pragma unroll
    for (int s = 0; s < NS; ++s) c0[s] = fx[s];
    vx[0] = face(base_of(cur.b[0][0]), a0, c0, cx[0], cxf[0]);
    if (dx == 0) vx[0] = zero;
    vx[1] = face(base_of(cur.b[0][1]), a1, a0, cx[1], cxf[1]);
#pragma unroll
    for (int s = 0; s < NS; ++s) { c0[s] = fy[s][0]; c1[s] = fy[s][1]; }
    vy[0] = face(base_of(cur.b[1][0]), a0, c0, cy, cyf);
    vy[1] = face(base_of(cur.b[1][1]), a1, c1, cy, cyf);
    if (dy == 0) vy[0] = vy[1] = zero;
    float2* sx = sh + (k & 1) * 3 * kPassThreads;
    float4* sy = reinterpret_cast<float4*>(sx + kPassThreads);
    sx[tid] = to2(vx[0]);
    sy[tid] = make_float4(vy[0].hi, vy[0].lo, vy[1].hi, vy[1].lo);
    __syncthreads();
    if (own) {
      const ff x2 = i + 2 < nx ? of2(sx[tid + 1]) : zero;
      const float4 y2 = j + 1 < ny ? sy[tid + LX] : make_float4(0.f, 0.f, 0.f, 0.f);
      px[0] = div_term<ACC>(VEC || in1 ? vx[1] : zero, vx[0], dxi[0]);
      px[1] = div_term<ACC>(x2, vx[1], dxi[1]);
      py[0] = div_term<ACC>({y2.x, y2.y}, vy[0], dyi);
      py[1] = div_term<ACC>({y2.z, y2.w}, vy[1], dyi);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float u = fabsf(cur.f[NS - 1][q]);           // (beyond an odd row: the first cell again)
        if (!(u <= 3e38f)) u = __int_as_float(0x7f800000);
        aphi = fmaxf(aphi, u);
      }
      if (FOLD) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          if (q == 1 && !in1) break;
          const int e = k * nxy + col + q;
          const ff o[3] = {vx[q], vy[q], vz[q]};
#pragma unroll
          for (int c = 0; c < 3; ++c)
            vout[c * nc + e] = to2(o[c]);
          ff w = p_first ? ff{omega * cur.f[0][q], 0.f} : ff_add_f(of2(A.p[e]), omega * cur.f[0][q]);
#pragma unroll
          for (int s = 1; s < NS; ++s) w = ff_add_f(w, omega * cur.f[s][q]);
          A.p[e] = to2(w);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) vzp[q] = vz[q];
#pragma unroll
    for (int s = 0; s < NS; ++s) { fz[s][0] = cur.f[s][0]; fz[s][1] = cur.f[s][1]; }
  };
  Plane<NS, TB> P0, P1;
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

// IDX 0, 1, 2: the first three passes (a loop that ended earlier leaves them
// at once); 3: any later one.
template <bool FF, int IDX, bool VEC>
__global__ void __launch_bounds__(kPassThreads, 2) k_pass(PassArgs A) {
  __shared__ __align__(16) float2 sh[6 * kPassThreads];
  __shared__ float red[32];
  __shared__ unsigned last;
  tc5::pdl_trigger();   // the pressure transform that follows may start its set-up
  if (A.decide && A.ls->status != 0) return;   // ended before this pass
  float aphi = 0.f, adiv = 0.f;
  if constexpr (IDX < 3) {
    const float* phi[IDX + 1];
#pragma unroll
    for (int s = 0; s <= IDX; ++s) phi[s] = A.phi[s];
    if constexpr (FF) pass_body<true, IDX + 1, float2, false, VEC>(A, A.vff[1], phi, nullptr, true, aphi, adiv, sh);
    else pass_body<false, IDX + 1, float, false, VEC>(A, A.w32, phi, nullptr, true, aphi, adiv, sh);
  } else {
    const int done = A.ls->pass;               // the result of fold f is in vff[f & 1], f = pass - 3
    if (done == 3) {
      const float* phi[4] = {A.phi[0], A.phi[1], A.phi[2], A.phi[3]};
      if constexpr (FF) pass_body<true, 4, float2, true, VEC>(A, A.vff[1], phi, A.vff[0], true, aphi, adiv, sh);
      else pass_body<false, 4, float, true, VEC>(A, A.w32, phi, A.vff[0], true, aphi, adiv, sh);
    } else {
      const float* phi[1] = {A.phi[3]};
      const bool odd = (done & 1) != 0;
      pass_body<FF, 1, float2, true, VEC>(A, odd ? A.vff[1] : A.vff[0], phi, odd ? A.vff[0] : A.vff[1], false, aphi,
                                     adiv, sh);
    }
  }
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
  MetFF m;
  const float* w32;
  const float2* vff[2];
  const float* phi[3];
  const float2* p;
  const CallBlock* cb;
  LoopState* ls;
  int kz;                  // planes per thread
};

// out = v - sigma x, p_out = p (float64): v and p from the terms that hold them
template <bool FF, int NS>
__device__ __forceinline__ void join_body(const JoinArgs& A) {
  const MetFF& m = A.m;
  const double* x = A.cb->x;
  double* out = A.cb->out;
  double* pout = A.cb->p;
  const float sigma = A.cb->sigma, omega = A.cb->omega;
  const int nx = m.n[0], ny = m.n[1], nz = m.n[2], nc = (int)m.ncell, nxy = nx * ny;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nxy) return;
  const int i = t % nx, j = t / nx;
  const int pos2[2] = {i, j}, st[3] = {1, nx, nxy};
  const int pass = A.ls->pass;
  const float2* v = A.vff[pass & 1];          // NS == 0: the last fold
#pragma unroll 1
  for (int k = blockIdx.y * A.kz; k < min(nz, (int)(blockIdx.y + 1) * A.kz); ++k) {
    const int e = k * nxy + t;
    float f[NS > 0 ? NS : 1];
#pragma unroll
    for (int s = 0; s < NS; ++s) f[s] = __ldg(A.phi[s] + e);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int q = c < 2 ? pos2[c] : k;
      ff a = {0.f, 0.f};
      if (q > 0) {
        if constexpr (NS == 0) {
          a = of2(v[c * nc + e]);
        } else {
          float g[NS];
#pragma unroll
          for (int s = 0; s < NS; ++s) g[s] = __ldg(A.phi[s] + e - st[c]);
          if constexpr (FF) {
            a = face_ff<NS, true>(of2(__ldg(A.vff[1] + c * nc + e)), f, g, scaled(m.idcf[c][q], omega));
          } else {
            a = face_mixed<NS>({__ldg(A.w32 + c * nc + e), 0.f}, f, g, m.idc[c][q], omega);
          }
        }
      }
      if (sigma != 0.f) a = ff_sub(a, ff_mul_f(f64_split(__ldg(x + c * nc + e)), sigma));
      out[c * nc + e] = ff_join(a.hi, a.lo);
    }
    if (pout) {
      ff q;
      if constexpr (NS == 0) {
        q = of2(A.p[e]);
      } else {
        q = {omega * f[0], 0.f};
#pragma unroll
        for (int s = 1; s < NS; ++s) q = ff_add_f(q, omega * f[s]);
      }
      pout[e] = ff_join(q.hi, q.lo);
    }
  }
}

template <bool FF>
__global__ void __launch_bounds__(kCellThreads) k_join(JoinArgs A) {
  const int pass = A.ls->pass;
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && A.ls->status > A.ls->worst)
    A.ls->worst = A.ls->status;
  if (pass == 3) join_body<FF, 3>(A);
  else if (pass == 2) join_body<FF, 2>(A);
  else if (pass == 1) join_body<FF, 1>(A);
  else join_body<FF, 0>(A);
}

template <bool FF, int IDX, bool VEC>
fv_status run_pass_v(const PassArgs& A0, cudaStream_t s) {
  PassArgs A = A0;
  static int per_sm = 0;       // residency of the kernel, the same for every grid
  if (!per_sm) {
    int q = 0;
    FV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, k_pass<FF, IDX, VEC>, kPassThreads, 0));
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
  k_pass<FF, IDX, VEC><<<grid, thr, 0, s>>>(A);
  FV_CHECK_LAUNCH();
  return FV_OK;
}

template <bool FF, int IDX>
fv_status run_pass(const PassArgs& A, cudaStream_t s) {
  return A.m.n[0] % 2 == 0 ? run_pass_v<FF, IDX, true>(A, s) : run_pass_v<FF, IDX, false>(A, s);
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
  if (prec == FV_FF) {
    if (idx == 0) return run_pass<true, 0>(A, g->stream);
    if (idx == 1) return run_pass<true, 1>(A, g->stream);
    if (idx == 2) return run_pass<true, 2>(A, g->stream);
    return run_pass<true, 3>(A, g->stream);
  }
  if (idx == 0) return run_pass<false, 0>(A, g->stream);
  if (idx == 1) return run_pass<false, 1>(A, g->stream);
  if (idx == 2) return run_pass<false, 2>(A, g->stream);
  return run_pass<false, 3>(A, g->stream);
}

fv_status launch_join(const fv_grid* g, int prec, const CallBlock* cb, LoopState* ls) {
  JoinArgs A;
  A.m = g->met_ff;
  A.w32 = g->w32;
  A.vff[0] = g->vff[0];
  A.vff[1] = g->vff[1];
  for (int s = 0; s < 3; ++s) A.phi[s] = g->phis[s];
  A.p = g->pff;
  A.cb = cb;
  A.ls = ls;
  A.kz = cell_planes(g);
  const int thr = cell_threads(g);
  LaunchScope ls_(g, FV_K_VECTOR);
  if (prec == FV_FF) k_join<true><<<cell_grid_fit(g), thr, 0, g->stream>>>(A);
  else k_join<false><<<cell_grid_fit(g), thr, 0, g->stream>>>(A);
  FV_CHECK_LAUNCH();
  return FV_OK;
}

}  // namespace fv
