// Multigrid solve of the pressure-correction equation (Section 3, step 1 of
// the SIMPLE-like loop: D G phi = r with d phi / dn = 0 on the walls).
//
// The equation is solved in its symmetric form A phi = b with
//   (A phi)_P = sum over the faces f of P of  a_f (phi_P - phi_nb(f)),
//   a_f = (area of f) / (distance between the centres across f),
//   b = -V (r - c),  c = sum(V r) / sum(V),
// V the cell volumes: A = -V D G on the stretched grid, b the right-hand side
// made compatible with the Neumann null space the way the tensor-product
// solve makes it (its null mode is the constant), and the solution is
// returned with zero volume-weighted mean, so both solvers return the same
// phi.
//
// Outer iteration: flexible conjugate gradients in float64 (Polak-Ribiere
// beta, which tolerates the rounding of a float32 preconditioner), stopped at
// ||b - A phi||_2 <= rtol ||b||_2.  Preconditioner: one float32 V-cycle.
//
// Hierarchy: full coarsening of every axis with more than two cells (coarse
// cell I = fine cells 2I and 2I+1; an odd count leaves a last coarse cell of
// one fine cell), until no axis has more than 32 cells.  Coarse operators
// are rediscretised from the coarse cells' widths and centre distances (the
// same a_f formula).  Prolongation: tensor product of 1-D linear
// interpolation between coarse cell centres in the stretched coordinate,
// constant beyond the first and last centre (the Neumann walls).
// Restriction: its transpose, so the integrated residual is conserved.
// Smoother: zebra line Gauss-Seidel, alternating the line direction -- the
// cosine-stretched grids have cells with aspect ratios of tens, for which
// point smoothers fail and line smoothers do not.  Each half-sweep solves
// every line of one colour (lines coloured like a checkerboard of their two
// transverse indices, so neighbour lines differ in colour) exactly, in place
// (k_line).  Pre-smoothing x, y, z (colours 0, 1) and post-smoothing in the
// exact reverse order, so the V-cycle is a symmetric preconditioner.  The last
// level is solved exactly by the separable eigenbases of its operator (A = sum
// over axes of K_d (x) W_others, K_d E_d = W_d E_d Lambda_d), null mode dropped,
// in place of the levels that coarsening to four cells would still have.
//
// The whole iteration, its stop test included, is one CUDA graph whose WHILE
// node runs the conjugate-gradient steps on the device; the host waits once.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fv_ff.cuh"
#include "fv_internal.cuh"
#include "fv_tc5.cuh"
#include "fvns_host.h"

namespace fv {

namespace {

constexpr int kMgMaxLevels = 16;
constexpr int kCoarseMax = 4;       // coarsening would end with at most this many cells per axis
constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 608;     // 4 x 152: fixed, so the reductions are deterministic

// ------------------------------------------------------------ host tables --
struct Axis1D {
  int n = 0;
  std::vector<double> x;   // faces, n + 1
  std::vector<double> w;   // widths
  std::vector<double> xc;  // centres
  std::vector<double> t;   // n + 1: 1 / (centre distance) at interior faces, 0 at walls
};

Axis1D axis_from_faces(const std::vector<double>& x) {
  Axis1D a;
  a.n = (int)x.size() - 1;
  a.x = x;
  a.w.resize(a.n);
  a.xc.resize(a.n);
  a.t.assign(a.n + 1, 0.0);
  for (int m = 0; m < a.n; ++m) {
    a.w[m] = x[m + 1] - x[m];
    a.xc[m] = 0.5 * (x[m] + x[m + 1]);
  }
  for (int f = 1; f < a.n; ++f) a.t[f] = 1.0 / (a.xc[f] - a.xc[f - 1]);
  return a;
}

// coarse faces: every other fine face, and the last one
Axis1D coarsen(const Axis1D& f) {
  if (f.n <= 2) return f;
  const int nc = (f.n + 1) / 2;
  std::vector<double> X(nc + 1);
  for (int I = 0; I < nc; ++I) X[I] = f.x[2 * I];
  X[nc] = f.x[f.n];
  return axis_from_faces(X);
}

// prolongation from coarse c to fine f along one axis: fine cell m takes
// (1 - w1[m]) x_c[c0[m]] + w1[m] x_c[c0[m] + 1] (w1 = 0 where it is the
// nearest-centre constant); the identity if the axis was not coarsened
void prolongation(const Axis1D& f, const Axis1D& c, std::vector<int>& c0, std::vector<double>& w1) {
  c0.assign(f.n, 0);
  w1.assign(f.n, 0.0);
  if (c.n == f.n) {
    for (int m = 0; m < f.n; ++m) c0[m] = m;
    return;
  }
  for (int m = 0; m < f.n; ++m) {
    const double p = f.xc[m];
    if (p <= c.xc[0]) { c0[m] = 0; continue; }
    if (p >= c.xc[c.n - 1]) { c0[m] = c.n - 1; continue; }
    int I = 0;
    while (I + 1 < c.n && c.xc[I + 1] < p) ++I;
    c0[m] = I;
    w1[m] = (p - c.xc[I]) / (c.xc[I + 1] - c.xc[I]);
  }
}

// restriction = prolongation transposed: coarse index I gathers from at most
// four fine cells (fine index, weight), weight 0 in the unused slots
void restriction(const std::vector<int>& c0, const std::vector<double>& w1, int nc,
                 std::vector<int>& rf, std::vector<double>& rw) {
  rf.assign((size_t)nc * 4, 0);
  rw.assign((size_t)nc * 4, 0.0);
  std::vector<int> cnt(nc, 0);
  auto add = [&](int I, int m, double wt) {
    if (wt == 0.0) return;
    const int q = cnt[I]++;
    rf[(size_t)I * 4 + q] = m;
    rw[(size_t)I * 4 + q] = wt;
  };
  for (int m = 0; m < (int)c0.size(); ++m) {
    add(c0[m], m, 1.0 - w1[m]);
    if (w1[m] != 0.0) add(c0[m] + 1, m, w1[m]);
  }
}

int count_levels(const int n[3]) {
  int m[3] = {n[0], n[1], n[2]};
  int L = 1;
  while (std::max(m[0], std::max(m[1], m[2])) > kCoarseMax && L < kMgMaxLevels) {
    for (int d = 0; d < 3; ++d)
      if (m[d] > 2) m[d] = (m[d] + 1) / 2;
    ++L;
  }
  return L;
}

// ---------------------------------------------------------- device views --
struct LevDev {
  int n[3];
  int64_t ncell;
  const float* w[3];
  const float* t[3];
  const float* ip[3];    // per direction: inverse pivots of the line solves, per cell
  // transfer between this level and the next coarser one
  const int* pc0[3];     // per index of this level
  const float* pw1[3];
  const int* rf[3];      // per index of the coarser level, 4 slots
  const float* rw[3];
};

struct Fine64 {
  int n[3];
  int64_t ncell;
  const double* w[3];
  const double* t[3];
};

struct CoarseDev {
  int n[3];
  const float* E[3];     // n x n row-major, W-orthonormal eigenvectors (columns)
  const float* lam[3];
};

// (3 n_cell < 2^31: 32-bit arithmetic)
__device__ __forceinline__ void cell_ijk(unsigned c, const int n[3], int& i, int& j, int& k) {
  const unsigned r = c / (unsigned)n[0];
  i = (int)(c - r * (unsigned)n[0]);
  k = (int)(r / (unsigned)n[1]);
  j = (int)(r - (unsigned)k * (unsigned)n[1]);
}

// A x at cell (i, j, k), as the sum of the fluxes to its neighbours (t is 0 at
// the walls, where the clamped neighbour is the cell itself)
template <typename T, typename Lv>
__device__ __forceinline__ T apply_at(const Lv& L, const T* __restrict__ x, int i, int j, int k, int c) {
  const int nx = L.n[0], ny = L.n[1], nz = L.n[2], sy = nx, sz = nx * ny;
  const T wx = L.w[0][i], wy = L.w[1][j], wz = L.w[2][k];
  const T xp = x[c];
  const T fx = L.t[0][i] * (xp - x[i > 0 ? c - 1 : c]) + L.t[0][i + 1] * (xp - x[i + 1 < nx ? c + 1 : c]);
  const T fy = L.t[1][j] * (xp - x[j > 0 ? c - sy : c]) + L.t[1][j + 1] * (xp - x[j + 1 < ny ? c + sy : c]);
  const T fz = L.t[2][k] * (xp - x[k > 0 ? c - sz : c]) + L.t[2][k + 1] * (xp - x[k + 1 < nz ? c + sz : c]);
  return wy * wz * fx + wx * (wz * fy + wy * fz);
}

// --------------------------------------------------------- V-cycle kernels --
// the thread's cell of line (a, b) along D at row m, as strides
template <int D>
__device__ __forceinline__ void line_cell(const LevDev& L, int a, int b, int& i0, int& j0, int& k0, int& c00,
                                          int& stride) {
  if (D == 0) { i0 = 0; j0 = a; k0 = b; stride = 1; }
  else if (D == 1) { i0 = a; j0 = 0; k0 = b; stride = L.n[0]; }
  else { i0 = a; j0 = b; k0 = 0; stride = L.n[0] * L.n[1]; }
  c00 = (k0 * L.n[1] + j0) * L.n[0] + i0;
}

// rows of a line eliminated from its low end; the others from its high end
__host__ __device__ inline int low_rows(int nl) { return (nl + 1) / 2; }

// Inverse pivots of the tridiagonal matrices of all lines along D, eliminated
// from both ends towards the middle: 1 / (diag_m - lo_m^2 ip_{m-1}) below it,
// 1 / (diag_m - up_m^2 ip_{m+1}) above, one thread per line; once per hierarchy.
template <int D>
__global__ void k_pivots(LevDev L, float* __restrict__ ip) {
  const int na = D == 0 ? L.n[1] : L.n[0], nb = D == 2 ? L.n[1] : L.n[2];
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= na * nb) return;
  int i0, j0, k0, c00, stride;
  line_cell<D>(L, t % na, t / na, i0, j0, k0, c00, stride);
  const float wa = D == 0 ? L.w[1][j0] : L.w[0][i0], wb = D == 2 ? L.w[1][j0] : L.w[2][k0];
  const float cross = wa * wb;
  const int nl = L.n[D], h = low_rows(nl);
  float q = 0.f;
  for (int s = 0; s < nl; ++s) {
    if (s == h) q = 0.f;
    const int m = s < h ? s : nl - 1 - (s - h);
    const int i = D == 0 ? m : i0, j = D == 1 ? m : j0, k = D == 2 ? m : k0;
    const float wx = L.w[0][i], wy = L.w[1][j], wz = L.w[2][k];
    const float dg = wy * wz * L.t[0][i] + wy * wz * L.t[0][i + 1] + wx * wz * L.t[1][j] +
                     wx * wz * L.t[1][j + 1] + wx * wy * L.t[2][k] + wx * wy * L.t[2][k + 1];
    const float o = cross * L.t[D][s < h ? m : m + 1];
    q = 1.f / (dg - o * o * q);
    ip[c00 + m * stride] = q;
  }
}

// The recurrences of the lines of a block, by one warp: lanes l and l + 16 own
// line l, eliminate it from its low and its high end, solve the two rows where
// they meet together and substitute back outwards, so a chain is nl and not
// 2 nl multiply-adds long.  S (residual times inverse pivot, entry m at
// m pitch) becomes the solution; Q the inverse pivots, cross the product of
// the two widths across the line (off-diagonals -cross t).
__device__ __forceinline__ void solve_line(float* S, const float* Q, int pitch, int nl, float cross,
                                           const float* __restrict__ t, bool high) {
  const int h = low_rows(nl), count = high ? nl - h : h;
  const int m0 = high ? nl - 1 : 0, dm = high ? -1 : 1;
  const float* ti = t + (high ? 1 : 0);          // coupling towards the end the row is eliminated from
  const float* to = t + (high ? 0 : 1);          // and towards the middle
  float d = 0.f;
#pragma unroll 8
  for (int q = 0; q < count; ++q) {
    const int m = m0 + dm * q;
    d = fmaf(cross * __ldg(ti + m) * Q[m * pitch], d, S[m * pitch]);
    S[m * pitch] = d;
  }
  const int ml = m0 + dm * (count - 1);
  const float al = cross * __ldg(t + h) * Q[ml * pitch];
  const float d2 = __shfl_xor_sync(0xffffffffu, d, 16), al2 = __shfl_xor_sync(0xffffffffu, al, 16);
  float e = (d + al * d2) / (1.f - al * al2);
  S[ml * pitch] = e;
#pragma unroll 8
  for (int q = count - 2; q >= 0; --q) {
    const int m = m0 + dm * q;
    e = fmaf(cross * __ldg(to + m) * Q[m * pitch], e, S[m * pitch]);
    S[m * pitch] = e;
  }
}

// One half-sweep of zebra line Gauss-Seidel along axis D: every line along
// D of colour `color` (the parity of its two transverse indices' sum) is
// solved exactly for the current values of its neighbour lines, which all
// have the other colour and are not written by this launch:
//   x_line += omega * D_line^-1 (b - A x)_line,
// D_line the tridiagonal part of A along the line.  In place.  Transverse
// indices: a (the faster one: i for y- and z-lines, j for x-lines) and b (k
// for x- and y-lines, j for z-lines); line t has a = 2 (t mod half) + ((b +
// color) & 1).
//
// A block owns 16 lines.  All its threads form the residuals of their cells,
// coalesced, times the inverse pivots, and keep both in shared memory; one
// warp then runs the recurrences (solve_line), one multiply-add of latency per
// row because the pivots do not depend on x and are stored with the hierarchy;
// all threads add the result to x.
// Measured at 100^3 (cold caches): 14-15 us a half-sweep in each direction.  The
// partition method it replaces (each line split over 8 warps, a division per
// row in every chain) took 26-28 us for y- and z-lines and 75 us for x-lines,
// whose threads read whole lines apart; 32 lines and 256 threads per block 23-25
// us (12 % of the warps active).  Three blocks per SM need at most 42 registers:
// at two the 313 blocks of 100^3 take a second wave (20 us).
//
// Sweeps follow one another by programmatic launch.  Each lets its successor in
// only after its own wait: the successor then knows that everything up to two
// kernels back is complete, which is what reading b ahead of its wait needs (on
// the levels below the finest b comes from k_restrict, just before the first
// sweep).  Letting it in at once and reading b after the wait is ordered too,
// but slower, since the successor's blocks arrive before they have anything to
// do: a solve at 100^3 to 1e-12 9.74 ms against 9.12, at 128^3 19.2 against 18.2.
constexpr int kLineThreads = 512, kLines = 16;

template <int D>
__global__ void __launch_bounds__(kLineThreads, 3) k_line(LevDev L, float* __restrict__ x,
                                              const float* __restrict__ b, float omega, int color,
                                              int b_early) {
  extern __shared__ float sm[];
  constexpr int NL = kLines, LP = NL + 1;    // pitch: rows and lines both conflict-free
  const int nx = L.n[0], ny = L.n[1], nz = L.n[2], sy = nx, sz = nx * ny;
  const int nl = L.n[D];
  const int na = D == 0 ? ny : nx, nb = D == 2 ? ny : nz;
  const int ha = (na + 1) >> 1;
  float* S = sm;                             // [nl][LP] residual times inverse pivot, then the solution
  float* Q = sm + nl * LP;                   // [nl][LP] inverse pivots
  __shared__ int sa[NL], sb[NL];             // the block's lines (sa < 0: none)
  const int tid = threadIdx.x;
  if (tid < NL) {
    const int t = blockIdx.x * NL + tid;
    int ta = -1, tb = 0;
    if (t < ha * nb) {
      tb = t / ha;
      ta = 2 * (t - tb * ha) + ((tb + color) & 1);
      if (ta >= na) ta = -1;
    }
    sa[tid] = ta;
    sb[tid] = tb;
  }
  __syncthreads();
  // cells in an order that is coalesced for D: x-lines row by row of one line,
  // the others line by line of one row.  Missing lines load line (0, 0), whose
  // values go nowhere, so that no branch keeps the loads of several cells apart.
  const int total = nl * NL;
  auto cell_of = [&](int e0, int& l, int& m, int& i, int& j, int& k) {
    const int e = min(e0 + tid, total - 1);  // (the last cell possibly by several threads)
    l = D == 0 ? e / nl : e % NL;
    m = D == 0 ? e - l * nl : e / NL;
    int c00, stride;
    line_cell<D>(L, max(sa[l], 0), sb[l], i, j, k, c00, stride);
    if (D == 0) i = m; else if (D == 1) j = m; else k = m;
    return c00 + m * stride;
  };
  // what the previous kernels do not write is fetched while they finish: the
  // pivots, and b unless the predecessor is the kernel that made it
#pragma unroll 4
  for (int e0 = 0; e0 < total; e0 += kLineThreads) {
    int l, m, i, j, k;
    const int c = cell_of(e0, l, m, i, j, k);
    Q[m * LP + l] = __ldg(L.ip[D] + c);
    if (b_early) S[m * LP + l] = b[c];
  }
  tc5::pdl_wait();
  tc5::pdl_trigger();        // not before the wait: see above
  if (!b_early) {
#pragma unroll 4
    for (int e0 = 0; e0 < total; e0 += kLineThreads) {
      int l, m, i, j, k;
      const int c = cell_of(e0, l, m, i, j, k);
      S[m * LP + l] = b[c];
    }
  }
  __syncthreads();     // the last cell's entry is shared
#pragma unroll 4
  for (int e0 = 0; e0 < total; e0 += kLineThreads) {
    if (e0 + tid >= total) break;
    int l, m, i, j, k;
    const int c = cell_of(e0, l, m, i, j, k);
    const float wx = __ldg(L.w[0] + i), wy = __ldg(L.w[1] + j), wz = __ldg(L.w[2] + k);
    const float xp = x[c];
    // fluxes towards the six neighbours (t is 0 at the walls, where the
    // clamped neighbour is the cell itself)
    const float fx = __ldg(L.t[0] + i) * (xp - x[i > 0 ? c - 1 : c]) +
                     __ldg(L.t[0] + i + 1) * (xp - x[i + 1 < nx ? c + 1 : c]);
    const float fy = __ldg(L.t[1] + j) * (xp - x[j > 0 ? c - sy : c]) +
                     __ldg(L.t[1] + j + 1) * (xp - x[j + 1 < ny ? c + sy : c]);
    const float fz = __ldg(L.t[2] + k) * (xp - x[k > 0 ? c - sz : c]) +
                     __ldg(L.t[2] + k + 1) * (xp - x[k + 1 < nz ? c + sz : c]);
    const int o = m * LP + l;
    S[o] = (S[o] - (wy * wz * fx + wx * wz * fy + wx * wy * fz)) * Q[o];
  }
  __syncthreads();
  if (tid < 32) {          // (missing lines hold line (0, 0)'s values)
    const int l = tid & 15;
    int i, j, k, c00, stride;
    line_cell<D>(L, max(sa[l], 0), sb[l], i, j, k, c00, stride);
    const float wa = D == 0 ? L.w[1][j] : L.w[0][i], wb = D == 2 ? L.w[1][j] : L.w[2][k];
    solve_line(S + l, Q + l, LP, nl, wa * wb, L.t[D], tid >= 16);
  }
  __syncthreads();
#pragma unroll 4
  for (int e = tid; e < total; e += kLineThreads) {
    const int l = D == 0 ? e / nl : e % NL, m = D == 0 ? e - l * nl : e / NL;
    const int ta = sa[l], tb = sb[l];
    if (ta < 0) continue;
    int i, j, k, c00, stride;
    line_cell<D>(L, ta, tb, i, j, k, c00, stride);
    const int c = c00 + m * stride;
    x[c] += omega * S[m * LP + l];
  }
}

__global__ void k_resid32(LevDev L, const float* __restrict__ x, const float* __restrict__ b,
                          float* __restrict__ res) {
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < (unsigned)L.ncell; c += gridDim.x * blockDim.x) {
    int i, j, k;
    cell_ijk(c, L.n, i, j, k);
    res[c] = b[c] - apply_at<float>(L, x, i, j, k, c);
  }
}

// (R res) at a coarse cell, R = P^T: four slots per axis (unused ones have
// weight 0 and index 0), all 64 loads at once
__device__ __forceinline__ float restricted(const LevDev& L, const float* res, int I, int J, int K) {
  const int nx = L.n[0], ny = L.n[1];
  const int4 fx = __ldg(reinterpret_cast<const int4*>(L.rf[0]) + I);
  const int4 fy = __ldg(reinterpret_cast<const int4*>(L.rf[1]) + J);
  const int4 fz = __ldg(reinterpret_cast<const int4*>(L.rf[2]) + K);
  const float4 wx = __ldg(reinterpret_cast<const float4*>(L.rw[0]) + I);
  const float4 wy = __ldg(reinterpret_cast<const float4*>(L.rw[1]) + J);
  const float4 wz = __ldg(reinterpret_cast<const float4*>(L.rw[2]) + K);
  const int ky[4] = {fy.x, fy.y, fy.z, fy.w}, kz[4] = {fz.x, fz.y, fz.z, fz.w};
  const float vy[4] = {wy.x, wy.y, wy.z, wy.w}, vz[4] = {wz.x, wz.y, wz.z, wz.w};
  float s = 0.f;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float* row = res + (kz[r] * ny + ky[q]) * nx;
      s += vz[r] * vy[q] * (wx.x * row[fx.x] + wx.y * row[fx.y] + wx.z * row[fx.z] + wx.w * row[fx.w]);
    }
  return s;
}

// bc = R res, per coarse cell; the coarse iterate starts at zero
__global__ void k_restrict(LevDev L, int nc0, int nc1, int nc2, const float* __restrict__ res,
                           float* __restrict__ bc, float* __restrict__ xc) {
  const int nc[3] = {nc0, nc1, nc2};
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < (unsigned)(nc0 * nc1 * nc2);
       c += gridDim.x * blockDim.x) {
    int I, J, K;
    cell_ijk(c, nc, I, J, K);
    const float s = restricted(L, res, I, J, K);
    bc[c] = s;
    xc[c] = 0.f;
  }
}

// (P xc) at a fine cell
__device__ __forceinline__ float prolonged(const LevDev& L, int nc0, int nc1, const float* xc, int i, int j,
                                           int k) {
  const int I = __ldg(L.pc0[0] + i), J = __ldg(L.pc0[1] + j), K = __ldg(L.pc0[2] + k);
  const float a = __ldg(L.pw1[0] + i), b = __ldg(L.pw1[1] + j), g = __ldg(L.pw1[2] + k);
  const int I1 = a != 0.f ? I + 1 : I, J1 = b != 0.f ? J + 1 : J, K1 = g != 0.f ? K + 1 : K;
  auto at = [&](int kk, int jj, int ii) { return xc[(kk * nc1 + jj) * nc0 + ii]; };
  const float v00 = (1.f - a) * at(K, J, I) + a * at(K, J, I1);
  const float v01 = (1.f - a) * at(K, J1, I) + a * at(K, J1, I1);
  const float v10 = (1.f - a) * at(K1, J, I) + a * at(K1, J, I1);
  const float v11 = (1.f - a) * at(K1, J1, I) + a * at(K1, J1, I1);
  return (1.f - g) * ((1.f - b) * v00 + b * v01) + g * ((1.f - b) * v10 + b * v11);
}

// x += P xc, per fine cell
__global__ void k_prolong_add(LevDev L, int nc0, int nc1, const float* __restrict__ xc,
                              float* __restrict__ x) {
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < (unsigned)L.ncell; c += gridDim.x * blockDim.x) {
    int i, j, k;
    cell_ijk(c, L.n, i, j, k);
    x[c] += prolonged(L, nc0, nc1, xc, i, j, k);
  }
}

// Exact solve x = E Lambda^+ E^T b (3-D Kronecker) of the first level whose
// axes have at most 32 cells, in one block and in place in shared memory: six
// passes of dense transforms along the axes, one line per thread, its results
// in registers, the rows of the eigenbasis broadcast four at a time.  It stands
// in for the rest of the hierarchy below that level: as launches, a V-cycle
// over 25^3, 13^3, 7^3 and 4^3 cells took 230 us of launch and chain latency
// (97 us as one block from 13^3 down, with barriers for launches); this takes
// 42 us for 25^3 (cold caches; one SM's multiply-adds alone 11 us) and saves a
// quarter of the iterations (39 -> 29 at 100^3 to 1e-12).
constexpr int kExactMax = 32;          // cells per axis
constexpr int kExactThreads = 1024;

template <int NM>
__global__ void __launch_bounds__(kExactThreads) k_exact(CoarseDev C, const float* __restrict__ b,
                                                         float* __restrict__ x) {
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x;
  tc5::pdl_trigger();
  const int n[3] = {C.n[0], C.n[1], C.n[2]};
  const int px = n[0] | 1;             // odd pitch: x-lines of a warp fall in different banks
  float* E = sm;                       // [axis][forward, inverse][in][out], NM x NM each
  float* a = sm + 6 * NM * NM;
  for (int e = tid; e < 6 * NM * NM; e += kExactThreads) {
    const int ax = e / (2 * NM * NM), inv = e / (NM * NM) & 1, i = e / NM % NM, o = e % NM, m = n[ax];
    E[e] = i < m && o < m ? __ldg(C.E[ax] + (inv ? o * m + i : i * m + o)) : 0.f;
  }
  tc5::pdl_wait();
  const int nc = n[0] * n[1] * n[2];
  for (int c = tid; c < nc; c += kExactThreads) {
    int i, j, k;
    cell_ijk(c, C.n, i, j, k);
    a[(k * n[1] + j) * px + i] = b[c];
  }
  __syncthreads();
#pragma unroll 1
  for (int s = 0; s < 6; ++s) {        // x, y, z forward; z, y, x back
    const int ax = s < 3 ? s : 5 - s;
    const int m = n[ax], la = ax == 0 ? n[1] : n[0], lb = ax == 2 ? n[1] : n[2];
    const float* Es = E + (2 * ax + (s >= 3)) * NM * NM;
    if (tid < la * lb) {
      const int q = tid / la, p = tid - q * la;
      const int stride = ax == 0 ? 1 : ax == 1 ? px : n[1] * px;
      float* line = a + (ax == 0 ? tid * px : ax == 1 ? q * n[1] * px + p : q * px + p);
      float acc[NM];
#pragma unroll
      for (int o = 0; o < NM; ++o) acc[o] = 0.f;
#pragma unroll 2
      for (int i = 0; i < m; ++i) {
        const float v = line[i * stride];
#pragma unroll
        for (int o = 0; o < NM; o += 4) {
          const float4 w = *reinterpret_cast<const float4*>(Es + i * NM + o);
          acc[o] = fmaf(v, w.x, acc[o]);
          acc[o + 1] = fmaf(v, w.y, acc[o + 1]);
          acc[o + 2] = fmaf(v, w.z, acc[o + 2]);
          acc[o + 3] = fmaf(v, w.w, acc[o + 3]);
        }
      }
      if (s == 2) {                    // z forward: p = mode along x, q along y
        const float l2 = __ldg(C.lam[0] + p) + __ldg(C.lam[1] + q);
#pragma unroll
        for (int o = 0; o < NM; ++o) {
          const float l = o < m ? l2 + __ldg(C.lam[2] + o) : 0.f;
          acc[o] = l > 0.f ? acc[o] / l : 0.f;
        }
      }
#pragma unroll
      for (int o = 0; o < NM; ++o)
        if (o < m) line[o * stride] = acc[o];
    }
    __syncthreads();
  }
  for (int c = tid; c < nc; c += kExactThreads) {
    int i, j, k;
    cell_ijk(c, C.n, i, j, k);
    x[c] = a[(k * n[1] + j) * px + i];
  }
}

inline size_t exact_smem(const int n[3], int NM) {
  return sizeof(float) * ((size_t)6 * NM * NM + (size_t)(n[0] | 1) * n[1] * n[2]);
}

// ---------------------------------------------------------- float64 CG part --
// scalar slots of the CG recurrences (device)
enum { S_RHO = 0, S_PQ, S_ALPHA, S_RR, S_RZ, S_RZO, S_BETA, S_VR, S_BB, S_VPHI, S_IT, S_N };

// one solve's arguments, read by the kernels of the iteration graph
struct MgCall {
  double* phi;
  double rtol;
  int max_iter;
};

// partial sums of a reduction and the count of blocks that have delivered
struct Reduce {
  double* part;
  unsigned* ticket;
  double* s;
};

__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w];
  return s;   // valid in thread 0
}

// Sums a (and b) over the grid: every block delivers its partial sums, the
// last one adds them in a fixed order and returns true in its thread 0 with
// the totals in a, b.
template <int NV>
__device__ __forceinline__ bool grid_sum(const Reduce& R, double& a, double& b, double* sh) {
  __shared__ unsigned last;
  const int nb = gridDim.x * gridDim.y, bid = blockIdx.y * gridDim.x + blockIdx.x;
  a = block_sum(a, sh);
  if (NV > 1) b = block_sum(b, sh);
  if (threadIdx.x == 0) {
    __stcg(R.part + NV * bid, a);
    if (NV > 1) __stcg(R.part + NV * bid + 1, b);
    __threadfence();
    last = atomicAdd(R.ticket, 1u);
  }
  __syncthreads();
  if (last != (unsigned)nb - 1) return false;
  __threadfence();
  a = b = 0.0;
  for (int q = threadIdx.x; q < nb; q += blockDim.x) {
    a += __ldcg(R.part + NV * q);
    if (NV > 1) b += __ldcg(R.part + NV * q + 1);
  }
  a = block_sum(a, sh);
  if (NV > 1) b = block_sum(b, sh);
  if (threadIdx.x != 0) return false;
  *R.ticket = 0;
  return true;
}

__device__ __forceinline__ double vol(const Fine64& F, unsigned c) {
  int i, j, k;
  cell_ijk(c, F.n, i, j, k);
  return F.w[0][i] * F.w[1][j] * F.w[2][k];
}

// s[dst] = sum V r
__global__ void k_sum_vr(Fine64 F, const double* __restrict__ r, Reduce R, int dst) {
  __shared__ double sh[32];
  double s = 0.0, u = 0.0;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < (unsigned)F.ncell; c += gridDim.x * blockDim.x)
    s += vol(F, c) * r[c];
  if (grid_sum<1>(R, s, u, sh)) R.s[dst] = s;
}

// b = -V (r - c), c = S_VR / vtot; rcg = b (phi = 0) or b - A phi (guess), its
// float32 copy for the first V-cycle, whose iterate and the previous
// preconditioned residual start at zero; |b|^2 and |rcg|^2
__global__ void k_rhs(Fine64 F, const double* __restrict__ r, double vtot, const double* __restrict__ phi,
                      double* __restrict__ rcg, float* __restrict__ b32, float* __restrict__ x32,
                      float* __restrict__ zo32, Reduce R) {
  __shared__ double sh[32];
  const double cm = R.s[S_VR] / vtot;
  double bb = 0.0, rr = 0.0;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < (unsigned)F.ncell; c += gridDim.x * blockDim.x) {
    const double b = -vol(F, c) * (r[c] - cm);
    bb += b * b;
    double v = b;
    if (phi) {
      int i, j, k;
      cell_ijk(c, F.n, i, j, k);
      v -= apply_at<double>(F, phi, i, j, k, (int)c);
    }
    rr += v * v;
    rcg[c] = v;
    b32[c] = f64_round_f32(v);
    x32[c] = 0.f;
    zo32[c] = 0.f;
  }
  if (grid_sum<2>(R, bb, rr, sh)) {
    R.s[S_BB] = bb;
    R.s[S_RR] = rr;
    R.s[S_RHO] = 0.0;
    R.s[S_IT] = 0.0;
  }
}

// whether another iteration is wanted: ||r|| > rtol ||b||, below the cap, finite
__device__ __forceinline__ bool go_on(const double* s, const MgCall* call) {
  const double rn = sqrt(fmax(s[S_RR], 0.0)), bn = sqrt(s[S_BB]);
  return bn > 0.0 && isfinite(s[S_RR]) && rn > call->rtol * bn && s[S_IT] < call->max_iter;
}

__global__ void k_begin(const double* s, const MgCall* call, cudaGraphConditionalHandle h) {
  cudaGraphSetConditional(h, go_on(s, call) ? 1u : 0u);
}

// r . z and r . z_old of the V-cycle's z = x32, then z_old = z and x32 = 0 (the
// next cycle's start); beta = (r.z - r.z_old) / rho (0 in the first
// iteration), rho = r . z
__global__ void k_dots2(unsigned n, const double* __restrict__ r, float* __restrict__ x32,
                        float* __restrict__ zo32, Reduce R) {
  __shared__ double sh[32];
  double a = 0.0, b = 0.0;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
    const double rc = r[c];
    const float z = x32[c];
    a += rc * f32_to_f64(z);                 // (integer conversions: the FP64 pipe converts at its own slow rate)
    b += rc * f32_to_f64(zo32[c]);
    zo32[c] = z;
    x32[c] = 0.f;
  }
  if (grid_sum<2>(R, a, b, sh)) {
    double* s = R.s;
    s[S_RZ] = a;
    s[S_RZO] = b;
    s[S_BETA] = s[S_RHO] == 0.0 ? 0.0 : (a - b) / s[S_RHO];
    s[S_RHO] = a;
  }
}

// p = z + beta p
__global__ void k_cg_dir(unsigned n, const double* __restrict__ s, const float* __restrict__ z,
                         double* __restrict__ p) {
  const double be = s[S_BETA];
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x)
    p[c] = be == 0.0 ? f32_to_f64(z[c]) : f32_to_f64(z[c]) + be * p[c];
}

// q = A p; alpha = rho / p . q (0 unless positive).  Bound by the FP64 pipe
// (~1 TFLOP/s): a thread marches up a chunk of planes of its column and keeps
// the z-flux of the face above, 16 float64 instructions per cell: 41 us at 100^3
// with cold caches, 47 us for the cell-wise form (28 us are the pipe's).
__global__ void k_apply64(Fine64 F, const double* __restrict__ p, double* __restrict__ q, int kz, Reduce R) {
  __shared__ double sh[32];
  const int nx = F.n[0], ny = F.n[1], nz = F.n[2], nxy = nx * ny;
  const int k0 = blockIdx.y * kz, k1 = min(k0 + kz, nz);
  double acc = 0.0, u = 0.0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nxy; t += gridDim.x * blockDim.x) {
    const int i = t % nx, j = t / nx;
    const double wx = F.w[0][i], wy = F.w[1][j], wxy = wx * wy;
    const double tx0 = F.t[0][i], tx1 = F.t[0][i + 1], ty0 = F.t[1][j], ty1 = F.t[1][j + 1];
    const int dxm = i > 0 ? 1 : 0, dxp = i + 1 < nx ? 1 : 0, dym = j > 0 ? nx : 0, dyp = j + 1 < ny ? nx : 0;
    int c = k0 * nxy + t;
    double pc = p[c];
    double below = k0 > 0 ? F.t[2][k0] * (p[c - nxy] - pc) : 0.0;   // flux out of the plane below, upwards
#pragma unroll 4
    for (int k = k0; k < k1; ++k, c += nxy) {
      const double pn = p[k + 1 < nz ? c + nxy : c];
      const double wz = F.w[2][k];
      const double fx = tx0 * (pc - p[c - dxm]) + tx1 * (pc - p[c + dxp]);
      const double fy = ty0 * (pc - p[c - dym]) + ty1 * (pc - p[c + dyp]);
      const double up = F.t[2][k + 1] * (pc - pn);
      const double v = wz * (wy * fx + wx * fy) + wxy * (up - below);
      q[c] = v;
      acc += pc * v;
      below = up;
      pc = pn;
    }
  }
  if (grid_sum<1>(R, acc, u, sh)) {
    R.s[S_PQ] = acc;
    R.s[S_ALPHA] = acc > 0.0 ? R.s[S_RHO] / acc : 0.0;
  }
}

// phi += alpha p, r -= alpha q (and its float32 copy), |r|^2, the stop test
__global__ void k_cg_step(unsigned n, const double* __restrict__ p, const double* __restrict__ q,
                          const MgCall* __restrict__ call, double* __restrict__ r, float* __restrict__ b32,
                          Reduce R, cudaGraphConditionalHandle h, int set_handle) {
  __shared__ double sh[32];
  const double al = R.s[S_ALPHA];
  double* phi = call->phi;
  double acc = 0.0, u = 0.0;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
    phi[c] += al * p[c];
    const double rv = r[c] - al * q[c];
    r[c] = rv;
    b32[c] = f64_round_f32(rv);
    acc += rv * rv;
  }
  if (grid_sum<1>(R, acc, u, sh)) {
    R.s[S_RR] = acc;
    R.s[S_IT] += 1.0;
    if (set_handle) cudaGraphSetConditional(h, go_on(R.s, call) ? 1u : 0u);
  }
}

// phi -= S_VPHI / vtot
__global__ void k_sub_mean(unsigned n, const double* __restrict__ s, double vtot, double* __restrict__ phi) {
  const double m = s[S_VPHI] / vtot;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) phi[c] -= m;
}

// ------------------------------------------------------------- the state --
struct MgLevelHost {
  Axis1D ax[3];
  LevDev dev;
  float* x = nullptr;
  float* b = nullptr;
  float* res = nullptr;
  float* ip[3] = {nullptr, nullptr, nullptr};
};

}  // namespace

struct MgState {
  int levels = 0;             // grids that the coarsening has
  int exact = 0;              // the one that k_exact solves, the last that is built
  MgLevelHost lev[kMgMaxLevels];
  Fine64 fine;
  CoarseDev coarse;
  double vtot = 0.0;
  void* d_tab = nullptr;      // 1-D tables of all levels (floats, ints, doubles)
  void* d_work = nullptr;     // level arrays
  double* r = nullptr;        // CG vectors (float64, n_cell each)
  double* p = nullptr;
  double* q = nullptr;
  float* zo = nullptr;        // the previous preconditioned residual
  Reduce red = {};            // 2 x kRedBlocks partials, S_N scalars
  MgCall* call = nullptr;     // device copy of the running solve's arguments
  struct Host {               // pinned
    double s[S_N];
    MgCall call;
  }* h = nullptr;
  // the captured iteration for (nu, omega)
  int nu = 0;
  float omega = 0.f;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
};

namespace {

constexpr size_t kLineSmemMax = 200 * 1024;

int blocks_for(int64_t n, int t = 256) {
  int64_t b = (n + t - 1) / t;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, 4 * 152 * 4));
}

fv_status build_mg(fv_grid* g) {
  MgState* M = new MgState();
  g->mg = M;
  const int n0[3] = {g->n[0], g->n[1], g->n[2]};
  M->levels = count_levels(n0);
  for (int d = 0; d < 3; ++d) M->lev[0].ax[d] = axis_from_faces(g->h_x[d]);
  // down to the exactly solved level; those below it are never visited
  auto longest = [&](const MgLevelHost& H) { return std::max(H.ax[0].n, std::max(H.ax[1].n, H.ax[2].n)); };
  for (M->exact = 0; longest(M->lev[M->exact]) > kExactMax; ++M->exact)
    for (int d = 0; d < 3; ++d) M->lev[M->exact + 1].ax[d] = coarsen(M->lev[M->exact].ax[d]);
  const int lc = M->exact, nlev = lc + 1;
  // table layout: per level and axis w (n), t (n + 1), pw1 (n), rw (4 n_coarse) as
  // floats; pc0 (n), rf (4 n_coarse) as ints; level-0 w, t as doubles; the coarse
  // eigenbases and eigenvalues as floats
  std::vector<float> tf;
  std::vector<int> ti;
  std::vector<double> td;
  struct Off { size_t w, t, pw1, rw, pc0, rf; } off[kMgMaxLevels][3];
  for (int l = 0; l < nlev; ++l) {
    for (int d = 0; d < 3; ++d) {
      const Axis1D& a = M->lev[l].ax[d];
      Off& o = off[l][d];
      o.w = tf.size();
      for (double v : a.w) tf.push_back((float)v);
      o.t = tf.size();
      for (double v : a.t) tf.push_back((float)v);
      if (l < lc) {
        std::vector<int> c0, rf;
        std::vector<double> w1, rw;
        const Axis1D& c = M->lev[l + 1].ax[d];
        prolongation(a, c, c0, w1);
        restriction(c0, w1, c.n, rf, rw);
        o.pw1 = tf.size();
        for (double v : w1) tf.push_back((float)v);
        while (tf.size() % 4) tf.push_back(0.f);   // four slots per coarse cell: one 16-byte load
        while (ti.size() % 4) ti.push_back(0);
        o.rw = tf.size();
        for (double v : rw) tf.push_back((float)v);
        o.rf = ti.size();
        ti.insert(ti.end(), rf.begin(), rf.end());
        o.pc0 = ti.size();
        ti.insert(ti.end(), c0.begin(), c0.end());
      } else {
        o.pw1 = o.rw = o.pc0 = o.rf = 0;
      }
    }
  }
  size_t w64[3], t64[3];
  for (int d = 0; d < 3; ++d) {
    w64[d] = td.size();
    td.insert(td.end(), M->lev[0].ax[d].w.begin(), M->lev[0].ax[d].w.end());
    t64[d] = td.size();
    td.insert(td.end(), M->lev[0].ax[d].t.begin(), M->lev[0].ax[d].t.end());
  }
  // the exactly solved level: W-orthonormal eigenvectors of K_d E = W_d E Lambda
  size_t cE[3], cL[3];
  for (int d = 0; d < 3; ++d) {
    const Axis1D& a = M->lev[lc].ax[d];
    const int n = a.n;
    std::vector<double> dg(n, 0.0), e(n > 1 ? n - 1 : 1, 0.0), lam, Z;
    for (int f = 1; f < n; ++f) {
      dg[f - 1] += a.t[f];
      dg[f] += a.t[f];
      e[f - 1] = -a.t[f] / std::sqrt(a.w[f - 1] * a.w[f]);
    }
    for (int m = 0; m < n; ++m) dg[m] /= a.w[m];
    if (!sym_tridiag_eig(n, dg, e, lam, Z)) {
      set_error("multigrid: coarse eigensolve did not converge");
      return FV_ENOCONV;
    }
    // the null eigenvalue is zero in exact arithmetic: make it so
    int null = 0;
    for (int q = 1; q < n; ++q)
      if (std::fabs(lam[q]) < std::fabs(lam[null])) null = q;
    lam[null] = 0.0;
    cE[d] = tf.size();
    for (int m = 0; m < n; ++m)
      for (int q = 0; q < n; ++q) tf.push_back((float)(Z[(size_t)m * n + q] / std::sqrt(a.w[m])));
    cL[d] = tf.size();
    for (double v : lam) tf.push_back((float)std::max(v, 0.0));
  }
  const size_t bf = tf.size() * 4, bi = ti.size() * 4, bd = td.size() * 8;
  const size_t oi = (bf + 255) / 256 * 256, od = oi + (bi + 255) / 256 * 256;
  FV_CUDA(cudaMalloc(&M->d_tab, od + bd));
  char* base = (char*)M->d_tab;
  FV_CUDA(cudaMemcpy(base, tf.data(), bf, cudaMemcpyHostToDevice));
  if (bi) FV_CUDA(cudaMemcpy(base + oi, ti.data(), bi, cudaMemcpyHostToDevice));
  FV_CUDA(cudaMemcpy(base + od, td.data(), bd, cudaMemcpyHostToDevice));
  const float* F = (const float*)base;
  const int* I = (const int*)(base + oi);
  const double* Dd = (const double*)(base + od);
  // level arrays: x and b, where lines are swept also res and the pivots of three
  // directions
  size_t floats = 0;
  for (int l = 0; l < nlev; ++l) {
    int64_t nc = 1;
    for (int d = 0; d < 3; ++d) nc *= M->lev[l].ax[d].n;
    floats += (size_t)(nc + 63) / 64 * 64 * (l < lc ? 6 : 2);
  }
  FV_CUDA(cudaMalloc(&M->d_work, floats * sizeof(float)));
  float* wp = (float*)M->d_work;
  for (int l = 0; l < nlev; ++l) {
    MgLevelHost& H = M->lev[l];
    LevDev& v = H.dev;
    int64_t nc = 1;
    for (int d = 0; d < 3; ++d) {
      v.n[d] = H.ax[d].n;
      nc *= v.n[d];
      v.w[d] = F + off[l][d].w;
      v.t[d] = F + off[l][d].t;
      const bool has = l < lc;
      v.pw1[d] = has ? F + off[l][d].pw1 : nullptr;
      v.rw[d] = has ? F + off[l][d].rw : nullptr;
      v.pc0[d] = has ? I + off[l][d].pc0 : nullptr;
      v.rf[d] = has ? I + off[l][d].rf : nullptr;
    }
    v.ncell = nc;
    const size_t stride = (size_t)(nc + 63) / 64 * 64;
    H.x = wp; wp += stride;
    H.b = wp; wp += stride;
    if (l == lc) continue;
    H.res = wp; wp += stride;
    for (int d = 0; d < 3; ++d) {
      H.ip[d] = wp;
      v.ip[d] = wp;
      wp += stride;
    }
  }
  for (int d = 0; d < 3; ++d) {
    M->fine.n[d] = g->n[d];
    M->fine.w[d] = Dd + w64[d];
    M->fine.t[d] = Dd + t64[d];
    M->coarse.n[d] = M->lev[lc].ax[d].n;
    M->coarse.E[d] = F + cE[d];
    M->coarse.lam[d] = F + cL[d];
  }
  M->fine.ncell = g->ncell;
  M->vtot = 1.0;
  for (int d = 0; d < 3; ++d) M->vtot *= g->h_x[d].back() - g->h_x[d].front();
  const size_t nb = (size_t)g->ncell * sizeof(double);
  const size_t tail = (2 * kRedBlocks + S_N) * sizeof(double) + 256 + sizeof(MgCall);
  char* cg = nullptr;
  FV_CUDA(cudaMalloc((void**)&cg, 3 * nb + tail + (size_t)g->ncell * sizeof(float)));
  M->r = (double*)cg;
  M->p = M->r + g->ncell;
  M->q = M->p + g->ncell;
  M->red.part = M->q + g->ncell;
  M->red.s = M->red.part + 2 * kRedBlocks;
  M->call = (MgCall*)(M->red.s + S_N);
  M->red.ticket = (unsigned*)((char*)M->call + sizeof(MgCall));
  M->zo = (float*)(cg + 3 * nb + tail);
  FV_CUDA(cudaMemset(M->red.part, 0, tail));
  FV_CUDA(cudaMallocHost((void**)&M->h, sizeof(*M->h)));
  for (int l = 0; l < lc; ++l) {
    const MgLevelHost& H = M->lev[l];
    const LevDev& v = H.dev;
    auto blocks = [](int lines) { return (lines + 127) / 128; };
    k_pivots<0><<<blocks(v.n[1] * v.n[2]), 128, 0, g->stream>>>(v, H.ip[0]);
    k_pivots<1><<<blocks(v.n[0] * v.n[2]), 128, 0, g->stream>>>(v, H.ip[1]);
    k_pivots<2><<<blocks(v.n[0] * v.n[1]), 128, 0, g->stream>>>(v, H.ip[2]);
    FV_CHECK_LAUNCH();
  }
  FV_CUDA(cudaDeviceSynchronize());
  return FV_OK;
}

// shared memory of a line kernel for lines of nl cells
size_t line_smem(int nl) { return sizeof(float) * (size_t)2 * nl * (kLines + 1); }

fv_status set_line_attributes() {
  static bool done = false;
  if (!done) {
    const void* k[3] = {(const void*)k_line<0>, (const void*)k_line<1>, (const void*)k_line<2>};
    for (const void* f : k)
      FV_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLineSmemMax));
    const int n32[3] = {32, 32, 32};
    const void* e[5] = {(const void*)k_exact<16>, (const void*)k_exact<20>, (const void*)k_exact<24>,
                        (const void*)k_exact<28>, (const void*)k_exact<32>};
    for (const void* f : e)
      FV_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)exact_smem(n32, 32)));
    done = true;
  }
  return FV_OK;
}

// a launch, timed under `kind` by the grid's profiler and counted
#define MG_LAUNCH(kind, ...)          \
  do {                                \
    LaunchScope ls_(g, kind);         \
    __VA_ARGS__;                      \
    FV_CHECK_LAUNCH();                \
  } while (0)

fv_status line_sweep(const fv_grid* g, const MgLevelHost& H, int D, int color, float omega, bool b_early,
                     cudaStream_t st) {
  const LevDev& L = H.dev;
  const int na = D == 0 ? L.n[1] : L.n[0], nb = D == 2 ? L.n[1] : L.n[2];
  const int nblk = ((na + 1) / 2 * nb + kLines - 1) / kLines;
  const size_t sm = line_smem(L.n[D]);
  void (*kern)(LevDev, float*, const float*, float, int, int) =
      D == 0 ? k_line<0> : D == 1 ? k_line<1> : k_line<2>;
  LaunchScope ls_(g, FV_K_MG_SMOOTH);
  FV_CUDA(tc5::launch_pdl(kern, dim3(nblk), dim3(kLineThreads), sm, st, L, H.x, (const float*)H.b, omega, color,
                          b_early ? 1 : 0));
  return FV_OK;
}

// one V-cycle on level l: lev[l].b -> lev[l].x (which starts at zero)
fv_status vcycle(const fv_grid* g, MgState* M, int l, int nu, float omega, cudaStream_t st) {
  MgLevelHost& H = M->lev[l];
  const LevDev& L = H.dev;
  if (l == M->exact) {
    const int m = std::max(L.n[0], std::max(L.n[1], L.n[2]));
    LaunchScope ls_(g, FV_K_MG_OTHER);
    auto run = [&](void (*kern)(CoarseDev, const float*, float*), int NM) {
      return tc5::launch_pdl(kern, dim3(1), dim3(kExactThreads), exact_smem(L.n, NM), st, M->coarse,
                             (const float*)H.b, H.x);
    };
    FV_CUDA(m <= 16 ? run(k_exact<16>, 16) : m <= 20 ? run(k_exact<20>, 20) : m <= 24 ? run(k_exact<24>, 24)
            : m <= 28 ? run(k_exact<28>, 28) : run(k_exact<32>, 32));
    return FV_OK;
  }
  // 16 lines per block: at 100^3 two blocks per SM (1024 cells per line still
  // fit one block's shared memory)
  bool b_early = false;      // the first sweep follows the kernel that wrote b
  auto sweep = [&](int D, int color) {
    const fv_status r = line_sweep(g, H, D, color, omega, b_early, st);
    b_early = true;
    return r;
  };
  // symmetric Gauss-Seidel: x, y, z (colours 0, 1) before, the exact reverse after
  for (int s = 0; s < nu; ++s)
    for (int D = 0; D < 3; ++D)
      for (int c = 0; c < 2; ++c) FV_TRY(sweep(D, c));
  const MgLevelHost& C = M->lev[l + 1];
  MG_LAUNCH(FV_K_MG_OTHER, k_resid32<<<blocks_for(L.ncell), 256, 0, st>>>(L, H.x, H.b, H.res));
  MG_LAUNCH(FV_K_MG_OTHER, k_restrict<<<blocks_for(C.dev.ncell), 256, 0, st>>>(L, C.dev.n[0], C.dev.n[1], C.dev.n[2],
                                                                             H.res, C.b, C.x));
  FV_TRY(vcycle(g, M, l + 1, nu, omega, st));
  MG_LAUNCH(FV_K_MG_OTHER, k_prolong_add<<<blocks_for(L.ncell), 256, 0, st>>>(L, C.dev.n[0], C.dev.n[1], C.x, H.x));
  for (int s = 0; s < nu; ++s)
    for (int D = 2; D >= 0; --D)
      for (int c = 1; c >= 0; --c) FV_TRY(sweep(D, c));
  return FV_OK;
}

// one conjugate-gradient iteration on the stream st; h: the WHILE node's
// handle when captured
fv_status iteration(const fv_grid* g, MgState* M, int nu, float omega, cudaStream_t st,
                    const cudaGraphConditionalHandle* h) {
  const unsigned n = (unsigned)g->ncell;
  MgLevelHost& H = M->lev[0];
  FV_TRY(vcycle(g, M, 0, nu, omega, st));
  MG_LAUNCH(FV_K_MG_OTHER, k_dots2<<<kRedBlocks, kRedThreads, 0, st>>>(n, M->r, H.x, M->zo, M->red));
  MG_LAUNCH(FV_K_MG_OTHER, k_cg_dir<<<blocks_for(n), 256, 0, st>>>(n, M->red.s, M->zo, M->p));
  {
    // about kRedBlocks blocks over plane tiles x chunks of planes
    const int tiles = std::min(kRedBlocks, (g->n[0] * g->n[1] + kRedThreads - 1) / kRedThreads);
    const int chunks = std::min(g->n[2], std::max(1, kRedBlocks / tiles));
    const int kz = (g->n[2] + chunks - 1) / chunks;
    MG_LAUNCH(FV_K_MG_OTHER, k_apply64<<<dim3(tiles, (g->n[2] + kz - 1) / kz), kRedThreads, 0, st>>>(
                                 M->fine, M->p, M->q, kz, M->red));
  }
  cudaGraphConditionalHandle hh = {};
  if (h) hh = *h;
  MG_LAUNCH(FV_K_MG_OTHER, k_cg_step<<<kRedBlocks, kRedThreads, 0, st>>>(n, M->p, M->q, M->call, M->r, H.b,
                                                                       M->red, hh, h ? 1 : 0));
  return FV_OK;
}

void drop_mg_graph(MgState* M) {
  if (M->exec) cudaGraphExecDestroy(M->exec);
  if (M->graph) cudaGraphDestroy(M->graph);
  M->exec = nullptr;
  M->graph = nullptr;
}

// The iterations as a graph: k_begin -> WHILE { iteration }
fv_status build_mg_graph(fv_grid* g, MgState* M, int nu, float omega) {
  drop_mg_graph(M);
  cudaStream_t cs, bs;
  FV_TRY(capture_streams(&cs, &bs));
  const bool prof = g->prof_on;
  g->prof_on = false;
  g->capturing = true;
  cudaGraph_t graph = nullptr;
  bool begun = false;
  auto capture = [&]() -> fv_status {
    FV_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    begun = true;
    cudaStreamCaptureStatus cst;
    cudaGraph_t cap;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    FV_CUDA(cudaStreamGetCaptureInfo(cs, &cst, nullptr, &cap, &deps, nullptr, &nd));
    cudaGraphConditionalHandle h;
    FV_CUDA(cudaGraphConditionalHandleCreate(&h, cap, 0, cudaGraphCondAssignDefault));
    k_begin<<<1, 1, 0, cs>>>(M->red.s, M->call, h);
    FV_CHECK_LAUNCH();
    FV_CUDA(cudaStreamGetCaptureInfo(cs, &cst, nullptr, &cap, &deps, nullptr, &nd));
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t cnode;
    FV_CUDA(cudaGraphAddNode(&cnode, cap, deps, nullptr, nd, &cp));
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    FV_CUDA(cudaStreamBeginCaptureToGraph(bs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    const fv_status s2 = iteration(g, M, nu, omega, bs, &h);
    cudaGraph_t bg = body;
    const cudaError_t e2 = cudaStreamEndCapture(bs, &bg);
    FV_TRY(s2);
    FV_CUDA(e2);
    FV_CUDA(cudaStreamUpdateCaptureDependencies(cs, &cnode, nullptr, 1, cudaStreamSetCaptureDependencies));
    return FV_OK;
  };
  fv_status s = capture();
  const cudaError_t ec = begun ? cudaStreamEndCapture(cs, &graph) : cudaSuccess;
  g->prof_on = prof;
  g->capturing = false;
  if (s == FV_OK && ec != cudaSuccess) s = cuda_fail(ec, "cudaStreamEndCapture", __FILE__, __LINE__);
  if (s == FV_OK) {
    const cudaError_t ei = cudaGraphInstantiate(&M->exec, graph, 0);
    if (ei != cudaSuccess) s = cuda_fail(ei, "cudaGraphInstantiate", __FILE__, __LINE__);
  }
  if (s != FV_OK) {
    if (graph) cudaGraphDestroy(graph);
    M->exec = nullptr;
    drop_capture_streams();
    (void)cudaGetLastError();
    return s;
  }
  M->graph = graph;
  M->nu = nu;
  M->omega = omega;
  return FV_OK;
}

}  // namespace

void destroy_mg(fv_grid* g) {
  MgState* M = (MgState*)g->mg;
  if (!M) return;
  if (M->d_tab) cudaFree(M->d_tab);
  if (M->d_work) cudaFree(M->d_work);
  if (M->r) cudaFree(M->r);
  if (M->h) cudaFreeHost(M->h);
  drop_mg_graph(M);
  delete M;
  g->mg = nullptr;
}

fv_status mg_solve(fv_grid* g, const double* r, double* phi, const double* guess,
                   const fv_mg_opts& o, fv_mg_stats* stats) {
  if (!g->mg) {
    const fv_status s = build_mg(g);
    if (s != FV_OK) {
      destroy_mg(g);
      return s;
    }
  }
  MgState* M = (MgState*)g->mg;
  FV_TRY(set_line_attributes());
  cudaStream_t st = g->stream;
  const unsigned n = (unsigned)g->ncell;
  const int nb = kRedBlocks;
  const float omega = (float)o.omega;
  MgLevelHost& H = M->lev[0];
  // compatible right-hand side and the initial residual
  M->h->call = {phi, o.rtol, o.max_iter};
  FV_CUDA(cudaMemcpyAsync(M->call, &M->h->call, sizeof(MgCall), cudaMemcpyHostToDevice, st));
  MG_LAUNCH(FV_K_MG_OTHER, k_sum_vr<<<nb, kRedThreads, 0, st>>>(M->fine, r, M->red, S_VR));
  if (guess && guess != phi)
    FV_CUDA(cudaMemcpyAsync(phi, guess, n * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (!guess) FV_CUDA(cudaMemsetAsync(phi, 0, n * sizeof(double), st));
  MG_LAUNCH(FV_K_MG_OTHER, k_rhs<<<nb, kRedThreads, 0, st>>>(M->fine, r, M->vtot, guess ? phi : nullptr, M->r, H.b,
                                                            H.x, M->zo, M->red));
  auto fetch = [&]() -> fv_status {
    FV_CUDA(cudaMemcpyAsync(M->h->s, M->red.s, S_N * sizeof(double), cudaMemcpyDeviceToHost, st));
    FV_CUDA(cudaStreamSynchronize(st));
    return FV_OK;
  };
  const double* hs = M->h->s;
  auto rnorm = [&]() { return std::sqrt(std::max(hs[S_RR], 0.0)); };
  if (g->use_graph && !g->prof_on) {
    if (!M->exec || M->nu != o.nu || M->omega != omega) FV_TRY(build_mg_graph(g, M, o.nu, omega));
    count_launch();
    FV_CUDA(cudaGraphLaunch(M->exec, st));
  } else {                 // launch by launch (per-kernel timing)
    FV_TRY(fetch());
    while (std::isfinite(hs[S_RR]) && hs[S_BB] > 0.0 && rnorm() > o.rtol * std::sqrt(hs[S_BB]) &&
           hs[S_IT] < o.max_iter) {
      FV_TRY(iteration(g, M, o.nu, omega, st, nullptr));
      FV_TRY(fetch());
    }
  }
  // zero volume-weighted mean
  MG_LAUNCH(FV_K_MG_OTHER, k_sum_vr<<<nb, kRedThreads, 0, st>>>(M->fine, phi, M->red, S_VPHI));
  MG_LAUNCH(FV_K_MG_OTHER, k_sub_mean<<<blocks_for(n), 256, 0, st>>>(n, M->red.s, M->vtot, phi));
  FV_TRY(fetch());
  const double bnorm = std::sqrt(hs[S_BB]);
  fv_mg_stats sv = {};
  sv.levels = M->levels;
  sv.iterations = (int)hs[S_IT];
  sv.rel_res = bnorm > 0.0 ? rnorm() / bnorm : 0.0;
  if (stats) *stats = sv;
  // (a NaN right-hand side gives a NaN norm; max() above would hide it)
  if (!std::isfinite(hs[S_RR]) || !std::isfinite(bnorm)) {
    set_error("fv_pressure_solve_mg: NaN in the residual");
    return FV_ENAN;
  }
  if (bnorm > 0.0 && rnorm() > o.rtol * bnorm) {
    set_error("fv_pressure_solve_mg: no convergence within max_iter");
    return FV_ENOCONV;
  }
  return FV_OK;
}

}  // namespace fv

using namespace fv;

extern "C" fv_status fv_pressure_solve_mg(fv_grid* g, const double* r, double* phi,
                                          const double* guess, const fv_mg_opts* opts,
                                          fv_mg_stats* stats) {
  if (!g || !r || !phi) {
    set_error("fv_pressure_solve_mg: NULL argument");
    return FV_EINVAL;
  }
  fv_mg_opts o = {};
  if (opts) o = *opts;
  if (o.rtol <= 0) o.rtol = 1e-10;
  if (o.max_iter <= 0) o.max_iter = 100;
  if (o.nu <= 0) o.nu = 1;
  if (o.omega <= 0) o.omega = 1.0;
  if (o.nu > 8 || o.omega >= 2.0) {
    set_error("fv_pressure_solve_mg: bad option (nu <= 8, 0 < omega < 2)");
    return FV_EINVAL;
  }
  return mg_solve(g, r, phi, guess, o, stats);
}

// host-only: the 1-D multigrid hierarchy of one axis
extern "C" int fv_host_mg_axis(int n, int map, int level, int* n_out, double* faces,
                               int* pc0, double* pw1) {
  if (n < 1 || level < 0 || !n_out || map < 0 || map > 2) return FV_EINVAL;
  std::vector<Axis1D> ax;
  ax.push_back(axis_from_faces(map_faces(n, map)));
  for (int l = 0; l < level; ++l) ax.push_back(coarsen(ax.back()));
  const Axis1D& a = ax[level];
  *n_out = a.n;
  if (faces) std::memcpy(faces, a.x.data(), (a.n + 1) * sizeof(double));
  if (pc0 || pw1) {
    const Axis1D c = coarsen(a);
    std::vector<int> c0;
    std::vector<double> w1;
    prolongation(a, c, c0, w1);
    if (pc0) std::memcpy(pc0, c0.data(), a.n * sizeof(int));
    if (pw1) std::memcpy(pw1, w1.data(), a.n * sizeof(double));
  }
  return FV_OK;
}

extern "C" int fv_host_mg_levels(int nx, int ny, int nz) {
  const int n[3] = {nx, ny, nz};
  if (nx < 1 || ny < 1 || nz < 1) return -1;
  return count_levels(n);
}
