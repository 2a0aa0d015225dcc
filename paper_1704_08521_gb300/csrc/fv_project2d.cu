// Divergence-free projections of a velocity field onto coordinate planes and
// their vector potentials (Section 4, Eqs. 11-17), in float64.
//
// For the planes (a, c) with normal direction b the projection keeps the two
// in-plane components, sets the normal one to zero and removes the part that
// is not divergence-free in the plane (Eqs. 12-14): plane by plane, the
// two-dimensional Leray projection  v_b = q - G_ac phi  with
// (L_a (+) L_c) phi = D_ac q  (Neumann walls, phi of zero mean in every
// plane), solved exactly by the eigenbases of the pressure operator along a
// and c: two forward transforms, division by lam_a + lam_c (the plane's
// constant null mode set to zero), two inverse transforms.  With this exact
// solve the paper's 2-D SIMPLE-like loop ends after its first correction.
// The vector potential (Eqs. 15-17) has the single component Psi^(b) on the
// corners of the plane's cells, zero on the walls: the running integral
// along a of the in-plane component c,
//   (x, z): Psi_{i+1} = Psi_i + w dx_i     (w = dPsi/dx, u = -dPsi/dz)
//   (y, z): Psi_{j+1} = Psi_j - w dy_j     (w = -dPsi/dy, v = dPsi/dz)
//   (x, y): Psi_{i+1} = Psi_i - v dx_i     (v = -dPsi/dx, u = dPsi/dy)
#include "fv_internal.cuh"

namespace fv {

namespace {

constexpr int kPlaneA[3] = {0, 1, 0}, kPlaneC[3] = {2, 2, 1}, kPlaneB[3] = {1, 0, 2};

// at most 1024 cells per axis: a cell number fits in 32 bits
__device__ __forceinline__ void cell_of(unsigned e, const int n[3], int (&p)[3]) {
  const unsigned r = e / (unsigned)n[0];
  p[0] = (int)(e - r * n[0]);
  p[2] = (int)(r / (unsigned)n[1]);
  p[1] = (int)(r - (unsigned)p[2] * n[1]);
}

__device__ __forceinline__ double factor(const TpfDev<double>& tp, int a, int c, int i, int k) {
  return i == tp.null_index[a] && k == tp.null_index[c] ? 0.0 : 1.0 / (tp.lam[a][i] + tp.lam[c][k]);
}

// r = D_ac q (the in-plane divergence; wall faces read as zero), and the plane's
// n_a n_c factors 1 / (lam_a + lam_c) (0 at the constant mode) for the transform
// along c: a division per cell is 21 us at 100^3, GB300's float64 rate being
// what it is.  What is left, 14 -> 12 us, is mostly four float64 operations per cell.
__global__ void k_div2d(Met<double> m, TpfDev<double> tp, const double* __restrict__ q, int a, int c,
                        double* __restrict__ r, double* __restrict__ inv) {
  const unsigned nc = (unsigned)m.ncell, stride = gridDim.x * blockDim.x;
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned st[3] = {1, (unsigned)m.n[0], (unsigned)m.n[0] * m.n[1]};
  const double *qa = q + a * m.ncell, *qc = q + c * m.ncell;
  for (unsigned e = t; e < (unsigned)m.n[a] * m.n[c]; e += stride)
    inv[e] = factor(tp, a, c, (int)(e / (unsigned)m.n[c]), (int)(e % (unsigned)m.n[c]));
  for (unsigned e = t; e < nc; e += stride) {
    int p[3];
    cell_of(e, m.n, p);
    const double la = p[a] > 0 ? qa[e] : 0.0, ha = p[a] + 1 < m.n[a] ? qa[e + st[a]] : 0.0;
    const double lc = p[c] > 0 ? qc[e] : 0.0, hc = p[c] + 1 < m.n[c] ? qc[e + st[c]] : 0.0;
    r[e] = (ha - la) * m.idx[a][p[a]] + (hc - lc) * m.idx[c][p[c]];
  }
}

// hat *= 1 / (lam_a + lam_c) where the transform does not cover axis c
__global__ void k_scale2d(Met<double> m, const double* __restrict__ inv, int a, int c, double* __restrict__ h) {
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < (unsigned)m.ncell; e += gridDim.x * blockDim.x) {
    int p[3];
    cell_of(e, m.n, p);
    h[e] *= inv[p[a] * m.n[c] + p[c]];
  }
}

// vp = q - G_ac phi on the in-plane components (walls zero), vp_b = 0
__global__ void k_correct2d(Met<double> m, const double* __restrict__ q, const double* __restrict__ phi,
                            int a, int c, int b, double* __restrict__ vp) {
  const unsigned nc = (unsigned)m.ncell;
  const unsigned st[3] = {1, (unsigned)m.n[0], (unsigned)m.n[0] * m.n[1]};
  const double *qa = q + a * m.ncell, *qc = q + c * m.ncell;
  double *va = vp + a * m.ncell, *vc = vp + c * m.ncell, *vb = vp + b * m.ncell;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < nc; e += gridDim.x * blockDim.x) {
    int p[3];
    cell_of(e, m.n, p);
    const double f = phi[e];
    va[e] = p[a] > 0 ? qa[e] - (f - phi[e - st[a]]) * m.idc[a][p[a]] : 0.0;
    vc[e] = p[c] > 0 ? qc[e] - (f - phi[e - st[c]]) * m.idc[c][p[c]] : 0.0;
    vb[e] = 0.0;
  }
}

// Psi on the corners, the running integral along a.  Corner array: [z][y][x]
// with n + 1 along a and c.
//
// a = x: a block takes 32 lines; runs of kRun cells pass through shared memory,
// so that memory is read and written along x, and 32 threads add up one line
// each.  One thread per line straight from memory took 44 us at 100^3 (32 lines
// per request); this takes 18, of which the dependent float64 additions are most.
constexpr int kLines = 32, kRun = 128;

__global__ void __launch_bounds__(256) k_potential_x(Met<double> m, const double* __restrict__ vc, int c, int b,
                                                     double sgn, double* __restrict__ psi) {
  __shared__ double tile[kLines][kRun + 1];
  __shared__ int64_t src[kLines], dst[kLines];
  const int nx = m.n[0], nb = m.n[b], nc1 = m.n[c] + 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned l0 = blockIdx.x * kLines, lines = (unsigned)nb * nc1;
  if (tid < kLines) {
    const unsigned l = l0 + tid;
    // y and z of the line, y fastest in memory
    const unsigned ny1 = c == 1 ? nc1 : nb;
    const int y = (int)(l % ny1), z = (int)(l / ny1);
    const bool wall = (c == 1 ? y : z) == m.n[c];        // the last face: a wall
    src[tid] = l >= lines || wall ? -1 : ((int64_t)z * m.n[1] + y) * nx;
    dst[tid] = l >= lines ? -1 : (int64_t)l * (nx + 1);
    if (l < lines) psi[dst[tid]] = 0.0;
  }
  __syncthreads();
  double s = 0.0;
  for (int x0 = 0; x0 < nx; x0 += kRun) {
    const int cnt = min(kRun, nx - x0);
    for (int l = warp; l < kLines; l += 8)
      for (int i = lane; i < kRun; i += 32)
        tile[l][i] = i < cnt && src[l] >= 0 ? vc[src[l] + x0 + i] * (sgn * m.dx[0][x0 + i]) : 0.0;
    __syncthreads();
    if (tid < kLines)
      for (int i = 0; i < cnt; i += 8) {     // the loads first: a store could alias the next one
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = tile[tid][i + q];
#pragma unroll
        for (int q = 0; q < 8; ++q) tile[tid][i + q] = s += v[q];
      }
    __syncthreads();
    for (int l = warp; l < kLines; l += 8)
      if (dst[l] >= 0)
        for (int i = lane; i < cnt; i += 32) psi[dst[l] + x0 + i + 1] = tile[l][i];
    __syncthreads();
  }
}

// a = y (b = x, c = z): one thread per line, lines along x, eight loads ahead
__global__ void __launch_bounds__(64) k_potential_y(Met<double> m, const double* __restrict__ vc, double sgn,
                                                    double* __restrict__ psi) {
  const int nx = m.n[0], ny = m.n[1];
  const unsigned l = blockIdx.x * 64 + threadIdx.x;
  const int z = (int)(l / (unsigned)nx), x = (int)(l - (unsigned)z * nx);
  if (z > m.n[2]) return;
  const bool wall = z == m.n[2];
  const double* p = vc + (int64_t)z * nx * ny + x;
  double* o = psi + (int64_t)z * nx * (ny + 1) + x;
  double s = 0.0;
  *o = 0.0;
  for (int y0 = 0; y0 < ny; y0 += 8) {
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = !wall && y0 + q < ny ? p[(int64_t)(y0 + q) * nx] : 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (y0 + q < ny) {
        s += v[q] * (sgn * m.dx[1][y0 + q]);
        o[(int64_t)(y0 + q + 1) * nx] = s;
      }
  }
}

inline unsigned blocks_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 8) b = 152 * 8;
  return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

fv_status plane_projection(const fv_grid* g, const double* v, int plane, double* vp, double* psi) {
  const int a = kPlaneA[plane], c = kPlaneC[plane], b = kPlaneB[plane];
  double* r = g->cell_buf[0];
  double* inv = g->cell_buf[1];              // n_a n_c factors
  double* t0 = (double*)g->tpf_buf[0];
  double* t1 = (double*)g->tpf_buf[1];
  {
    LaunchScope ls_(g, FV_K_DIVERGENCE);
    k_div2d<<<blocks_for(g->ncell), 256, 0, g->stream>>>(g->met_d, g->tpf_d, v, a, c, r, inv);
  }
  FV_CHECK_LAUNCH();
  FV_TRY(transform_axis_f64(g, a, 0, r, t0));
  if (oz_ok(g, c)) {
    FV_TRY(oz_transform(g, c, 0, OzScale{inv, a == 0 ? 1 : g->n[0], g->n[a]}, t0, t1));
  } else {
    FV_TRY(transform_axis_f64(g, c, 0, t0, t1));
    LaunchScope ls_(g, FV_K_VECTOR);
    k_scale2d<<<blocks_for(g->ncell), 256, 0, g->stream>>>(g->met_d, inv, a, c, t1);
  }
  FV_CHECK_LAUNCH();
  FV_TRY(transform_axis_f64(g, c, 1, t1, t0));
  FV_TRY(transform_axis_f64(g, a, 1, t0, r));   // r = phi
  {
    LaunchScope ls_(g, FV_K_CORRECT);
    k_correct2d<<<blocks_for(g->ncell), 256, 0, g->stream>>>(g->met_d, v, r, a, c, b, vp);
  }
  FV_CHECK_LAUNCH();
  if (psi) {
    const double sgn = plane == 0 ? 1.0 : -1.0;
    const double* vc = vp + c * g->ncell;
    const unsigned lines = (unsigned)g->n[b] * (g->n[c] + 1);
    LaunchScope ls_(g, FV_K_VECTOR);
    if (a == 0)
      k_potential_x<<<(lines + kLines - 1) / kLines, 256, 0, g->stream>>>(g->met_d, vc, c, b, sgn, psi);
    else
      k_potential_y<<<(lines + 63) / 64, 64, 0, g->stream>>>(g->met_d, vc, sgn, psi);
  }
  FV_CHECK_LAUNCH();
  return FV_OK;
}

}  // namespace fv

extern "C" fv_status fv_plane_projection(const fv_grid* g, const double* v, int plane, double* vp,
                                         double* psi) {
  if (!g || !v || !vp) { fv::set_error("fv_plane_projection: NULL argument"); return FV_EINVAL; }
  if (plane < 0 || plane > 2) { fv::set_error("fv_plane_projection: plane must be 0, 1 or 2"); return FV_EINVAL; }
  if (v == vp) { fv::set_error("fv_plane_projection: v and vp alias"); return FV_EINVAL; }
  return fv::plane_projection(g, v, plane, vp, psi);
}
