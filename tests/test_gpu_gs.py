"""Gram-Schmidt step as one kernel (fv_gs.cu), float-float bases on small
grids, against the FP64 form, whose basis keeps the separate kernels.

The Stokes operator (U = 0) is self-adjoint in the W-inner product, so an
eigenvalue whose Ritz residual is at most tol |lambda| is off by at most that:
two converged values differ by 2 tol |lambda|, and round-off (1e-13) is far
below.  Newton: both end at |F| < 1e-10; with |J^-1| of a few and quadratic
convergence the velocities differ by less than 1e-8 of the lid's."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402

TOL = 1e-8


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as m
    return m


# entries of w: fewer than a warp per block, odd ends of slices, the longest
# basis, one and several runs per slice, slices near the limit and beyond it
@pytest.mark.parametrize("shape,m", [((4, 5, 4), 8), ((9, 11, 13), 31), ((16, 16, 16), 128), ((33, 20, 17), 40),
                                     ((40, 36, 44), 25), ((54, 52, 54), 30), ((58, 60, 56), 30)])
def test_arnoldi(fv, shape, m):
    nx, ny, nz = shape
    g = fv.Grid(nx, ny, nz, "uniform", re=1.0)
    U = torch.zeros(g.n_vel, dtype=torch.float64, device="cuda")
    v0 = torch.as_tensor(synth.gaussian_velocity((nx, ny, nz), 3)).to("cuda")
    lam = {p: fv.arnoldi_leading(g, U, v0, m=m, nev=1, tol=TOL, prec=p)[0][0] for p in ("ff", "fp64")}
    assert abs(lam["ff"] - lam["fp64"]) <= 2 * TOL * abs(lam["fp64"]) + 1e-12 * abs(lam["fp64"])
    again = fv.arnoldi_leading(g, U, v0, m=m, nev=1, tol=TOL, prec="ff")[0][0]
    assert again == lam["ff"]


@pytest.mark.parametrize("shape", [(9, 8, 10), (13, 12, 11), (16, 16, 16)])
def test_newton(fv, shape):
    U = {}
    for p in ("ff", "fp64"):
        g = fv.Grid(*shape, "cosine", re=100.0)
        U[p] = torch.zeros(g.n_vel, dtype=torch.float64, device="cuda")
        P = torch.zeros(g.n_cell, dtype=torch.float64, device="cuda")
        assert fv.newton_steady(g, U[p], P, prec=p)["res_final"] < 1e-10
    assert float((U["ff"] - U["fp64"]).abs().max()) < 1e-8
