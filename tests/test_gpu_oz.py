"""The float64 pressure solve whose transforms run as digit products on the
tensor cores (axes of up to 128 cells; longer axes take the float64 kernels,
also mixed with the former in one solve).

Reference: the same six transforms and the division in extended precision
(numpy longdouble), with the library's own eigenbases.  The error of the same
sequence in float64 matrix products of numpy is the yardstick: a digit
transform rounds each result once (2^-53) and drops what is below 2^-54 of
(largest matrix entry of the row) x (largest entry of the vector); a float64
product rounds every partial sum.  On axes of 4 cells a float64 product has
hardly any sums to round, so both roundings, six transforms deep, are allowed:
error <= 2 x that of numpy + 6 x 2^-52 of max |phi|.
The digit transform is scale-free: scaling r by a power of two scales every
vector's exponent and nothing else, so phi must scale bit for bit."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402

MAPS = {"sine0975": 0, "cosine": 1}


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as m
    return m


def _solve(fv, g, r):
    phi = torch.empty(g.n_cell, dtype=torch.float64, device="cuda")
    fv.fv_pressure_solve(g, torch.tensor(np.ascontiguousarray(r).ravel(), device="cuda"), phi, prec="fp64")
    return phi.cpu().numpy()


def _basis(fv, n, kind):
    E, Ei, lam = np.empty((n, n)), np.empty((n, n)), np.empty(n)
    null = ctypes.c_int()
    assert fv.lib.fv_host_axis_basis(n, MAPS[kind], E.ctypes.data, Ei.ctypes.data, lam.ctypes.data,
                                     ctypes.addressof(null)) == 0
    return E, Ei, lam, null.value


def _reference(bases, r, t):
    """The tensor-product solve with the given bases (x, y, z) in arithmetic t."""
    den = np.zeros((), t)
    a = r.astype(t)
    for d in range(3):
        _, Ei, lam, _ = bases[d]
        a = np.moveaxis(np.moveaxis(a, 2 - d, -1) @ Ei.T.astype(t), -1, 2 - d)
        shape = [1, 1, 1]
        shape[2 - d] = -1
        den = den + lam.astype(t).reshape(shape)
    den[tuple(bases[d][3] for d in (2, 1, 0))] = np.inf
    a = a / den
    for d in range(3):
        a = np.moveaxis(np.moveaxis(a, 2 - d, -1) @ bases[d][0].T.astype(t), -1, 2 - d)
    return a.ravel()


def _check(bases, r, got):
    ref = _reference(bases, r, np.longdouble)
    top = np.abs(ref).max()
    e64 = np.abs(_reference(bases, r, np.float64) - ref).max() / top
    err = np.abs(got - ref).max() / top
    print(f"\n{r.shape}: device {float(err):.2e}, numpy float64 {float(e64):.2e}")
    assert err <= 2 * e64 + 6 * 2.0 ** -52


# (nz, ny, nx): one chunk of 16, ragged chunks, the 80 / 64-vector edge (112 /
# 113 cells), full 128 rows, and one axis beyond the kernel's range
SHAPES = [(4, 4, 4), (16, 15, 17), (5, 128, 6), (112, 7, 113), (9, 113, 81), (128, 8, 33), (130, 20, 12), (12, 9, 140),
          (10, 144, 16)]


@pytest.mark.parametrize("kind", ["cosine", "sine0975"])
@pytest.mark.parametrize("shape", SHAPES)
def test_solve_matches_extended_precision(fv, shape, kind):
    nz, ny, nx = shape
    g = fv.Grid(nx, ny, nz, kind)
    bases = [_basis(fv, n, kind) for n in (nx, ny, nz)]
    r = synth.gaussian_cells(shape, 5).reshape(shape)
    got = _solve(fv, g, r)
    _check(bases, r, got)
    # entries that differ by hundreds of orders of magnitude, and zeros
    r2 = r * 10.0 ** np.random.default_rng(1).integers(-160, 2, r.shape)
    r2[0] = 0.0
    _check(bases, r2, _solve(fv, g, r2))
    assert not _solve(fv, g, np.zeros(shape)).any()
    if max(shape) <= 128:
        for s in (-900, -3, 800):
            assert np.array_equal(_solve(fv, g, np.ldexp(r, s)), np.ldexp(got, s))


def test_nan_and_inf_are_reported(fv):
    shape = (20, 18, 22)
    nz, ny, nx = shape
    g = fv.Grid(nx, ny, nz, "cosine", re=500.0)
    U = torch.tensor(synth.vortex_base_flow(shape, "cosine", 0.0), device="cuda")
    v = synth.gaussian_velocity(shape, 2)
    out = torch.empty(g.n_vel, dtype=torch.float64, device="cuda")
    for bad in (np.nan, np.inf):
        r = synth.gaussian_cells(shape, 5)
        r[777] = bad
        assert not np.isfinite(_solve(fv, g, r)).any()
        w = v.copy()
        w[4321] = bad
        with pytest.raises(fv.FvError) as e:
            fv.simple_krylov_solve(g, U, torch.tensor(w, device="cuda"), out, prec="fp64")
        assert e.value.status == 5
    fv.simple_krylov_solve(g, U, torch.tensor(v, device="cuda"), out, prec="fp64")
    assert torch.isfinite(out).all()
