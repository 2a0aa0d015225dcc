"""One Gram-Schmidt step of the Krylov drivers (fv_gs.cu up to about 54^3 cells,
the separate kernels beyond) against extended precision: coefficients, norm,
the new vector and its W-orthogonality to the basis, for float64 and for
float-float bases.

Entries are taken to 2^-46 (truncated to two floats), products drop 2^-46 and
sums round at 2^-47 of their running value: by |(W a, b)| <= |a| |b| a
coefficient is off by at most about 4 2^-46 |w| = 6e-14 |w|, and the rest of w,
formed by a sum over the basis and orthogonalised twice, by as much again.
Tolerance 2e-13 |w|; without the lower parts it would be 1e-7."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import layout  # noqa: E402
import synth  # noqa: E402
from oracle import fv as ofv, grid as og  # noqa: E402

FV_ETIMEOUT = 6
TOL = 2e-13


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as m
    return m


def _problem(shape, j1):
    nz, ny, nx = shape
    W = layout.from_oracle(ofv.weights(og.Grid(nx, ny, nz, "cosine")))
    n = W.size
    rng = np.random.default_rng(7)
    root = np.sqrt(W)
    inside = root > 0
    V = np.zeros((n, j1))
    V[inside] = np.linalg.qr(rng.standard_normal((int(inside.sum()), j1)))[0] / root[inside, None]
    w = np.where(inside, synth.gaussian_velocity(shape, 3), 0.0)
    w += V @ rng.standard_normal(j1) * np.sqrt(np.sum(W * w * w))          # coefficients of the size of w
    return W, V, w


def _step(fv, g, V, w, pairs):
    """Coefficients, norm and new vector as the library leaves them; the basis it used."""
    n, j1 = V.shape
    h = np.empty(j1 + 1)
    wd = torch.tensor(w, device="cuda")
    if pairs:
        hi = V.astype(np.float32)
        P = np.zeros((j1 + 1, n, 2), np.float32)
        P[:j1, :, 0], P[:j1, :, 1] = hi.T, (V - hi).T.astype(np.float32)
        V = (P[:j1, :, 0].astype(np.float64) + P[:j1, :, 1]).T
        Vd = torch.tensor(P, device="cuda")
    else:
        Vd = torch.tensor(np.ascontiguousarray(V.T), device="cuda")
    assert fv.lib.fv_debug_gram_schmidt(g.handle, ctypes.c_void_p(Vd.data_ptr()), pairs, j1,
                                        ctypes.c_void_p(wd.data_ptr()), h.ctypes.data) == 0
    new = Vd[j1].double().sum(1) if pairs else wd
    return h, new.cpu().numpy(), V


# entries per block: fewer than a warp, odd ends of slices, one and several runs,
# near the limit of the one-kernel form, beyond it
@pytest.mark.parametrize("pairs", [0, 1])
@pytest.mark.parametrize("shape,j1", [((4, 5, 4), 1), ((9, 11, 13), 30), ((16, 16, 16), 128), ((17, 20, 33), 5),
                                      ((44, 36, 40), 12), ((54, 52, 54), 7), ((56, 60, 58), 6)])
def test_step(fv, shape, j1, pairs):
    nz, ny, nx = shape
    g = fv.Grid(nx, ny, nz, "cosine")
    W, V, w = _problem(shape, j1)
    h, new, V = _step(fv, g, V, w, pairs)
    L = np.longdouble
    Wl, Vl, x = W.astype(L), V.astype(L), w.astype(L)
    size = float(np.sqrt(np.sum(Wl * x * x)))
    ref = np.zeros(j1, L)
    for _ in range(2):
        c = Vl.T @ (Wl * x)
        ref += c
        x = x - Vl @ c
    norm = np.sqrt(np.sum(Wl * x * x))
    assert np.abs(h[:j1] - ref).max() <= TOL * size
    assert abs(h[j1] - norm) <= TOL * size
    d = new * h[j1] - x
    assert np.sqrt(np.sum(Wl * d * d)) <= TOL * size
    assert np.abs(Vl.T @ (Wl * new)).max() * float(norm) <= TOL * size


@pytest.mark.parametrize("pairs", [0, 1])
def test_results_are_nan_once_the_timeout_word_is_set(fv, pairs):
    shape = (9, 11, 13)
    nz, ny, nx = shape
    g = fv.Grid(nx, ny, nz, "cosine")
    _, V, w = _problem(shape, 6)
    fv.fv_debug_inject_status(g, FV_ETIMEOUT)
    h, new, _ = _step(fv, g, V, w, pairs)
    assert np.isnan(h).all() and np.isnan(new).all()
