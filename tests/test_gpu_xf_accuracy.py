"""Accuracy of one pressure solve by the long-axis tensor-core kernel: the first
correction of a float-float evaluation (its pressure after one pass) against the
float64 solve of the same float32 right-hand side.

Yardstick: the FP32 kernels on the same data (fv_pressure_solve, mixed form).
They round a sum of n terms n times at random, about sqrt(n) / 4 ulp; the tensor
core cuts, n / 32 additions of half an ulp each where the main accumulator is
halved, n / 16 where it is not: for the axes here no more than the yardstick in
the mean square, and within a factor of two in the largest value.  All six products
in one accumulator (6 n / 16 cuts) would miss both by a factor of three, a lost
third part (2^-17) by one of ten.  A second solve then leaves about 1e-6 squared
of the first correction: three passes to 1e-8."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402
from oracle import grid as og, poisson  # noqa: E402


# (nz, ny, nx): one chunk of rows, two (80 rows, three accumulators), one of
# 176 .. 256 rows, several, an odd axis, all three axes long
@pytest.mark.parametrize("kind", ["sine0975", "uniform"])
@pytest.mark.parametrize("shape", [(20, 20, 125), (20, 160, 18), (150, 16, 17), (24, 20, 176), (20, 256, 16), (257, 12, 20),
                                   (16, 18, 400), (113, 131, 150)])
def test_first_correction(shape, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as fv
    nz, ny, nx = shape
    g = fv.Grid(nx, ny, nz, kind, alpha=0.3, re=900.0)
    U = torch.tensor(synth.vortex_base_flow(shape, kind, 0.3), device="cuda")
    v = torch.tensor(synth.gaussian_velocity(shape, 4), device="cuda")
    out = torch.empty_like(v)
    phi, fp32, r = (torch.empty(g.n_cell, dtype=torch.float64, device="cuda") for _ in range(3))
    o = fv.fv_simple_opts(1e-8, 1, fv.PRECS["ff"], 1.0, 0.0, 0)
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (U, v, out, phi)]
    assert fv.lib.simple_krylov_solve(g.handle, *ptr, ctypes.byref(o), None) == 4      # the cap of one pass
    fv.ns_jacvec(g, U, v, out)
    fv.ns_divergence(g, out, r)
    r = r.float().double()
    fv.fv_pressure_solve(g, r, fp32, prec="mixed")
    ref = poisson.TPF(og.Grid(nx, ny, nz, kind)).solve(r.cpu().numpy().reshape(shape)).ravel()
    e, y = (t.cpu().numpy() - ref for t in (phi, fp32))
    rms = [float(np.sqrt(np.mean(d * d) / np.mean(ref * ref))) for d in (e, y)]
    top = [float(np.abs(d).max() / np.abs(ref).max()) for d in (e, y)]
    print(f"\n{shape} {kind}: rms {rms[0]:.2e} ({rms[1]:.2e}), max {top[0]:.2e} ({top[1]:.2e})")
    assert rms[0] <= rms[1] and top[0] <= 2 * top[1]
    assert fv.simple_krylov_solve(g, U, v, out, eps=1e-8, prec="ff")["passes"] == 3
