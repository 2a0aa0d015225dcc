"""The multigrid solve at the edges of its kernels: the exactly solved level
at each of its register widths (16, 20, 24, 28, 32 cells), one cell beyond it
(33: the first grid with line sweeps), lines of odd and of 1000 cells, blocks
of 16 lines that end early, axes of 4 cells; by graph and launch by launch
(FVNS_NO_GRAPH), with other sweep counts and relaxations on one grid (the
captured iteration is rebuilt), guess and phi the same array, and a NaN.

phi against the oracle's exact solve: 1e-8 of its largest value at a relative
residual of 1e-12, the tolerance of test_gpu_mg.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import layout  # noqa: E402
import synth  # noqa: E402
from oracle import fv as ofv, grid as og, poisson  # noqa: E402


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as m
    return m


def _problem(fv, shape, kind):
    nz, ny, nx = shape
    G = og.Grid(nx, ny, nz, kind)
    r = ofv.divergence(G, layout.to_oracle(synth.gaussian_velocity(shape, 3), shape))
    g = fv.Grid(nx, ny, nz, kind, re=1000.0)
    return g, torch.tensor(np.ascontiguousarray(r).ravel(), device="cuda"), poisson.TPF(G).solve(r).ravel()


def _err(phi, ref):
    return float(np.abs(phi.cpu().numpy() - ref).max() / np.abs(ref).max())


@pytest.mark.parametrize("shape,kind", [((4, 16, 5), "cosine"), ((20, 17, 19), "cosine"), ((24, 21, 4), "sine0975"),
                                        ((25, 28, 27), "cosine"), ((32, 31, 32), "cosine"), ((33, 4, 5), "uniform"),
                                        ((5, 33, 34), "cosine"), ((35, 37, 65), "sine0975"), ((4, 6, 1000), "uniform")])
@pytest.mark.parametrize("graph", [True, False])
def test_shapes(fv, shape, kind, graph, monkeypatch):
    if not graph:
        monkeypatch.setenv("FVNS_NO_GRAPH", "1")
    g, r, ref = _problem(fv, shape, kind)
    phi = torch.empty_like(r)
    st = fv.fv_pressure_solve_mg(g, r, phi, rtol=1e-12, max_iter=300)
    assert st["rel_res"] <= 1e-12 and _err(phi, ref) < 1e-8
    assert st["levels"] == fv.lib.fv_host_mg_levels(shape[2], shape[1], shape[0])


def test_options_and_reuse(fv):
    g, r, ref = _problem(fv, (36, 40, 34), "cosine")
    phi = torch.empty_like(r)
    its = {}
    for nu, omega in ((1, 1.0), (2, 1.0), (1, 0.8), (1, 1.0)):
        st = fv.fv_pressure_solve_mg(g, r, phi, rtol=1e-12, nu=nu, omega=omega)
        assert _err(phi, ref) < 1e-8
        its.setdefault((nu, omega), st["iterations"])
        assert its[(nu, omega)] == st["iterations"]
    st = fv.fv_pressure_solve_mg(g, r, phi, guess=phi, rtol=1e-11)
    assert st["iterations"] == 0 and _err(phi, ref) < 1e-8
    bad = r.clone()
    bad[100] = float("nan")
    with pytest.raises(fv.FvError) as e:
        fv.fv_pressure_solve_mg(g, bad, phi)
    assert e.value.status == 5
    fv.fv_pressure_solve_mg(g, r, phi, rtol=1e-12)
    assert _err(phi, ref) < 1e-8
    st = fv.fv_pressure_solve_mg(g, torch.zeros_like(r), phi)
    assert st["iterations"] == 0 and not phi.any()
