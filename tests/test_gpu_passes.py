"""The passes of the evaluation graph (three in a row that keep the corrections
apart, then a WHILE node that folds them) against the host-driven loop, which
updates the float-float velocity pass by pass with kernels of its own: loops
that end after one, two, three and many passes, under-relaxation, pass caps,
odd sizes, tiles and chunks of one cell.

Both run the same transforms; the loops differ in how the divergence is summed
(about 2^-45 of its terms).  Mixed form: with omega < 1 the second correction is
as large as the first, so a right-hand side that rounds the other way moves a
correction by a float32 ulp: 1e-6 of the largest value, against 2e-5 for the
form's own accuracy.  Float-float form: 1e-10, as in test_gpu_parity.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402


@pytest.fixture(scope="module")
def fv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as m
    return m


def _grids(fv, shape, monkeypatch):
    nz, ny, nx = shape
    out = []
    for no_graph in ("0", "1"):
        monkeypatch.setenv("FVNS_NO_GRAPH", no_graph)
        out.append(fv.Grid(nx, ny, nz, "cosine", alpha=0.3, re=700.0))
    return out


@pytest.mark.parametrize("prec,tol", [("mixed", 1e-6), ("ff", 1e-10)])
@pytest.mark.parametrize("shape", [(4, 4, 4), (7, 9, 33), (5, 34, 64), (20, 18, 22), (6, 8, 130)])
def test_graph_matches_host_loop(fv, monkeypatch, shape, prec, tol):
    g, h = _grids(fv, shape, monkeypatch)
    U = torch.tensor(synth.vortex_base_flow(shape, "cosine", 0.3), device="cuda")
    v = torch.tensor(synth.gaussian_velocity(shape, 6), device="cuda")
    a, b = torch.empty_like(v), torch.empty_like(v)
    pa, pb = (torch.empty(g.n_cell, dtype=torch.float64, device="cuda") for _ in range(2))
    seen = set()
    for eps, omega, sigma, cap in [(10.0, 1.0, 0.0, 200), (1e-3, 1.0, 0.0, 200), (1e-8, 1.0, 10.0, 200),
                                   (1e-8, 0.9, 0.0, 200), (1e-6, 0.5, 3.0, 200), (1e-8, 1.0, 0.0, 2),
                                   (1e-8, 0.5, 0.0, 4), (1e-8, 0.5, 0.0, 5)]:
        res = []
        for grid, o, p in ((g, a, pa), (h, b, pb)):
            try:
                st = fv.simple_krylov_solve(grid, U, v, o, p, eps=eps, omega=omega, sigma=sigma, max_pass=cap,
                                            prec=prec)
                res.append((0, st["passes"]))
            except fv.FvError as e:
                res.append((e.status, cap))
        assert res[0] == res[1], (eps, omega, res)
        seen.add(res[0][1])
        for x, y in ((a, b), (pa, pb)):
            assert float((x - y).abs().max()) <= tol * float(y.abs().max()), (eps, omega)
    assert {1, 2, 3, 4, 5} <= seen and max(seen) > 6


@pytest.mark.parametrize("prec", ["mixed", "ff"])
def test_zero_and_nan_and_reuse(fv, monkeypatch, prec):
    shape = (9, 10, 11)
    g, h = _grids(fv, shape, monkeypatch)
    U = torch.tensor(synth.vortex_base_flow(shape, "cosine", 0.3), device="cuda")
    v = torch.tensor(synth.gaussian_velocity(shape, 6), device="cuda")
    a, b = torch.empty_like(v), torch.empty_like(v)
    st = fv.simple_krylov_solve(g, U, torch.zeros_like(v), a, prec=prec)
    assert st["passes"] == 1 and not a.any()
    bad = v.clone()
    bad[500] = float("nan")
    with pytest.raises(fv.FvError) as e:
        fv.simple_krylov_solve(g, U, bad, a, prec=prec)
    assert e.value.status == 5
    fv.simple_krylov_solve(g, U, v, a, prec=prec)
    fv.simple_krylov_solve(h, U, v, b, prec=prec)
    assert float((a - b).abs().max()) <= 1e-9 * float(b.abs().max())
