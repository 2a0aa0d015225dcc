"""The passes of the evaluation graph do the arithmetic of the host-driven loop
in its order, every float-float sum renormalised: vector, pressure and all
statistics (the largest divergence that is left among them) agree bit for bit,
so there is no tolerance.  Loops of one to some twenty passes and pass caps,
under-relaxation, a shift; grids of a single tile, odd and even rows, an axis
of the fused transforms' limit and one beyond it."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402

# eps, omega, sigma, max_pass
LOOPS = [(10.0, 1.0, 0.0, 200), (1e-3, 1.0, 0.0, 200), (1e-8, 1.0, 10.0, 200), (1e-8, 0.9, 0.0, 200),
         (1e-6, 0.5, 3.0, 200), (1e-8, 1.0, 0.0, 2), (1e-8, 0.5, 0.0, 3), (1e-8, 0.5, 0.0, 4), (1e-8, 0.5, 0.0, 5)]


@pytest.mark.parametrize("prec", ["mixed", "ff"])
@pytest.mark.parametrize("shape", [(4, 4, 4), (7, 9, 33), (5, 34, 64), (20, 18, 22), (6, 8, 112), (9, 131, 6)])
def test_graph_is_the_host_loop_bit_for_bit(shape, prec, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as fv
    nz, ny, nx = shape
    grids = []
    for no_graph in ("0", "1"):
        monkeypatch.setenv("FVNS_NO_GRAPH", no_graph)
        grids.append(fv.Grid(nx, ny, nz, "cosine", alpha=0.3, re=700.0))
    U = torch.tensor(synth.vortex_base_flow(shape, "cosine", 0.3), device="cuda")
    x = torch.tensor(synth.gaussian_velocity(shape, 6), device="cuda")
    seen = set()
    for eps, omega, sigma, cap in LOOPS:
        got = []
        for g in grids:
            v = torch.empty_like(x)
            p = torch.empty(g.n_cell, dtype=torch.float64, device="cuda")
            o = fv.fv_simple_opts(eps, cap, fv.PRECS[prec], omega, sigma, 0)
            s = fv.fv_simple_stats()
            ptr = [ctypes.c_void_p(t.data_ptr()) for t in (U, x, v, p)]
            st = fv.lib.simple_krylov_solve(g.handle, *ptr, ctypes.byref(o), ctypes.byref(s))
            got.append((v, p, (st, s.passes, s.phi_first, s.phi_last, s.div_max)))
        (va, pa, sa), (vb, pb, sb) = got
        assert sa == sb, (eps, omega)
        assert torch.equal(va, vb) and torch.equal(pa, pb), (eps, omega)
        seen.add(sa[1])
    assert {1, 2, 3, 4, 5} <= seen and max(seen) > 6
