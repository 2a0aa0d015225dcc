"""Multigrid solves whose V-cycle sweeps more than one level (an axis of more
than 64 cells), where a sweep's right-hand side comes from the restriction just
before the first sweep: every reduction has a fixed order, so solves repeat bit
for bit, as one graph and launch by launch alike."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402


@pytest.mark.parametrize("shape,nu", [((66, 70, 68), 1), ((8, 140, 9), 2), ((131, 6, 7), 1)])
def test_solves_repeat_bit_for_bit(shape, nu, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as fv
    nz, ny, nx = shape
    grids = []
    for no_graph in ("0", "1"):
        monkeypatch.setenv("FVNS_NO_GRAPH", no_graph)
        grids.append(fv.Grid(nx, ny, nz, "cosine"))
    r = torch.empty(grids[0].n_cell, dtype=torch.float64, device="cuda")
    fv.ns_divergence(grids[0], torch.tensor(synth.gaussian_velocity(shape, 3), device="cuda"), r)
    ref, phi = torch.empty_like(r), torch.empty_like(r)
    its = fv.fv_pressure_solve_mg(grids[1], r, ref, rtol=1e-11, nu=nu)["iterations"]
    assert its > 2
    for _ in range(6):
        assert fv.fv_pressure_solve_mg(grids[0], r, phi, rtol=1e-11, nu=nu)["iterations"] == its
        assert torch.equal(phi, ref)
