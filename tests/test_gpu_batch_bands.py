"""Work items of the batched J.v (bands of at most 1024 cells of a z-tile's
planes) at the edges of their ranges: a plane of exactly one band, of one cell
more, of several bands with a remainder, and planes far below a band; tiles of
one plane, of more planes than divide nz, and of more planes than the grid has.
Against single-instance evaluations, whose float32 J.v sums the same fluxes in
another order: 1e-6 of the largest entry, as for the other batches."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402


@pytest.mark.parametrize("planes", [1, 3, 64])
def test_batch_bands(planes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as fv
    shapes = [(6, 5, 4), (7, 32, 32), (5, 25, 41), (8, 47, 51), (9, 4, 7)]      # nz, ny, nx
    grids, U, X, O = [], [], [], []
    for i, (nz, ny, nx) in enumerate(shapes):
        g = fv.Grid(nx, ny, nz, "cosine", alpha=0.3, re=400.0 + 100 * i)
        grids.append(g)
        U.append(torch.tensor(synth.vortex_base_flow((nz, ny, nx), "cosine", 0.3), device="cuda"))
        X.append(torch.tensor(synth.gaussian_velocity((nz, ny, nx), 31 + i), device="cuda"))
        O.append(torch.full((g.n_vel,), float("nan"), dtype=torch.float64, device="cuda"))
    b = fv.Batch(grids)
    assert fv.lib.fv_batch_set_tile(b.handle, planes) == 0
    b.krylov(U, X, O, eps=1e-8, sigma=10.0)
    for i, g in enumerate(grids):
        r = torch.empty_like(O[i])
        fv.simple_krylov_solve(g, U[i], X[i], r, None, eps=1e-8, prec="mixed", sigma=10.0)
        assert (O[i] - r).abs().max() <= 1e-6 * r.abs().max(), i
