"""A grid may be made on one stream and used on another at once
(fv_grid_set_stream): what its creation computes on the device, the factors of
the float64 solve and the weights of the inner product, is there by then, even
if the stream it was made on has work queued before it.  Compared bit for bit
with a grid that lives on one stream."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402


@pytest.mark.parametrize("shape", [(12, 14, 16), (60, 50, 70)])
def test_first_use_on_another_stream(shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as fv
    nz, ny, nx = shape
    x = torch.tensor(synth.gaussian_velocity(shape, 3), device="cuda")
    r = torch.tensor(synth.gaussian_cells(shape, 5), device="cuda")

    def results(g):
        phi = torch.empty_like(r)
        fv.fv_pressure_solve(g, r, phi, prec="fp64")
        return phi, fv.fv_dot_w(g, x, x)

    want, dot = results(fv.Grid(nx, ny, nz, "cosine"))
    torch.cuda.synchronize()
    made, used = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(made):
        torch.cuda._sleep(int(1e8))                  # about 50 ms of work queued first
    with torch.cuda.stream(used):
        g = fv.Grid(nx, ny, nz, "cosine", stream=made.cuda_stream)
        g.set_stream(used.cuda_stream)
        phi, d = results(g)
        used.synchronize()
    assert torch.equal(phi, want) and d == dot
