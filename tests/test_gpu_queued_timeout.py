"""A timeout in a call that only queues work (fv_pressure_solve and
fv_plane_projection in float64 run transforms with bounded waits): such a call
cannot return it, so the grid's timeout word stays set over it, the next call
that reports says where it may come from, and only that one call does.  The word is
set from the host, as an expired wait would set it."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402

FV_ETIMEOUT = 6


@pytest.mark.parametrize("prec", ["mixed", "ff"])
@pytest.mark.parametrize("call", ["solve", "planes"])
def test_reported_once_by_the_next_evaluation(call, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as fv
    shape = (12, 14, 16)
    nz, ny, nx = shape
    g = fv.Grid(nx, ny, nz, "cosine", re=500.0)
    U = torch.tensor(synth.vortex_base_flow(shape, "cosine", 0.0), device="cuda")
    v = torch.tensor(synth.gaussian_velocity(shape, 2), device="cuda")
    out, vp = torch.empty_like(v), torch.empty_like(v)
    r, phi = (torch.empty(g.n_cell, dtype=torch.float64, device="cuda") for _ in range(2))
    fv.simple_krylov_solve(g, U, v, out, prec=prec)
    ref = out.clone()
    fv.ns_divergence(g, v, r)

    def queued():
        if call == "solve":
            fv.fv_pressure_solve(g, r, phi, prec="fp64")
            return phi
        fv.fv_plane_projection(g, v, "xz", vp)
        return vp

    want = queued().clone()
    fv.fv_debug_inject_status(g, FV_ETIMEOUT)
    assert torch.equal(queued(), want)                       # queued, nothing to return
    fv.simple_krylov_solve(g, U, v, out, prec=prec, async_=True)
    with pytest.raises(fv.FvError) as e:
        fv.simple_krylov_solve(g, U, v, out, prec=prec)
    assert e.value.status == FV_ETIMEOUT and "queued before it" in str(e.value)
    assert torch.equal(queued(), want)
    fv.simple_krylov_solve(g, U, v, out, prec=prec)
    assert torch.equal(out, ref)
