"""The float-float Krylov vector on grids whose pressure transforms run on the
long-axis tensor-core kernel (some axis beyond what the fused kernels hold),
against the oracle: axes around its 16-entry chunks, its 128-vector blocks,
the 256-row edge where the matrix is cut in two, odd sizes (scalar accesses)
and 4 cells.  Tolerance 1e-10 of the largest value, that of the other
float-float parity tests (test_gpu_parity.py): the loop removes what the
float32 solve rounds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import layout  # noqa: E402
import synth  # noqa: E402
from oracle import grid as og, poisson, simple  # noqa: E402


# (nz, ny, nx)
SHAPES = [(4, 5, 160), (129, 8, 6), (7, 144, 9), (16, 129, 130), (5, 4, 257), (4, 272, 7), (300, 6, 4), (12, 11, 150)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("graph", [True, False])
def test_ff_krylov_vector(shape, graph, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as fv
    if not graph:
        monkeypatch.setenv("FVNS_NO_GRAPH", "1")
    nz, ny, nx = shape
    g = fv.Grid(nx, ny, nz, "sine0975", alpha=0.3, re=900.0)
    U, v = synth.vortex_base_flow(shape, "sine0975", 0.3), synth.gaussian_velocity(shape, 4)
    out = torch.empty(g.n_vel, dtype=torch.float64, device="cuda")
    fv.simple_krylov_solve(g, torch.tensor(U, device="cuda"), torch.tensor(v, device="cuda"), out, eps=1e-10,
                           prec="ff")
    G = og.Grid(nx, ny, nz, "sine0975")
    ref, _ = simple.krylov_vector(G, poisson.TPF(G), layout.to_oracle(U, shape), layout.to_oracle(v, shape), 900.0)
    ref = layout.from_oracle(ref)
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
