"""Kernels of the plane projections where they change their path: axes beyond
the tensor-core transforms (128 cells) in every role, running integrals longer
than one run of 128 cells, line counts that do not fill the last block.
Against the oracle, element by element; uniform cells, whose eigenbases the
oracle has to 1e-13, so 1e-10 of the largest entry leaves only the kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402
import layout  # noqa: E402
from oracle import grid as og, projection2d as pr  # noqa: E402


@pytest.mark.parametrize("plane", ["xz", "yz", "xy"])
@pytest.mark.parametrize("nz,ny,nx", [(4, 5, 129), (6, 4, 300), (131, 6, 7), (5, 133, 9), (128, 4, 128)])
def test_long_and_ragged_axes(nz, ny, nx, plane):
    import paper_1704_08521_gb300 as fv
    shape = (nz, ny, nx)
    g = fv.Grid(nx, ny, nz, "uniform", re=100.0)
    G = og.Grid(nx, ny, nz, "uniform")
    v = synth.gaussian_velocity(shape, 5)
    tv = torch.tensor(v, device="cuda")
    vp = torch.full_like(tv, float("nan"))
    a, c, b = pr.PLANES[plane]
    dims = [nx, ny, nz]
    dims[a] += 1
    dims[c] += 1
    psi = torch.full((dims[0] * dims[1] * dims[2],), float("nan"), dtype=torch.float64, device="cuda")
    fv.fv_plane_projection(g, tv, plane, vp, psi)
    torch.cuda.synchronize()
    ref_v, _ = pr.project(G, layout.to_oracle(v, shape), plane)
    ref_psi = pr.potential(G, ref_v, plane)
    ref = layout.from_oracle(ref_v)
    assert np.abs(vp.cpu().numpy() - ref).max() < 1e-10 * np.abs(ref).max()
    gp = psi.cpu().numpy().reshape(dims[2], dims[1], dims[0])
    assert np.abs(gp - ref_psi).max() < 1e-10 * np.abs(ref_psi).max()
