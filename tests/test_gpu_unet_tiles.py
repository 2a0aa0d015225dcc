"""The learned guess on grids whose levels end inside the 8 x 4 x 4 cell tiles
of the contraction kernels: level 3 has an odd number of cells along every
axis, levels 1 and 2 end in partial tiles, and one axis is a single cell thick
at level 3.  Forward pass and gradients against the oracle with BF16 storage
emulated; the tolerances are those of test_gpu_unet.py (BF16 rounding
decisions move the output by up to 2.8e-3 and single gradients by up to
8e-2; a wrong tap, halo cell or channel moves them by 0.3 to 1)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import unet as ou  # noqa: E402
from test_gpu_unet import FWD_TOL, GRAD_TOL, GRAD_TOL_ALL, _net, _params, _rel  # noqa: E402


@pytest.mark.parametrize("shape", [(24, 40, 8), (8, 24, 56), (40, 8, 24)])
def test_partial_tiles(shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1704_08521_gb300 as fv
    nx, ny, nz = shape
    n = nx * ny * nz
    p = _params(8)
    rng = np.random.default_rng(9)
    planes = rng.standard_normal((4, nz, ny, nx)).astype(np.float32).astype(np.float64)
    target = rng.standard_normal((nz, ny, nx)).astype(np.float32).astype(np.float64)
    net = _net(fv, p)
    out = torch.empty(n, dtype=torch.float32, device="cuda")
    net.forward(shape, torch.tensor(planes.ravel(), dtype=torch.float32, device="cuda"), out)
    ref, _ = ou.forward(p, planes, emulate=True)
    assert _rel(out.cpu().numpy().reshape(nz, ny, nx), ref) <= FWD_TOL
    net.backward(torch.tensor(target.ravel(), dtype=torch.float32, device="cuda"))
    grads = torch.empty(net.n_param, dtype=torch.float32, device="cuda")
    net.get_params(grads=grads)
    g = grads.cpu().numpy().astype(np.float64)
    _, ref_g, _ = ou.loss_and_grad(p, planes, target, emulate=True)
    assert _rel(g, ref_g) <= GRAD_TOL_ALL
    wo, bo, hw, hb, _ = ou.layout()
    for c, (_, ci, co) in enumerate(ou.CONVS):
        for o, m in ((wo[c], 27 * ci * co), (bo[c], co)):
            assert _rel(g[o:o + m], ref_g[o:o + m]) <= GRAD_TOL, (c, o)
