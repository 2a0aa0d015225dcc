"""Graph evaluations on both sides of the size from which the divergence of w
and the join take four planes per thread (2^19 cells), on axes that four does
not divide, against the float64 form: 2e-5 for the mixed form (float32 J.v on
stretched cells), 1e-11 for the float-float one (2^-46 per operation, some
hundred of them, on cells whose widths differ 100-fold).  The pressure is a sum
of float32 corrections in both forms: 2e-5."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import synth  # noqa: E402


@pytest.mark.parametrize("shape", [(4, 5, 7), (17, 9, 6), (80, 81, 80), (81, 81, 80)])
@pytest.mark.parametrize("prec,tol", [("mixed", 2e-5), ("ff", 1e-11)])
def test_evaluation(shape, prec, tol):
    import paper_1704_08521_gb300 as fv
    g = fv.Grid(*shape, "cosine", alpha=0.3, re=500.0)
    U, v = (torch.as_tensor(synth.gaussian_velocity(shape[::-1], s)).to("cuda") for s in (1, 2))
    out = {}
    for p in (prec, "fp64"):
        out[p] = torch.full_like(v, float("nan")), torch.full((g.n_cell,), float("nan"), dtype=torch.float64,
                                                              device="cuda")
        fv.simple_krylov_solve(g, U, v, out[p][0], out[p][1], eps=1e-10, prec=p, sigma=10.0)
    for a, b, t in zip(out[prec], out["fp64"], (tol, 2e-5)):
        assert float((a - b).norm() / b.norm()) < t
