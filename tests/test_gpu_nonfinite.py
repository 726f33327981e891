"""A state that is not finite gives time derivatives that are not, in every form of the element
solves, and the call says so where it iterates."""
import numpy as np
import pytest

from paper_2105_01722_gb300 import gdg, inputs

pytestmark = pytest.mark.gpu

FORMS = {"pcg": {}, "mixed": {"precision": gdg.MIXED}, "inverse": {"solver": gdg.SOLVE_INVERSE}}


def _gpu(a):
    import torch
    return torch.tensor(np.ascontiguousarray(a, dtype=np.float64).ravel(), device="cuda")


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("kind", ["mapped", "cartesian"])     # (parallelograms: the mass solve starts with an FP64 step)
def test_non_finite_state(form, bad, kind):
    """u of element 1 has a NaN or infinity at its middle: dV/dt and dU/dt there are NaN at every node,
    elements 3 and 4, which do not touch it, keep their bits, and an iterative form returns GDG_ENOCONV."""
    import torch
    n = (5, 1)
    X, Y = inputs.mapped_nodes(n, 8, 0.05) if kind == "mapped" else inputs.cartesian_nodes(n, 8)
    ctx = gdg.Context(gdg.make_problem(2, n, 8, 5, coef=gdg.COEF_NODAL, x_nodes=X, y_nodes=Y, c2_nodes=inputs.c2_sine(X, Y),
                                       pcg_maxit=60, **FORMS[form]))
    out = []
    for value in (None, bad):
        u, v = (_gpu(inputs.random_state((5, 81), k)) for k in (5, 6))
        if value is not None:
            u[81 + 40] = value
        du, dv = torch.zeros_like(u), torch.zeros_like(u)
        status = gdg.OK
        try:
            ctx.rhs(u, v, du, dv)
        except gdg.GdgError as e:
            status = e.status
        assert status == (gdg.OK if value is None or form == "inverse" else gdg.ENOCONV)
        if value is not None and form != "inverse":
            assert max(s["unconverged"] for s in ctx.step_stats()) >= 1
        out.append((du.view(5, 81), dv.view(5, 81)))
    assert bool(torch.isnan(out[1][1][1]).all()) and bool(torch.isnan(out[1][0][1]).all())
    for k in (3, 4):
        assert torch.equal(out[0][0][k], out[1][0][k]) and torch.equal(out[0][1][k], out[1][1][k])
    ctx.close()
