"""Integer products round to nearest: what is rounded for -x is minus what is rounded for
x.  A sum that is cut off downwards instead errs to one side whatever the field, and
its error adds up over a run (linearly in the conserved 1^T M v)."""
import numpy as np
import pytest

from paper_2105_01722_gb300 import gdg, inputs

pytestmark = pytest.mark.gpu


def _gpu(a):
    import torch
    return torch.tensor(np.ascontiguousarray(a, dtype=np.float64).ravel(), device="cuda")


@pytest.mark.parametrize("form", ["pcg", "inverse"])
@pytest.mark.parametrize("flux", [gdg.FLUX_CENTRAL, gdg.FLUX_UPWIND, gdg.FLUX_ALTERNATING])
@pytest.mark.parametrize("N,p", [(4, 3), (7, 5), (8, 5), (9, 7)])
def test_mapped_elements_are_odd_in_the_state(N, p, flux, form):
    """Residuals (products with S and the face operators by both kinds of stage kernel),
    and with element inverses time derivatives and steps, of (-u, -v) are minus those of
    (u, v), bit for bit.  (Not the iterates of the PCG forms: on the unit element the
    constant mode of the preconditioner can be a power of two, so that its sums end in exact halves.
    It steers the iteration only.)"""
    import torch
    n = (5, 4)
    X, Y = inputs.mapped_nodes(n, N, 0.05)
    ctx = gdg.Context(gdg.make_problem(2, n, N, p, coef=gdg.COEF_NODAL, x_nodes=X, y_nodes=Y, c2_nodes=inputs.c2_sine(X, Y),
                                       bc=(gdg.BC_PERIODIC, gdg.BC_PERIODIC), flux=flux,
                                       solver=gdg.SOLVE_INVERSE if form == "inverse" else gdg.SOLVE_PCG))
    state = [_gpu(inputs.random_state((20, (N + 1) ** 2), k)) for k in (1, 2)]
    out = []
    for sign in (1.0, -1.0):
        u, v = (sign * f for f in state)
        fields = [torch.empty_like(u) for _ in range(2)]
        ctx.residuals(u, v, *fields)
        if form == "inverse":
            du, dv = (torch.empty_like(u) for _ in range(2))
            ctx.rhs(u, v, du, dv)
            ctx.step(u, v, 0.0, 1e-3, 2)
            fields += [du, dv, u, v]
        out.append([sign * f for f in fields])
    for a, b in zip(*out):
        assert torch.equal(a, b)
    ctx.close()


@pytest.mark.parametrize("dim,n,N,p", [(2, (5, 4), 3, 3), (2, (21, 13), 7, 5), (2, (5, 4), 8, 5), (2, (7, 3), 12, 5), (3, (3, 2, 4), 4, 3),
                                       (3, (3, 3, 2), 8, 5)])
def test_cartesian_elements_are_odd_in_the_state(dim, n, N, p):
    """The transforms between nodes and modes, alone (time derivative) and around the stages: 1^T M v, which is
    conserved, must not drift as it does where entries are cut off downwards on the way."""
    import torch
    routes = [gdg.ROUTE_MODAL] + ([gdg.ROUTE_NODAL] if dim == 2 else [])
    for route in routes:
        ctx = gdg.Context(gdg.make_problem(dim, n, N, p, bc=(gdg.BC_PERIODIC,) * dim, c2=1.3, route=route))
        state = [_gpu(inputs.random_state((ctx.n,), k)) for k in (1, 2)]
        out = []
        for sign in (1.0, -1.0):
            u, v = (sign * f for f in state)
            du, dv = torch.empty_like(u), torch.empty_like(u)
            ctx.rhs(u, v, du, dv)
            ctx.step(u, v, 0.0, 1e-4, 3)
            out.append([sign * f for f in (du, dv, u, v)])
        for a, b in zip(*out):
            assert torch.equal(a, b)
        ctx.close()
