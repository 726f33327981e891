"""Element products on integers (gdg_fx.cuh): every element size, the edges of
their range, and non-finite input, against dense FP64 products and solves."""
import numpy as np
import pytest

from oracle import dg_var as dv
from paper_2105_01722_gb300 import gdg, inputs

pytestmark = pytest.mark.gpu


def _setup(n, N, p, **kw):
    X, Y = inputs.mapped_nodes(n, N, 0.05)
    C2 = inputs.c2_sine(X, Y)
    ctx = gdg.Context(gdg.make_problem(2, n, N, p, coef=gdg.COEF_NODAL, x_nodes=X, y_nodes=Y, c2_nodes=C2, **kw))
    return ctx, dv.VarProblem(n=n, N=N, p=p, X=X, Y=Y, C2=C2)


def _gpu(a):
    import torch
    return torch.tensor(np.ascontiguousarray(a, dtype=np.float64).ravel(), device="cuda")


# N + 1 = 2..10 nodes a line: 4 to 100 rows, blocks of 1 to 4 warps (64 rows fill
# two exactly), an odd and an even number of packed entries
SIZES = [(1, 1), (2, 1), (3, 3), (4, 3), (5, 5), (6, 3), (7, 7), (8, 5), (9, 7)]


@pytest.mark.parametrize("N,p", SIZES)
@pytest.mark.parametrize("which", [gdg.OP_M, gdg.OP_S])
def test_products_at_every_size(N, p, which):
    """With b = A x0 and rtol = 1, gdg_pcg stops before its first iteration and reports ||b - A x0|| / ||b||:
    the rounding of the two products, each at most n eps of the sum of its terms'
    magnitudes."""
    ctx, vp = _setup((3, 2), N, p, pcg_rtol=1.0, pcg_maxit=1)
    ops = dv.assemble(vp)
    na = (N + 1) ** 2
    x0 = inputs.random_state((6, na), 31)
    A = [dv.spd_u_matrix(ops, e) if which == gdg.OP_S else ops.M[e] for e in range(6)]
    b = np.stack([A[e] @ x0[e] for e in range(6)])
    stats = ctx.pcg(which, _gpu(b), _gpu(x0))
    bound = max(np.linalg.norm(np.abs(A[e]) @ np.abs(x0[e])) / np.linalg.norm(b[e]) for e in range(6))
    assert stats["max_iters"] == 0
    assert stats["max_rel_resid"] <= 2 * na * np.finfo(float).eps * bound
    ctx.close()


@pytest.mark.parametrize("N,p", SIZES)
@pytest.mark.parametrize("flux", ["upwind", "central", "alternating"])
def test_inverse_route_at_every_size(N, p, flux):
    """dU/dt and dV/dt (face operators, stiffness, both inverses) against direct
    solves, within 50 kappa eps as for the inverse route elsewhere."""
    import torch
    n = (3, 2)
    ctx, vp = _setup(n, N, p, solver=gdg.SOLVE_INVERSE, flux=getattr(gdg, "FLUX_" + flux.upper()))
    vp.flux = flux
    ops = dv.assemble(vp)
    u, v = inputs.random_state((6, (N + 1) ** 2), 11), inputs.random_state((6, (N + 1) ** 2), 12)
    du, dvv = dv.solve_direct(ops, v, *dv.residuals(vp, ops, u, v))
    tu, tv = _gpu(u), _gpu(v)
    gu, gv = torch.empty_like(tu), torch.empty_like(tv)
    ctx.rhs(tu, tv, gu, gv)
    kappa = max(np.linalg.cond(A) for e in range(6) for A in (dv.spd_u_matrix(ops, e), ops.M[e]))
    want = np.concatenate([du.ravel(), dvv.ravel()])
    got = torch.cat([gu, gv]).cpu().numpy()
    assert np.linalg.norm(got - want) <= max(1e-12, 50 * kappa * np.finfo(float).eps) * np.linalg.norm(want)
    ctx.close()


@pytest.mark.parametrize("scale_u,scale_v", [(1e-200, 1e-200), (1e150, 1e150), (1.0, 1e-9), (1e-9, 1.0), (0.0, 1.0)])
def test_products_scale_with_their_vectors(scale_u, scale_v):
    """dU/dt and dV/dt are linear: each vector is scaled by its own largest entry,
    so u and v may differ by any factor.  The central flux keeps dU/dt a function
    of v alone and dV/dt one of u alone."""
    import torch
    ctx, vp = _setup((3, 3), 8, 5, solver=gdg.SOLVE_INVERSE, flux=gdg.FLUX_CENTRAL)
    u, v = _gpu(inputs.random_state((9, 81), 3)), _gpu(inputs.random_state((9, 81), 4))
    du, dvv, su, sv = (torch.empty_like(u) for _ in range(4))
    ctx.rhs(u, v, du, dvv)
    ctx.rhs(u * scale_u, v * scale_v, su, sv)
    for got, want in ((su, du * scale_v), (sv, dvv * scale_u)):
        # the same integers up to a power of two, or two roundings of inputs and outputs
        assert torch.linalg.norm(got - want) <= 1e-11 * torch.linalg.norm(want)
        assert bool(torch.isfinite(got).all())
    ctx.close()


@pytest.mark.parametrize("solver,precision", [(gdg.SOLVE_PCG, gdg.FP64), (gdg.SOLVE_INVERSE, gdg.FP64)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_entries_stay_visible(solver, precision, bad):
    """A NaN or infinity in one element's u gives non-finite dV/dt there and
    leaves elements that do not touch it as they were."""
    import torch
    ctx, _ = _setup((5, 1), 8, 5, solver=solver, precision=precision, pcg_maxit=30)
    u, v = _gpu(inputs.random_state((5, 81), 5)), _gpu(inputs.random_state((5, 81), 6))
    out = []
    for value in (None, bad):
        if value is not None:
            u[81 * 1 + 40] = value
        du, dvv = torch.empty_like(u), torch.empty_like(u)
        try:
            ctx.rhs(u, v, du, dvv)
        except gdg.GdgError as e:
            assert e.status == gdg.ENOCONV
        out.append((du.view(5, 81).clone(), dvv.view(5, 81).clone()))
    assert not bool(torch.isfinite(out[1][1][1]).any())
    for k in (3, 4):
        assert torch.equal(out[0][0][k], out[1][0][k]) and torch.equal(out[0][1][k], out[1][1][k])
    ctx.close()


@pytest.mark.parametrize("precision", [gdg.FP64, gdg.MIXED])
@pytest.mark.parametrize("which", [gdg.OP_M, gdg.OP_S])
@pytest.mark.parametrize("N,p", [(2, 1), (4, 3), (7, 5), (9, 7)])
def test_pcg_meets_its_tolerance_by_the_dense_residual(N, p, which, precision):
    """The residual of the returned iterate, formed with the dense FP64 matrix,
    is within rtol of the right-hand side (plus that product's own rounding)."""
    import torch
    ctx, vp = _setup((3, 2), N, p, pcg_rtol=1e-9, pcg_maxit=400, precision=precision)
    ops = dv.assemble(vp)
    b, x0 = inputs.random_state((6, (N + 1) ** 2), 21), inputs.random_state((6, (N + 1) ** 2), 22)
    x = _gpu(x0)
    stats = ctx.pcg(which, _gpu(b), x)
    x = x.cpu().numpy().reshape(b.shape)
    for e in range(6):
        A = dv.spd_u_matrix(ops, e) if which == gdg.OP_S else ops.M[e]
        r = np.linalg.norm(b[e] - A @ x[e])
        assert r <= 1e-9 * np.linalg.norm(b[e]) + 1e-12 * np.linalg.norm(np.abs(A) @ np.abs(x[e]))
    assert stats["unconverged"] == 0
    ctx.close()
