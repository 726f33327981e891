"""Element operators at scales other than 1: the mapped path through gdg_rhs, gdg_step and
gdg_batch_step where c^2 or the mesh is not of order 1, and where a matrix is not finite."""
import numpy as np
import pytest

from oracle import dg_var as dv
from paper_2105_01722_gb300 import gdg, inputs

pytestmark = pytest.mark.gpu


def _problem(n, N, p, c2_factor=1.0, size=1.0, **kw):
    X, Y = inputs.mapped_nodes(n, N, 0.05)
    return gdg.make_problem(2, n, N, p, coef=gdg.COEF_NODAL, x_nodes=X * size, y_nodes=Y * size,
                            c2_nodes=inputs.c2_sine(X, Y) * c2_factor, **kw)


def _gpu(a):
    import torch
    return torch.tensor(np.ascontiguousarray(a, dtype=np.float64).ravel(), device="cuda")


# the wave equation is the same under c^2 -> s^2 c^2, v -> s v, t -> t / s; with s a power of two
# every product, sum, quotient and square root of the inverse route scales by one too
SCALES = [-10, 7, 10, 13]


@pytest.mark.parametrize("k", SCALES)
@pytest.mark.parametrize("N,p", [(7, 3), (8, 5), (9, 7)])
def test_inverse_route_does_not_depend_on_the_unit_of_time(N, p, k):
    """c^2 from 1e-6 to 7e7: the same bits, up to the scale, as with c^2 of order 1."""
    import torch
    n, na = (4, 4), 16 * (N + 1) ** 2
    out = []
    for s in (1.0, 2.0**k):
        ctx = gdg.Context(_problem(n, N, p, c2_factor=s * s, solver=gdg.SOLVE_INVERSE))
        u, v = _gpu(inputs.random_state((na,), 1)), _gpu(inputs.random_state((na,), 2)) * s
        du, dv = torch.empty_like(u), torch.empty_like(u)
        ctx.rhs(u, v, du, dv)
        ctx.step(u, v, 0.0, 1e-3 / s, 2)
        out.append([du / s, dv / s**2, u, v / s])
        ctx.close()
    for a, b in zip(*out):
        assert bool(torch.isfinite(a).all()) and torch.equal(a, b)


@pytest.mark.parametrize("k", SCALES)
def test_batched_inverses_do_not_depend_on_the_unit_of_time(k):
    import torch
    out = []
    for s in (1.0, 2.0**k):
        batch = gdg.Batch([_problem((3, 2), 8, p, c2_factor=s * s, solver=gdg.SOLVE_INVERSE) for p in (3, 7)])
        us = [_gpu(inputs.random_state((6 * 81,), 1 + i)) for i in range(2)]
        vs = [_gpu(inputs.random_state((6 * 81,), 5 + i)) * s for i in range(2)]
        batch.step(us, vs, [1e-3 / s] * 2, 2)
        out.append(us + [v / s for v in vs])
        batch.close()
    for a, b in zip(*out):
        assert bool(torch.isfinite(a).all()) and torch.equal(a, b)


@pytest.mark.parametrize("k", [-133, 133])
@pytest.mark.parametrize("form", ["pcg", "inverse"])
@pytest.mark.parametrize("what", ["length", "time"])
def test_far_scales(what, form, k):
    """Meshes of 1e-40 and 1e40, c^2 of 1e-80 and 1e80: matrix entries far beyond 2^+-240, the same
    bits as at scale 1.  (The iteration of the PCG form sees c^2 against its rank-one term: there the residuals
    alone are the same.)"""
    import torch
    n, N, p = (3, 2), 8, 5
    out = []
    for s in (1.0, 2.0**k):
        size, c2 = (s, 1.0) if what == "length" else (1.0, s * s)
        rate = 1.0 / s if what == "length" else s            # time runs faster by this factor
        ctx = gdg.Context(_problem(n, N, p, c2_factor=c2, size=size,
                                   solver=gdg.SOLVE_INVERSE if form == "inverse" else gdg.SOLVE_PCG))
        u, v = _gpu(inputs.random_state((6 * 81,), 1)), _gpu(inputs.random_state((6 * 81,), 2)) * rate
        ru, rv, du, dv = (torch.empty_like(u) for _ in range(4))
        ctx.residuals(u, v, ru, rv)
        fields = [ru / rate / c2, rv / c2]
        if form == "inverse" or what == "length":
            ctx.rhs(u, v, du, dv)
            fields += [du / rate, dv / rate / rate]
        out.append(fields)
        ctx.close()
    for a, b in zip(*out):
        assert bool(torch.isfinite(a).all()) and torch.equal(a, b)


def test_inverses_that_are_not_finite_stay_visible():
    """A node pushed through its neighbours folds an element: its matrices are not positive definite, the
    Cholesky factors not finite, and neither are its time derivatives; the other elements' are."""
    import torch
    X, Y = inputs.cartesian_nodes((2, 2), 8)
    X = X.copy()
    X[0, 0, 4, 4] += 0.2
    ctx = gdg.Context(gdg.make_problem(2, (2, 2), 8, 5, coef=gdg.COEF_NODAL, x_nodes=X, y_nodes=Y, c2_nodes=np.ones_like(X),
                                       solver=gdg.SOLVE_INVERSE))
    u, v = _gpu(inputs.random_state((4 * 81,), 5)), _gpu(inputs.random_state((4 * 81,), 6))
    du, dv = torch.zeros_like(u), torch.zeros_like(u)
    ctx.rhs(u, v, du, dv)
    for f in (du.view(4, 81), dv.view(4, 81)):
        assert not bool(torch.isfinite(f[0]).any()) and bool(torch.isfinite(f[1:]).all())
    ctx.close()


@pytest.mark.parametrize("form", ["pcg", "mixed", "inverse"])
def test_face_operators_that_are_not_finite_stay_visible(form):
    """Positive nodal c^2 whose interpolant dips below zero on two faces of one element: its local
    wave speed is NaN there.  So are r_u in the element (the lifts of a face's line integrals reach every node,
    if with factor zero) and r_v at the nodes of those faces, as in FP64 sums, and nothing else."""
    import torch
    n, N, p = (4, 1), 8, 5
    X, Y = inputs.cartesian_nodes(n, N)
    C2 = np.ones_like(X)
    C2[0, 1, 0::2, :] = 1e-3          # element 1: dips between its rows, on its left and right faces
    with np.errstate(invalid="ignore"):
        c = dv.assemble(dv.VarProblem(n=n, N=N, p=p, X=X, Y=Y, C2=C2)).c
    assert [bool(np.isnan(c[f]).any()) for f in dv.FACES] == [True, True, False, False]
    assert not any(np.isnan(c[f][[0, 2, 3]]).any() for f in dv.FACES)
    kw = {"pcg": {}, "mixed": {"precision": gdg.MIXED}, "inverse": {"solver": gdg.SOLVE_INVERSE}}[form]
    ctx = gdg.Context(gdg.make_problem(2, n, N, p, coef=gdg.COEF_NODAL, x_nodes=X, y_nodes=Y, c2_nodes=C2, pcg_maxit=30, **kw))
    u, v = _gpu(inputs.random_state((4, 81), 5)), _gpu(inputs.random_state((4, 81), 6))
    ru, rv = torch.empty_like(u), torch.empty_like(u)
    ctx.residuals(u, v, ru, rv)
    ru, rv = (torch.isnan(f).cpu().numpy().reshape(4, 9, 9) for f in (ru, rv))
    assert ru[1].all() and rv[1][:, [0, 8]].all() and not rv[1][:, 1:8].any()
    assert not ru[[0, 2, 3]].any() and not rv[[0, 2, 3]].any()
    ctx.close()
