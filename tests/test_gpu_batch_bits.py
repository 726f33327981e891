"""A batched step takes a mapped problem where the problem's own gdg_step takes it,
bit for bit: the two run different kernels (in the inverse route the face operators
are read in another order), whose sums are rounded at the same places."""
import numpy as np
import pytest

from paper_2105_01722_gb300 import gdg, inputs

pytestmark = pytest.mark.gpu

FORMS = {"pcg": {}, "mixed": {"precision": gdg.MIXED}, "inverse": {"solver": gdg.SOLVE_INVERSE}}


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("N,p", [(7, 5), (8, 3), (9, 7)])
def test_batched_steps_are_the_problems_own_to_the_last_bit(N, p, form):
    import torch
    sizes, na = [(3, 2), (5, 4)], (N + 1) ** 2
    gpu = lambda a: torch.tensor(np.ascontiguousarray(a).ravel(), device="cuda")  # noqa: E731
    problems, states = [], []
    for i, n in enumerate(sizes):
        X, Y = inputs.mapped_nodes(n, N, 0.05)
        problems.append(gdg.make_problem(2, n, N, p, coef=gdg.COEF_NODAL, x_nodes=X, y_nodes=Y, c2_nodes=inputs.c2_sine(X, Y),
                                         bc=(gdg.BC_PERIODIC, gdg.BC_DIRICHLET), **FORMS[form]))
        states.append([inputs.random_state((n[0] * n[1], na), 7 + i), inputs.random_state((n[0] * n[1], na), 17 + i)])
    us, vs = ([gpu(s[k]) for s in states] for k in range(2))
    batch = gdg.Batch(problems)
    batch.step(us, vs, [1e-3, 2e-3], 5)
    for i, problem in enumerate(problems):
        ctx = gdg.Context(problem)
        u, v = (gpu(f) for f in states[i])
        ctx.step(u, v, 0.0, [1e-3, 2e-3][i], 5)
        assert torch.equal(u, us[i]) and torch.equal(v, vs[i])
        ctx.close()
    batch.close()


@pytest.mark.parametrize("N,p", [(3, 3), (4, 3), (8, 5)])
def test_large_and_small_meshes_give_the_same_bits(N, p):
    """Inverse route on 3000 elements and on 3 x 3 of them: N + 1 = 4 and 5 stage their face operators on
    the large mesh only."""
    import torch
    X, Y = inputs.mapped_nodes((60, 50), N, 0.05)
    C2, na = inputs.c2_sine(X, Y), (N + 1) ** 2
    U, V = (inputs.random_state((50, 60, na), k) for k in (1, 2))

    def rhs(rows, cols):
        x, y, c2 = (np.ascontiguousarray(f[rows, cols]) for f in (X, Y, C2))
        ctx = gdg.Context(gdg.make_problem(2, (x.shape[1], x.shape[0]), N, p, coef=gdg.COEF_NODAL, x_nodes=x, y_nodes=y,
                                           c2_nodes=c2, solver=gdg.SOLVE_INVERSE))
        u, v = (torch.tensor(np.ascontiguousarray(f[rows, cols]).ravel(), device="cuda") for f in (U, V))
        out = torch.empty_like(u), torch.empty_like(u)
        ctx.rhs(u, v, *out)
        ctx.close()
        return [f.view(x.shape[0], x.shape[1], na) for f in out]

    whole = rhs(slice(0, 50), slice(0, 60))
    for ey, ex in ((1, 1), (25, 31), (48, 58)):
        part = rhs(slice(ey - 1, ey + 2), slice(ex - 1, ex + 2))
        for a, b in zip(whole, part):
            assert torch.equal(a[ey, ex], b[1, 1])
