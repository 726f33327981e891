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
