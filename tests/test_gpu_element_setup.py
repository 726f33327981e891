"""What a context of mapped elements keeps on the device, and its setup, which forms the
matrices of a large mesh a part at a time."""
import numpy as np
import pytest

from paper_2105_01722_gb300 import gdg, inputs

pytestmark = pytest.mark.gpu

FORMS = {"pcg": {}, "mixed": {"precision": gdg.MIXED}, "inverse": {"solver": gdg.SOLVE_INVERSE}}


def _context(X, Y, C2, N, p, **kw):
    n = (X.shape[1], X.shape[0])
    return gdg.Context(gdg.make_problem(2, n, N, p, coef=gdg.COEF_NODAL, x_nodes=X, y_nodes=Y, c2_nodes=C2, **kw))


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("N,p", [(4, 3), (8, 5), (9, 7)])
def test_memory_an_element(N, p, form):
    """Per element: packed triangles of the two matrices (four with inverses) and the face operators, 8 bytes an
    entry; the face data of 16 Q doubles; 24 N1 doubles of face lines; at most 24 doubles a node (state, stages,
    diagonals, w, features); no squared matrices."""
    import torch
    n1, n = N + 1, (100, 100)
    na, Q = n1 * n1, N * (p + 1)
    X, Y = inputs.mapped_nodes(n, N, 0.05)
    C2 = inputs.c2_sine(X, Y)
    torch.cuda.synchronize()
    _context(X[:1, :1], Y[:1, :1], C2[:1, :1], N, p, **FORMS[form]).close()     # (the module's own memory first)
    before = torch.cuda.mem_get_info()[0]
    ctx = _context(X, Y, C2, N, p, **FORMS[form])
    used = (before - torch.cuda.mem_get_info()[0]) / (n[0] * n[1])
    ctx.close()
    matrices = (4 if form == "inverse" else 2) * (na * (na + 1) // 2 + 1)
    granules = 40 * 2 * 2**20 / (n[0] * n[1])       # some 30 allocations, each a whole number of 2 MB
    assert used <= 8 * (matrices + 72 * na + 16 * Q + 24 * n1 + 24 * na) + granules


@pytest.mark.parametrize("form", ["pcg", "inverse"])
def test_large_meshes_are_assembled_in_parts(form):
    """Elements on both sides of a part's end (N1 = 9: 5113 elements a part, 2556 with inverses), the first and the last:
    the bits of a 3 x 3 patch of the mesh."""
    import torch
    n, N, p = (80, 65), 8, 5
    X, Y = inputs.mapped_nodes(n, N, 0.05)
    C2 = inputs.c2_sine(X, Y)
    U, V = inputs.random_state((5200, 81), 3), inputs.random_state((5200, 81), 4)
    gpu = lambda a: torch.tensor(np.ascontiguousarray(a).ravel(), device="cuda")  # noqa: E731

    def rhs(X, Y, C2, U, V):
        ctx = _context(X, Y, C2, N, p, **FORMS[form])
        u, v = gpu(U), gpu(V)
        du, dv = torch.empty_like(u), torch.empty_like(u)
        ctx.rhs(u, v, du, dv)
        ctx.close()
        return du.view(X.shape[0], X.shape[1], 81), dv.view(X.shape[0], X.shape[1], 81)

    whole = rhs(X, Y, C2, U, V)
    per = (512 << 20) // ((4 if form == "inverse" else 2) * 81 * 81 * 8)
    for e in (0, per - 1, per, 5199):
        ey, ex = divmod(e, 80)
        rows, cols = slice(max(ey - 1, 0), ey + 2), slice(max(ex - 1, 0), ex + 2)
        patch = rhs(X[rows, cols], Y[rows, cols], C2[rows, cols], U.reshape(65, 80, 81)[rows, cols], V.reshape(65, 80, 81)[rows, cols])
        for a, b in zip(whole, patch):
            assert torch.equal(a[ey, ex], b[ey - rows.start, ex - cols.start])
