"""Edges of the modal step kernels: windows of 1-D meshes, the entry-per-thread
persistent step, and transforms by node pairs, against the oracle and against
each other.  Tolerances: one step or transform 1e-12 relative (stacked state),
k steps k times that, as elsewhere."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import dg_const as dc, timeint as ti
from paper_2105_01722_gb300 import gdg, inputs

TOL = 1e-12
FLUX = {"upwind": gdg.FLUX_UPWIND, "central": gdg.FLUX_CENTRAL, "alternating": gdg.FLUX_ALTERNATING}


def _context(n, N, p, flux, periodic, hi=None):
    bc = tuple(gdg.BC_PERIODIC if q else gdg.BC_DIRICHLET for q in periodic)
    return gdg.Context(gdg.make_problem(len(n), n, N, p, hi=hi or (1.0,) * len(n), lo=(0.0,) * len(n), bc=bc,
                                        flux=FLUX[flux], c2=1.3))


def _state(n, N, seed):
    shape = (int(np.prod(n)), (N + 1) ** len(n))
    return [torch.tensor(inputs.random_state(shape, seed + k).ravel(), device="cuda") for k in (0, 1)]


def _rel(got, want):
    a, b = (np.concatenate([np.ravel(x.cpu().numpy() if torch.is_tensor(x) else x) for x in s]) for s in (got, want))
    return np.linalg.norm(a - b) / np.linalg.norm(b)


# one window up to 32 elements, then windows of 8 owned elements and 8 on either
# side (the last one ragged), 2 steps a launch: 1, 2 and 5 steps are a lone launch,
# a full one, and a remainder
@pytest.mark.parametrize("flux,periodic", [("upwind", False), ("central", True), ("alternating", False), ("alternating", True)])
@pytest.mark.parametrize("n,N,p", [(1, 3, 3), (2, 8, 5), (3, 1, 1), (32, 8, 3), (33, 8, 5), (41, 6, 3), (100, 12, 5)])
def test_line_windows(n, N, p, flux, periodic):
    ctx = _context((n,), N, p, flux, (periodic,))
    prob = dc.Problem(dim=1, n=(n,), N=N, p=p, periodic=(periodic,), flux=flux, c2=1.3)
    ops = dc.operators(prob)
    f = lambda t, U, V: dc.time_derivative(prob, U, V, ops)
    dt = 0.05 / (n * N)
    for steps in (1, 2, 5):
        u, v = _state((n,), N, 7)
        U, V = u.cpu().numpy().reshape(n, -1), v.cpu().numpy().reshape(n, -1)
        ctx.step(u, v, 0.0, dt, steps)
        for _ in range(steps):
            U, V = ti.rk4_step(f, U, V, 0.0, dt)
        assert _rel((u, v), (U, V)) < steps * TOL
    ctx.close()


def test_line_windows_agree_with_one_step_calls():
    """7 steps at once and one at a time, on a mesh with more windows than SMs."""
    n, N = 3001, 8
    ctx = _context((n,), N, 5, "upwind", (True,))
    u, v = _state((n,), N, 3)
    a, b = u.clone(), v.clone()
    dt = 0.05 / (n * N)
    ctx.step(u, v, 0.0, dt, 7)
    for _ in range(7):
        ctx.step(a, b, 0.0, dt, 1)
    assert _rel((u, v), (a, b)) < 7 * TOL
    ctx.close()


# 1 to 4 elements a block, a ragged last block, every flux and boundary, a mesh
# one element wide; N + 1 = 8, 9, 10 have this kernel, 7 and 11 do not
@pytest.mark.parametrize("flux,periodic", [("upwind", (False, False)), ("central", (True, False)),
                                           ("alternating", (False, True)), ("upwind", (True, True))])
@pytest.mark.parametrize("n,N,p", [((1, 1), 8, 5), ((1, 7), 8, 3), ((5, 3), 7, 7), ((21, 13), 7, 7), ((23, 17), 9, 3),
                                   ((37, 29), 8, 5), ((41, 37), 7, 5), ((9, 8), 6, 3)])
def test_persistent_step_equals_the_stage_kernels(n, N, p, flux, periodic):
    ctx = _context(n, N, p, flux, periodic)
    out = []
    for variant in (0, 3):
        u, v = _state(n, N, 11)
        ctx.set_stage_variant(variant)
        ctx.step(u, v, 0.0, 0.02 / (max(n) * N), 3)
        out.append((u, v))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    ctx.close()


@pytest.mark.parametrize("n,N,p", [((3, 2), 1, 1), ((2, 3), 2, 1), ((3, 3), 7, 3), ((2, 2), 8, 7), ((2, 1), 15, 7),
                                   ((2, 1, 3), 3, 3), ((1, 2, 2), 8, 5), ((2, 2, 1), 9, 7)])
def test_transforms_by_node_pairs(n, N, p):
    """gdg_mass_solve transforms to the modified basis and back; in place too."""
    ctx = _context(n, N, p, "upwind", (False,) * len(n))
    prob = dc.Problem(dim=len(n), n=n, N=N, p=p, periodic=(False,) * len(n), lo=(0.0,) * len(n), hi=(1.0,) * len(n), c2=1.3)
    M = np.ones((1, 1))
    for k in reversed(range(len(n))):
        M = np.kron(M, dc.operators(prob).M1[k])
    b, _ = _state(n, N, 5)
    want = np.linalg.solve(M, b.cpu().numpy().reshape(-1, M.shape[0]).T).T
    x = torch.empty_like(b)
    ctx.mass_solve(gdg.OP_M, b, x)
    # a solve rounds by the conditioning of M
    tol = max(TOL, 10 * np.linalg.cond(M) * np.finfo(float).eps)
    assert _rel((x,), (want,)) < tol
    ctx.mass_solve(gdg.OP_M, b, b)
    assert torch.equal(x, b)
    ctx.close()


@pytest.mark.parametrize("n", [(16,), (12, 9), (3, 2, 2)])
def test_step_sizes_of_a_captured_graph(n):
    """A captured step replayed between steps of another size, against contexts
    that see one size each."""
    N, dt = 8, (0.01 / (max(n) * 8), 0.02 / (max(n) * 8))
    ctx, plain = _context(n, N, 5, "upwind", (False,) * len(n)), _context(n, N, 5, "upwind", (False,) * len(n))
    u, v = _state(n, N, 5)
    a, b = u.clone(), v.clone()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        for w in (dt[0], dt[1], dt[0]):   # (the first call of a context times its kernels)
            ctx.step(u, v, 0.0, w, 1, stream=s)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            ctx.step(u, v, 0.0, dt[1], 1, stream=s)
        ctx.step(u, v, 0.0, dt[0], 1, stream=s)
        g.replay()
        ctx.step(u, v, 0.0, dt[0], 1, stream=s)
        s.synchronize()
    for w in (dt[0], dt[1], dt[0], dt[0], dt[1], dt[0]):
        plain.step(a, b, 0.0, w, 1)
    torch.cuda.synchronize()
    assert _rel((u, v), (a, b)) < 6 * TOL
    ctx.close()
    plain.close()
