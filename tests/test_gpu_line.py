"""1-D steps on both sides of the rule that picks windows (k_run1) or stages: a long mesh near its
ends, and a periodic one, move as a short mesh with the same elements does."""
import numpy as np
import pytest

from paper_2105_01722_gb300 import gdg, inputs

pytestmark = pytest.mark.gpu

FLUXES = [gdg.FLUX_UPWIND, gdg.FLUX_CENTRAL, gdg.FLUX_ALTERNATING]


def _gpu(a):
    import torch
    return torch.tensor(np.ascontiguousarray(a).ravel(), device="cuda")


def _run(n, N, p, u, v, steps, dt, **kw):
    ctx = gdg.Context(gdg.make_problem(1, (n,), N, p, hi=(0.01 * n,), c2=1.3, **kw))
    u, v = _gpu(u), _gpu(v)
    ctx.step(u, v, 0.0, dt, steps)
    ctx.close()
    return u.cpu().numpy().reshape(n, N + 1), v.cpu().numpy().reshape(n, N + 1)


# 152 SMs: the last mesh of one wave of windows and the first beyond (N1 = 16: of two waves), and far beyond
SIZES = [(1, 1, 75392), (1, 1, 75393), (4, 3, 28577), (8, 5, 14744), (8, 5, 14745), (8, 5, 40001), (11, 5, 20977), (15, 7, 14593), (15, 7, 60000)]


@pytest.mark.parametrize("N,p,n", SIZES)
@pytest.mark.parametrize("steps", [1, 3, 18])       # 18: a graph of 16 and two more
def test_ends_of_a_long_mesh(N, p, n, steps):
    """A stage carries information one element far: 4 steps elements from a cut 4 steps + 1 away from
    the end, the end is that of a mesh of 200 elements.  Both within the rounding of two transforms."""
    flux = FLUXES[steps % 3]
    dt = 0.1 * 0.01 / N / np.sqrt(1.3)
    u, v = inputs.random_state((n, N + 1), 1), inputs.random_state((n, N + 1), 2)
    got = _run(n, N, p, u, v, steps, dt, flux=flux)
    for part, keep in ((slice(0, 200), slice(0, 100)), (slice(n - 200, n), slice(100, 200))):
        want = _run(200, N, p, u[part], v[part], steps, dt, flux=flux)
        for a, b in zip(got, want):
            assert np.abs(a[part][keep] - b[keep]).max() <= 2e-13 * np.abs(b).max()


@pytest.mark.parametrize("N,p,n", [(2, 1, 64000), (8, 5, 14720), (8, 5, 40000), (15, 7, 32000)])
@pytest.mark.parametrize("flux", FLUXES)
def test_periodic_mesh_of_equal_pieces(N, p, n, flux):
    """A state that repeats every 20 elements stays one, equal to that of 20 periodic elements."""
    dt = 0.1 * 0.01 / N / np.sqrt(1.3)
    u, v = inputs.random_state((20, N + 1), 1), inputs.random_state((20, N + 1), 2)
    want = _run(20, N, p, u, v, 5, dt, flux=flux, bc=(gdg.BC_PERIODIC,))
    got = _run(n, N, p, np.tile(u, (n // 20, 1)), np.tile(v, (n // 20, 1)), 5, dt, flux=flux, bc=(gdg.BC_PERIODIC,))
    for a, b in zip(got, want):
        assert np.abs(a.reshape(n // 20, 20, N + 1) - b).max() <= 2e-13 * np.abs(b).max()


@pytest.mark.parametrize("n", [1000, 14745, 40001])
@pytest.mark.parametrize("warm", [False, True])
def test_captured_steps(n, warm):
    """A call inside a caller's capture, also a context's first one and more steps than the library's own
    graph has, replays to the bits of the call outside."""
    import torch
    problem = lambda: gdg.make_problem(1, (n,), 8, 5)  # noqa: E731
    u0, v0 = (_gpu(inputs.random_state((n, 9), k)) for k in (1, 2))
    ctx = gdg.Context(problem())
    want = u0.clone(), v0.clone()
    ctx.step(*want, 0.0, 1e-6, 18)
    if not warm:
        ctx.close()
        ctx = gdg.Context(problem())
    u, v = u0.clone(), v0.clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.step(u, v, 0.0, 1e-6, 18)
    u.copy_(u0)
    v.copy_(v0)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(u, want[0]) and torch.equal(v, want[1])
    ctx.close()
