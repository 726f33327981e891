"""Nodes to modes and back on integers with a block exponent an element: a step
of negligible length is the round trip.  Tolerance, against the largest entry of
the element: each of the 2 dim passes rounds by N + 4 units of 2^-57 of its
largest entry at most (its inputs' limbs, the table's, the products of low
limbs), carried through at most the norms of the tables that follow; twice that
allows the modes' rounding to doubles in between."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import gd_basis as gb
from paper_2105_01722_gb300 import gdg, inputs


def _tol(N, p, dim):
    M, S = gb.mass_stiffness(p, N)
    Psi, _ = gb.simultaneous_diagonalisation(M, S)
    norm = lambda A: np.abs(A).sum(axis=1).max()
    return 2 * 2 * dim * (N + 4) * 2.0 ** -57 * (norm(Psi) * norm(Psi.T @ M)) ** dim


def _round_trip(n, N, p, u, v):
    ctx = gdg.Context(gdg.make_problem(len(n), n, N, p, hi=(1.0,) * len(n), lo=(0.0,) * len(n),
                                       bc=(gdg.BC_DIRICHLET,) * len(n)))
    a, b = (torch.tensor(x.ravel(), device="cuda") for x in (u, v))
    ctx.step(a, b, 0.0, 1e-300, 1)
    ctx.close()
    return a.cpu().numpy().reshape(u.shape), b.cpu().numpy().reshape(v.shape)


# odd and even line lengths; one element, a ragged last block, more elements than a block
@pytest.mark.parametrize("n", [(1, 1), (5, 3), (61, 37), (1, 1, 1), (3, 2, 5)])
@pytest.mark.parametrize("N,p", [(1, 1), (2, 1), (3, 3), (6, 5), (7, 3), (8, 5), (9, 7), (12, 5), (15, 7)])
def test_round_trip(n, N, p):
    if len(n) == 3 and N > 9:
        pytest.skip("3-D elements end at N = 9")
    shape = (int(np.prod(n)), (N + 1) ** len(n))
    scale = 10.0 ** np.random.default_rng(N).integers(-150, 100, size=(shape[0], 1))   # every element its own
    u, v = inputs.random_state(shape, 5) * scale, inputs.random_state(shape, 6) * scale
    u[shape[0] // 2] = 0.0
    got = _round_trip(n, N, p, u, v)
    big = np.maximum(np.abs(u).max(axis=1), np.abs(v).max(axis=1))[:, None]
    for x, y in zip(got, (u, v)):
        assert (np.abs(x - y) <= _tol(N, p, len(n)) * big).all()
    assert np.abs(got[0][shape[0] // 2]).max() < 1e-190   # zero but for the step itself


@pytest.mark.parametrize("n", [(4, 3), (2, 3, 2)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_not_finite(n, bad):
    N = 8
    shape = (int(np.prod(n)), (N + 1) ** len(n))
    u, v = inputs.random_state(shape, 5), inputs.random_state(shape, 6)
    u[1, 7] = bad
    x, _ = _round_trip(n, N, 5, u, v)
    assert not np.isfinite(x[1]).any()
