"""The fixed-point products of gdg_fx.cuh restated in Python integers: how far they are
from 80-bit sums, against FP64 sums of the same terms, on the element matrices and
inverses of mapped elements.  (A model of the scheme, no GPU.)"""
import numpy as np
import pytest

from oracle import dg_var as dv
from paper_2105_01722_gb300 import inputs

LD = np.longdouble
if np.finfo(LD).nmant < 60:
    pytest.skip("needs an extended long double", allow_module_level=True)


def integers(a):
    return np.vectorize(int, otypes=[object])(np.rint(a))


def fixed_point(A, x, nearest=True):
    """A x with A_ij = 2^(d_i + d_j) a_ij 2^-57 and x_j 2^d_j = X_j 2^(E - 57), the exact sums
    rounded once, in units of 2^58."""
    d = -((-np.frexp(np.diag(A))[1]) // 2)
    a = integers(np.ldexp(A, 57 - d[:, None] - d[None, :]))
    assert max(abs(v) for v in a.ravel()) <= 1 << 57
    scaled = np.ldexp(x, d)
    E = np.frexp(np.abs(scaled).max())[1]
    X = integers(np.ldexp(scaled, 57 - E))
    T = np.array([float((int(v) + ((1 << 57) if nearest else 0)) >> 58) for v in a @ X])
    return np.ldexp(T, 58 - 57 - 57 + E + d)


def fp64(A, x):
    """Row sums by FP64 multiply-adds (each rounded once)."""
    s = np.zeros(len(x))
    for k in range(len(x)):
        s = (A[:, k].astype(LD) * LD(x[k]) + s).astype(np.float64)
    return s


def cholesky_inverse(A):
    n = len(A)
    L, Li = np.linalg.cholesky(A), np.zeros_like(A)
    for i in range(n):
        Li[i] = (np.eye(n)[i] - L[i, :i] @ Li[:i]) / L[i, i]
    return Li.T @ Li


def element_matrices(N, p, c2):
    n = (4, 4)
    X, Y = inputs.mapped_nodes(n, N, 0.05)
    ops = dv.assemble(dv.VarProblem(n=n, N=N, p=p, X=X, Y=Y, C2=inputs.c2_sine(X, Y) * c2))
    sym = lambda A: np.tril(A) + np.tril(A, -1).T  # noqa: E731
    for e in (0, 5, 10):
        S, M, w = sym(ops.S[e]), sym(ops.M[e]), ops.w[e]
        sigma = 2.0 ** np.floor(np.log2(np.trace(S)))
        yield {"S": S, "M": M, "A": sym(cholesky_inverse(S + sigma * np.outer(w, w))) - 1 / sigma, "V": sym(cholesky_inverse(M))}


def vectors(kind, N, rng):
    s, t = np.meshgrid(np.arange(N + 1) / N, np.arange(N + 1) / N)
    for _ in range(6):
        a, b, c = rng.uniform(0, 6), rng.uniform(0, 6), rng.uniform(-0.2, 1.2, 2)
        if kind == "random":
            yield rng.standard_normal((N + 1) ** 2)
        elif kind == "smooth":
            yield (np.sin(2 * s + a) * np.cos(t + b) + rng.uniform(-1, 1)).ravel()
        else:
            yield np.exp(-10 * ((s - c[0]) ** 2 + (t - c[1]) ** 2)).ravel()


@pytest.mark.parametrize("N,p", [(4, 3), (6, 3), (8, 3), (8, 5), (9, 7), (9, 1)])
@pytest.mark.parametrize("c2", [1.0, 1e6])
def test_products_are_as_accurate_as_fp64_sums(N, p, c2):
    """2-norm errors of the products over the FP64 sums': on average (geometric mean) at most 1 for
    every matrix and kind of vector."""
    rng = np.random.default_rng(5)
    ratios = {}
    for matrices in element_matrices(N, p, c2):
        for name, A in matrices.items():
            for kind in ("random", "smooth", "pulse"):
                for x in vectors(kind, N, rng):
                    truth = A.astype(LD) @ x.astype(LD)
                    err = [np.linalg.norm((y - truth).astype(np.float64)) for y in (fixed_point(A, x), fp64(A, x))]
                    ratios.setdefault((name, kind), []).append(err[0] / err[1])
    for key, r in ratios.items():
        assert np.exp(np.mean(np.log(r))) <= 1.0, key


def test_rounding_is_to_nearest():
    """Sums of the errors over an element: no drift to one side (as cut-off sums have it)."""
    rng = np.random.default_rng(6)
    S = next(element_matrices(8, 5, 1.0))["S"]
    unit = np.abs(S).max() * 2.0**-53
    sums = {True: [], False: []}
    for _ in range(40):
        x = rng.standard_normal(81)
        truth = S.astype(LD) @ x.astype(LD)
        for nearest in sums:
            sums[nearest].append(float(np.sum(fixed_point(S, x, nearest) - truth)) / unit)
    # 81 roundings of at most 2^-57 of the row's scale each way against as many of half a unit downwards
    assert abs(np.mean(sums[True])) < 4 * np.std(sums[True]) / np.sqrt(40)
    assert np.mean(sums[False]) < -4 * np.std(sums[False]) / np.sqrt(40)
