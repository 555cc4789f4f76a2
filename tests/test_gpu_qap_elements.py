"""The tensor-core form of the QAP operator (autotune = 1, d >= 8), element by element, on data whose rows and
columns span more than the digits hold: every element is within the bound of an FP64 evaluation,
(4 d + 4) 2^-53 (|Ahat| |X| |Bhat| + |S| |X| + |X| |T|)_ij (d products and sums in T1, 3 d in the result), and NaN
and infinities lie where the FP64 contractions (autotune = 0) have them."""
import numpy as np
import pytest

import qpgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2507_02470_gb300 as p
    p.build()
    return p


def problem(mats):
    d = mats[0].shape[0]
    n, e = d * d, np.zeros(0, np.int32)
    return qpgen.QP(n, 0, np.zeros(1, np.int32), e, np.zeros(0), np.zeros(n), np.zeros(0), np.zeros(0), np.zeros(n),
                    np.full(n, np.inf), 0, 0.0,
                    [qpgen.QTerm("qap", p=d, dense=np.concatenate(mats).reshape(-1))])


def sym(M):
    return np.triu(M) + np.triu(M, 1).T


def graded(kind, d, rng):
    """(Ahat, Bhat, S, T), X"""
    A, B = (sym(rng.random((d, d))) for _ in range(2))
    S, T = (sym(rng.standard_normal((d, d))) for _ in range(2))
    X = rng.standard_normal((d, d))
    if kind == "column":          # X T with T diagonal and one small column of X, nothing beside it
        A, S, T = 0.0 * A, 0.0 * S, np.diag(1.0 + rng.random(d))
        X[:, d // 2] *= 1e-12
    elif kind == "spike":         # a huge entry of S (of Ahat) meets a zero of X
        S[3, 5] = S[5, 3] = 1e18
        A[2, 6] = A[6, 2] = 1e20
        X[[5, 3, 2, 6], : d // 2] = 0.0
    elif kind == "wide":
        A, B, S, T = (sym(M * 10.0 ** rng.integers(-20, 1, (d, d))) for M in (A, B, S, T))
        X *= 10.0 ** rng.integers(-20, 1, (d, d))
    elif kind == "cancel":        # sums of terms that cancel to their rounding
        X[1::2][: d // 2] = -X[0::2][: d // 2]
        A[:, 1::2][:, : d // 2] = A[:, 0::2][:, : d // 2]
        A = sym(A)
    elif kind == "subnormal":     # neighbours of the smallest normal number
        A, B, S, T = (np.round(8 * M) for M in (A, B, S, T))
        X = np.ldexp(rng.random((d, d)), rng.integers(-1030, -1015, (d, d)))
    return (A, B, S, T), X


@pytest.mark.parametrize("kind", ["column", "spike", "wide", "cancel", "subnormal"])
@pytest.mark.parametrize("d", [8, 9, 64, 65, 129, 200])
def test_every_element(pkg, d, kind):
    mats, X = graded(kind, d, np.random.default_rng(d))
    with pkg.Solver(problem(mats)) as s:
        out = s.apply("Q", X.T.reshape(-1)).reshape(d, d).T
        again = s.apply("Q", X.T.reshape(-1)).reshape(d, d).T
    assert np.array_equal(out, again)
    A, B, S, T, Xl = (M.astype(np.longdouble) for M in (*mats, X))
    exact = A @ Xl @ B - S @ Xl - Xl @ T
    size = abs(A) @ abs(Xl) @ abs(B) + abs(S) @ abs(Xl) + abs(Xl) @ abs(T)
    # a product of two numbers near the smallest normal one may round by 2^-1074: d + 3 d of them
    bound = (4 * d + 4) * 2.0 ** -53 * size + 4 * d * np.longdouble(2.0) ** -1074 * (1 + abs(B).sum(axis=0))
    worst = np.unravel_index(np.argmax(abs(out - exact) - bound), (d, d))
    assert (abs(out - exact) <= bound).all(), (worst, out[worst], exact[worst], bound[worst])


@pytest.mark.parametrize("d", [9, 100])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_not_finite(pkg, d, bad):
    mats, X = graded("plain", d, np.random.default_rng(1))
    mats[2][4, :] = mats[2][:, 4] = 0.0
    X[d // 2, 4] = bad
    with pkg.Solver(problem(mats)) as s, pkg.Solver(problem(mats), autotune=0) as f:
        a, b = s.apply("Q", X.T.reshape(-1)), f.apply("Q", X.T.reshape(-1))
    fin = np.isfinite(b)
    assert np.array_equal(np.isfinite(a), fin) and np.array_equal(np.isnan(a), np.isnan(b))
    assert np.array_equal(a[~fin & ~np.isnan(a)], b[~fin & ~np.isnan(b)])
