"""The explicit entries of thin factor terms (sum_f B_f^T B_f as one CSR matrix, formed on the device) and the
device scan behind them and behind the stored transposes, at the scan's tile edges (4096 elements), with
empty rows and columns, repeated columns in a row, several terms, and an empty term."""
import numpy as np
import pytest

import oracle
import qpgen
from tests.parity import close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2507_02470_gb300 as p
    p.build()
    return p


def factor(rng, p, n, longest):
    """p rows of 0 .. longest entries, columns drawn with repetition from the lower two thirds of n."""
    rp = np.concatenate([[0], np.cumsum(rng.integers(0, longest + 1, p))]).astype(np.int32)
    ci = rng.integers(0, max(1, 2 * n // 3), rp[-1]).astype(np.int32)
    return qpgen.QTerm("factor", p=p, rowptr=rp, colidx=ci, vals=rng.standard_normal(rp[-1]) / 2)


@pytest.mark.parametrize("n,rows", [(1, (1,)), (5, (3, 2)), (700, (4096, 1)), (3000, (2050, 300, 40)),
                                    (9001, (8200, 5))])
def test_thin_terms_iterate_like_the_oracle(pkg, n, rows):
    """factor_inline = 2 takes every factor as explicit entries; iterates agree to 1e-10 element by element, the
    bound of every iterate test."""
    rng = np.random.default_rng(n)
    qp = qpgen.large_cqp(n=n, m=max(1, n // 3), seed=n) if n > 5 else qpgen.random_small(n=n, m=1, seed=3, eq_rows=0)
    qp.qterms += [factor(rng, p, n, 4) for p in rows][:4 - sum(t.kind == "factor" for t in qp.qterms)]
    lam = oracle.solve(qp, tol=1e-30, max_iter=1)
    lam = {"lambda_A": lam.lambda_A, "lambda_Q": lam.lambda_Q}
    ref = oracle.solve(qp, tol=1e-30, max_iter=40, **lam)
    with pkg.Solver(qp, factor_inline=2, **lam) as s:
        s.solve(tol=1e-30, max_iter=40)
        for a, b in zip(s.get()[:4], (ref.x, ref.y, ref.z, ref.w)):
            assert close(a, b) <= 1e-10


@pytest.mark.parametrize("n", [1, 4094, 4095, 4096, 8191, 8192, 12_289])
def test_transposes_at_the_scan_edges(pkg, n):
    """A^T y against the entries summed on the host: no further apart than the roundings of the longest row
    (its length times 2^-52, relative to the sum of magnitudes), and exactly 0 in an empty row."""
    rng = np.random.default_rng(n)
    m = 600
    qp = qpgen.large_cqp(n=max(n, 2), m=m, seed=1) if n > 1 else qpgen.random_small(n=1, m=1, seed=3, eq_rows=0)
    if n > 1:
        rp = np.concatenate([[0], np.cumsum(rng.integers(0, 12, m))]).astype(np.int32)
        qp.A_rowptr, qp.A_colidx = rp, rng.integers(0, n, rp[-1]).astype(np.int32)
        qp.A_vals = rng.standard_normal(rp[-1])
    y = rng.standard_normal(qp.m)
    terms = qp.A_vals * np.repeat(y, np.diff(qp.A_rowptr))
    want = np.bincount(qp.A_colidx, weights=terms, minlength=n)
    size = np.bincount(qp.A_colidx, weights=np.abs(terms), minlength=n)
    longest = np.bincount(qp.A_colidx, minlength=n).max()
    with pkg.Solver(qp, scaling=0) as s:
        got = s.apply("AT", y)
    assert np.all(np.abs(got - want) <= (longest + 1) * 2.0 ** -52 * size)
