"""The resident solver on problems without rows of A (m = 0).  A step then has no exchange behind its
products: the next wbar_{1/2} must not meet a block that still gathers the present one (explicit Q, bands,
thin factors; a long factor is gathered behind its own exchange).  Cluster and grid form, with and without
preconditioning; blocks of very uneven work, so that some run ahead.  Iterates agree with the oracle's to
1e-10 element by element (tests/parity.py), and repeated solves give the same bits."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
import qpgen
from tests.parity import close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2507_02470_gb300 as p
    p.build()
    return p


def box(n, terms, seed):
    rng = np.random.default_rng(seed)
    e = np.zeros(0, np.int32)
    return qpgen.QP(n, 0, np.zeros(1, np.int32), e, np.zeros(0), 2.0 * rng.standard_normal(n), np.zeros(0), np.zeros(0),
                    np.full(n, -1.0), np.full(n, 2.0), qpgen.PHI_BOX, 0.0, terms)


def uneven(n, seed):
    """An explicit Q whose first and last rows are long: three full rows beside rows of a few entries."""
    rng = np.random.default_rng(seed)
    M = sp.lil_matrix((n, n))
    for i in (0, n // 3, n - 1):
        M[i, :] = rng.standard_normal(n) * 0.3 / np.sqrt(n)
    M = sp.csr_matrix(M) + sp.random(n, n, 2.0 / n, random_state=seed, data_rvs=rng.standard_normal)
    M = M + M.T
    M = M + sp.diags(np.asarray(abs(M).sum(1)).reshape(-1) + 0.1)
    rp, ci, v = qpgen.csr_from_scipy(M)
    return qpgen.QTerm("csr", rowptr=rp, colidx=ci, vals=v)


def thin(n, seed):
    rp, ci, v = qpgen.csr_k_per_row(np.random.default_rng(seed), max(1, n // 40), n, 4)
    return qpgen.QTerm("factor", p=max(1, n // 40), rowptr=rp, colidx=ci, vals=v)


def long_factor(n, seed):
    p = max(4, n // 30)
    rp, ci, v = qpgen.csr_k_per_row(np.random.default_rng(seed), p, n, min(n // 8, 40), 0.2)
    return qpgen.QTerm("factor", p=p, rowptr=rp, colidx=ci, vals=v)


def diag(n, seed):
    return qpgen.QTerm("diag", dense=np.random.default_rng(seed).uniform(0.05, 1.0, n))


KINDS = {
    "explicit": lambda n: [uneven(n, n)],
    "band": lambda n: [qpgen.pentadiag_terms(np.random.default_rng(n), n)],
    "thin": lambda n: [diag(n, n), thin(n, n + 1)],
    "band_and_long_factor": lambda n: [qpgen.pentadiag_terms(np.random.default_rng(n), n), long_factor(n, n)],
    "all": lambda n: [uneven(n, n), qpgen.pentadiag_terms(np.random.default_rng(n), n), thin(n, n + 1), long_factor(n, n + 2)],
}


@pytest.mark.parametrize("n", [65, 700, 2561, 9001])    # cluster: 2 and 16 blocks; grid: 41 and 141 blocks
@pytest.mark.parametrize("kind,kw", [(k, {}) for k in KINDS] + [("explicit", {"scaling": 0})], ids=str)
def test_iterates_without_rows(pkg, kind, kw, n):
    qp = box(n, KINDS[kind](n), n)
    ref = oracle.solve(qp, tol=1e-30, max_iter=230, trace_len=230, **kw)
    with pkg.Solver(qp, lambda_Q=ref.lambda_Q, **kw) as s:
        for k in (1, 2, 11, 230):
            s.solve(tol=1e-30, max_iter=k)
            got = s.get()[:4]
            assert close(got[0], ref.trace["x"][k - 1]) <= 1e-10 and close(got[3], ref.trace["w"][k - 1]) <= 1e-10, k
        for a, b in zip(got, (ref.x, ref.y, ref.z, ref.w)):
            assert close(a, b) <= 1e-10
        assert s.kkt()["kernel_launches"] == 2           # the resident form: time stamp, the solve
        for _ in range(4):
            s.solve(tol=1e-30, max_iter=230)
            for a, b in zip(s.get()[:4], got):
                assert np.array_equal(a, b)
    with pkg.Solver(qp, lambda_Q=ref.lambda_Q, time_limit=1000.0, check_every=15, **kw) as s:   # in pieces of odd length
        s.solve(tol=1e-30, max_iter=230)
        for a, b in zip(s.get()[:4], got):
            assert np.array_equal(a, b)
