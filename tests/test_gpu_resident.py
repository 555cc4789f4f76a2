"""The resident solver (the default launch mode of problems whose state fits the SMs' shared memory)
against the oracle and against the separate kernels (tiled_factor = 0 asks for their schedule), at the
sizes where its split can go wrong: one block, partial last blocks, the edge between the cluster and the
grid form, empty blocks of R^m, rows long enough for a whole block, several factors, no rows of A, and
runs in pieces.  Iterates agree to 1e-10 element by element (tests/parity.py), as everywhere else."""
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


def two_factors(n, m, seed):
    """Two sparse factors (one thin), two dense ones, a diagonal, a band and an explicit part."""
    rng = np.random.default_rng(seed)
    qp = qpgen.large_cqp(n=n, m=m, seed=seed, s_rows=max(1, n // 50))
    M = qpgen.csr_bernoulli(rng, max(2, n // 20), n, 0.05)
    qp.qterms.append(qpgen.QTerm("factor", p=max(2, n // 20), rowptr=M[0], colidx=M[1], vals=M[2]))
    for k in (3, 5):
        qp.qterms.append(qpgen.QTerm("dense_factor", p=k, dense=rng.standard_normal((k, n)) / np.sqrt(n)))
    qp.qterms.append(qpgen.QTerm("diag", dense=rng.uniform(0.1, 1.0, n)))
    i = np.arange(n, dtype=np.int32)
    qp.qterms.append(qpgen.QTerm("csr", rowptr=np.arange(n + 1, dtype=np.int32), colidx=i, vals=np.full(n, 0.25)))
    return qp


CASES = {
    "one_row": lambda: qpgen.random_small(n=1, m=1, seed=3, eq_rows=0),
    "n63": lambda: qpgen.large_cqp(n=63, m=20, seed=1),
    "n64": lambda: qpgen.large_cqp(n=64, m=64, seed=2),
    "n65_m1": lambda: qpgen.large_cqp(n=65, m=1, seed=3),
    "m_over_n": lambda: qpgen.large_cqp(n=130, m=300, seed=4),
    "factor": lambda: qpgen.plain_cqp(n=999, m=333, seed=5),
    "cluster_edge": lambda: qpgen.large_cqp(n=2560, m=700, seed=6),
    "grid_edge": lambda: qpgen.large_cqp(n=2561, m=700, seed=6),
    "grid": lambda: qpgen.large_cqp(n=20_011, m=3001, seed=7),
    "csr_scaled": lambda: qpgen.large_cqp(n=5003, m=1500, seed=8, q_as="csr"),
    "lasso": lambda: qpgen.lasso(p=301, q=1999, density=0.02, seed=9),
    "portfolio": lambda: qpgen.portfolio(10, n=701),
    "portfolio_long_rows": lambda: qpgen.portfolio(11, n=3001),
    "terms_cluster": lambda: two_factors(400, 90, 12),
    "terms_grid": lambda: two_factors(3100, 900, 13),
}


@pytest.mark.parametrize("name", list(CASES))
def test_resident_iterates(pkg, name):
    qp = CASES[name]()
    ref = oracle.solve(qp, tol=1e-30, max_iter=230)
    lam = {"lambda_A": ref.lambda_A if qp.m else 0.0, "lambda_Q": ref.lambda_Q}
    with pkg.Solver(qp) as s:                            # the power methods, in their resident form too
        s.solve(tol=1e-30, max_iter=1)
        kk = s.kkt()
        assert kk["kernel_launches"] == 3                # power methods, time stamp, the solve
        assert abs(kk["lambda_Q"] - ref.lambda_Q) <= 1e-5 * ref.lambda_Q
        assert not qp.m or abs(kk["lambda_A"] - ref.lambda_A) <= 1e-5 * ref.lambda_A
    with pkg.Solver(qp, **lam) as s:
        for k in (1, 11, 230):
            r = oracle.solve(qp, tol=1e-30, max_iter=k, **lam)
            s.solve(tol=1e-30, max_iter=k)
            got = s.get()[:4]
            for a, b in zip(got, (r.x, r.y, r.z, r.w)):
                assert close(a, b) <= 1e-10, (name, k)
        kk = s.kkt()
        assert kk["kernel_launches"] == 2 and kk["iters"] == 230
        # the tests of the restart rule compare differences of the size of rel-KKT: at a point that is exact
        # to a few roundings (one_row, n65_m1) they compare noise
        exact = max(ref.eta_p, ref.eta_d, ref.eta_gap) < 1e-12
        assert exact or kk["restarts"] == ref.restarts
    with pkg.Solver(qp, tiled_factor=0, **lam) as s:     # the separate kernels
        s.solve(tol=1e-30, max_iter=230)
        assert (exact or s.kkt()["restarts"] == ref.restarts) and s.kkt()["kernel_launches"] > 3
        for a, b in zip(got, s.get()[:4]):
            assert close(a, b) <= 1e-10, name


def test_resident_in_pieces_under_a_time_limit(pkg):
    """A time limit runs one check period per launch: the same iterates, bit for bit."""
    qp = qpgen.large_cqp(n=1500, m=500, seed=21)
    with pkg.Solver(qp) as s:
        s.solve(tol=1e-30, max_iter=450)
        whole, launches = s.get()[:4], s.kkt()["kernel_launches"]
    with pkg.Solver(qp, time_limit=1000.0) as s:
        s.solve(tol=1e-30, max_iter=450)
        assert s.kkt()["kernel_launches"] == launches + 4
        for a, b in zip(whole, s.get()[:4]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("kw", [{"sigma_golden": 1}, {"halpern_total": 1}, {"restart_off": 1}, {"sigma_fixed": 1},
                                {"restart_every": 7}, {"check_every": 1}, {"restart_every": 1}], ids=str)
def test_resident_options(pkg, kw):
    qp = qpgen.large_cqp(n=700, m=200, seed=22)
    ref = oracle.solve(qp, tol=1e-30, max_iter=120, **kw)
    with pkg.Solver(qp, lambda_A=ref.lambda_A, lambda_Q=ref.lambda_Q, **kw) as s:
        s.solve(tol=1e-30, max_iter=120)
        assert s.kkt()["kernel_launches"] == 2 and s.kkt()["restarts"] == ref.restarts
        for a, b in zip(s.get()[:3], (ref.x, ref.y, ref.z)):
            # golden section fixes sigma to about 1e-9 only
            assert close(a, b) <= (1e-7 if "sigma_golden" in kw else 1e-10)
