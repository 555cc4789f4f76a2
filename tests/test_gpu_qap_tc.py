"""The tensor-core form of the QAP operator (autotune = 1, d >= 64) at the sizes where its tiling can go
wrong (one tile, partial tiles, one to several chunks of 64 k's per group), on iterates as they occur and on
hard ones: its distance to the product in extended precision is no larger than that of the FP64
contractions (autotune = 0), and the solve's iterates match the oracle's."""
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


def problem(d, seed, wide):
    """Symmetric matrices of the relaxation's kind; wide: entries over twelve orders of magnitude."""
    rng = np.random.default_rng(seed)
    F, D = qpgen.qap_matrices(d, seed)
    S, T = (rng.standard_normal((d, d)) for _ in range(2))
    if wide:
        S, T = S * 10.0 ** rng.integers(-12, 1, (d, d)), T * 10.0 ** rng.integers(-12, 1, (d, d))
    S, T = S + S.T, T + T.T
    if d == 65:
        F[3, :] = F[:, 3] = 0.0                        # a row without entries
    n = d * d
    e = np.zeros(0, np.int32)
    qp = qpgen.QP(n, 0, np.zeros(1, np.int32), e, np.zeros(0), np.zeros(n), np.zeros(0), np.zeros(0), np.zeros(n),
                  np.full(n, np.inf), 0, 0.0, [qpgen.QTerm("qap", p=d, dense=np.concatenate([F, D, S, T]).reshape(-1))])
    return qp, (F, D, S, T)


def exact(mats, x, d):
    F, D, S, T = (m.astype(np.longdouble) for m in mats)
    X = x.reshape(d, d).T.astype(np.longdouble)
    return (F @ X @ D - S @ X - X @ T).T.reshape(-1)


def vectors(d, rng):
    n = d * d
    yield "uniform", rng.random(n) / d
    yield "sparse", np.where(rng.random(n) < 0.03, rng.random(n), 0.0)
    yield "wide", rng.standard_normal(n) * 10.0 ** rng.integers(-10, 3, n)
    yield "one", np.eye(1, n, n // 3).reshape(-1)
    yield "zero", np.zeros(n)
    yield "tiny", rng.standard_normal(n) * 1e-290
    yield "subnormal", rng.standard_normal(n) * 1e-310


@pytest.mark.parametrize("d,wide", [(64, False), (65, False), (100, True), (128, False), (129, False), (191, True), (256, False), (330, False)])
def test_product_is_no_further_off(pkg, d, wide):
    qp, mats = problem(d, d, wide)
    with pkg.Solver(qp) as tc, pkg.Solver(qp, autotune=0) as fp:
        for name, x in vectors(d, np.random.default_rng(d)):
            a, b, e = tc.apply("Q", x), fp.apply("Q", x), exact(mats, x, d)
            scale = float(np.linalg.norm(e.astype(float)))
            if name in ("zero", "subnormal") or scale == 0.0:
                # entries below FP64's normal range count as 0
                assert float(np.max(np.abs(a - e))) <= 1e-300
                continue
            near = lambda v: float(np.linalg.norm((v - e).astype(float))) / scale  # noqa: E731
            assert near(a) <= max(near(b), 2.3e-16), (name, near(a), near(b))
        x = np.ones(d * d)
        x[d + 1] = np.nan
        assert np.isnan(tc.apply("Q", x)).any()


def test_iterates_and_objective(pkg):
    qp = qpgen.qap_relaxation(70, seed=2)
    ref = oracle.solve(qp, tol=1e-30, max_iter=120)
    lam = {"lambda_A": ref.lambda_A, "lambda_Q": ref.lambda_Q}
    with pkg.Solver(qp, **lam) as s:
        for k in (1, 11, 120):
            r = oracle.solve(qp, tol=1e-30, max_iter=k, **lam)
            s.solve(tol=1e-30, max_iter=k)
            for a, b in zip(s.get()[:4], (r.x, r.y, r.z, r.w)):
                assert close(a, b) <= 1e-10, k
    with pkg.Solver(qp) as s:
        s.solve(tol=1e-30, max_iter=1)
        assert abs(s.kkt()["lambda_Q"] - ref.lambda_Q) <= 1e-5 * ref.lambda_Q
