"""The resident solver's bounded waits: a grid barrier whose wait runs out (hprqp_set_wait_polls) ends the solve,
or the power methods before it, with HPRQP_TIMEOUT, and the same handle then solves as if nothing had
happened."""
import numpy as np
import pytest

import oracle
import qpgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2507_02470_gb300 as p
    p.build()
    return p


@pytest.mark.parametrize("given", [True, False], ids=["solve", "power_methods"])
@pytest.mark.parametrize("m", [0, 3001])
def test_wait_that_runs_out(pkg, given, m):
    qp = qpgen.large_cqp(n=20_011, m=m, seed=7)      # 152 blocks: some wait for longer than one poll
    lam = {}
    if given:
        r = oracle.solve(qp, tol=1e-30, max_iter=1)
        lam = {"lambda_A": r.lambda_A if m else 0.0, "lambda_Q": r.lambda_Q}
    with pkg.Solver(qp, **lam) as s:
        s.solve(tol=1e-30, max_iter=200)
        want = s.get()[:4]
    with pkg.Solver(qp, **lam) as s:
        for _ in range(2):
            s.set_wait_polls(1)
            with pytest.raises(pkg.HPRQPError) as e:
                s.solve(tol=1e-30, max_iter=200)
            assert e.value.status == 6                 # HPRQP_TIMEOUT
            s.set_wait_polls(0)
            s.solve(tol=1e-30, max_iter=200)
            for a, b in zip(s.get()[:4], want):
                assert np.array_equal(a, b)
