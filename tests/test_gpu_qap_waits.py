"""The tensor-core QAP product's bounded waits: a wait for operands that runs out (hprqp_set_wait_polls) ends a solve or
an apply with HPRQP_TIMEOUT, and the same handle then works as if nothing had happened."""
import numpy as np
import pytest

import qpgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2507_02470_gb300 as p
    p.build()
    return p


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_wait_that_runs_out(pkg, mode):
    qp = qpgen.qap_relaxation(70, seed=2)      # two chunks of k: a copy takes longer than one poll
    v = np.random.default_rng(0).standard_normal(qp.n)
    with pkg.Solver(qp, launch_mode=mode) as s:      # one handle: another may be tuned to other sums
        s.solve(tol=1e-30, max_iter=60)
        want, product = s.get()[:4], s.apply("Q", v)
        for _ in range(2):
            s.set_wait_polls(1)
            for call in (lambda: s.solve(tol=1e-30, max_iter=60), lambda: s.apply("Q", v)):
                with pytest.raises(pkg.HPRQPError) as e:
                    call()
                assert e.value.status == 6     # HPRQP_TIMEOUT
            s.set_wait_polls(0)
            assert np.array_equal(s.apply("Q", v), product)
            s.solve(tol=1e-30, max_iter=60)
            for a, b in zip(s.get()[:4], want):
                assert np.array_equal(a, b)
