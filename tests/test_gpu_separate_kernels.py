"""The separate kernels at the sizes that the resident solver and the tensor-core QAP product take by default: the
autotuned graphs with fused passes (tiled_factor = 0 asks for them and changes nothing else where no factor is
tiled), step by step against the oracle's trace, and the FP64 contractions of the QAP operator
(autotune = 0) with ragged tiles and split K ranges.  Iterates agree to 1e-10, operator products to 1e-13
(tests/parity.py), as everywhere else."""
import numpy as np
import pytest

import oracle
import qpgen
from tests.parity import close
from tests.test_gpu_parity import PROBLEMS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2507_02470_gb300 as p
    p.build()
    return p


@pytest.mark.parametrize("name", list(PROBLEMS))
def test_graphs(pkg, name):
    qp = PROBLEMS[name]
    K = 300
    ref = oracle.solve(qp, tol=1e-30, max_iter=K, trace_len=K)
    lam = {"lambda_A": ref.lambda_A if qp.m else 0.0, "lambda_Q": ref.lambda_Q}
    with pkg.Solver(qp, tiled_factor=0, **lam) as s:
        for k in (1, 2, 3, 10, 11, 20, 21, 33, 50, 100, 101, 200, 300):
            s.solve(tol=1e-30, max_iter=k)
            x, y, z, w, kkt = s.get()
            assert kkt["iters"] == k and kkt["tiled_terms"] == 0
            assert kkt["kernel_launches"] >= 2 * k          # not the one launch of the resident solver
            assert close(x, ref.trace["x"][k - 1]) <= 1e-10, k
            if qp.qterms:
                assert close(w, ref.trace["w"][k - 1]) <= 1e-10, k
            if qp.m:
                assert close(y, ref.trace["y"][k - 1]) <= 1e-10, k


@pytest.mark.parametrize("d", [3, 7, 8, 31, 50, 65, 200])
def test_qap_contractions(pkg, d):
    qp = qpgen.qap_relaxation(d=d, seed=d)
    v = np.random.default_rng(d).standard_normal(qp.n)
    ref = oracle.qmul(qp, v)
    with pkg.Solver(qp, autotune=0) as s:
        out, again = s.apply("Q", v), s.apply("Q", v)
    assert close(out, ref) <= 1e-13, close(out, ref)
    assert np.array_equal(out, again)


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("d", [7, 12, 40])
def test_qap_iterates_with_contractions(pkg, d, mode):
    qp = qpgen.qap_relaxation(d=d, seed=d)
    ref = oracle.solve(qp, tol=1e-30, max_iter=120, trace_len=120)
    with pkg.Solver(qp, lambda_A=ref.lambda_A, lambda_Q=ref.lambda_Q, launch_mode=mode, autotune=0) as s:
        for k in (1, 2, 11, 21, 120):
            s.solve(tol=1e-30, max_iter=k)
            x, y, *_ = s.get()
            assert close(x, ref.trace["x"][k - 1]) <= 1e-10, k
            assert close(y, ref.trace["y"][k - 1]) <= 1e-10, k
