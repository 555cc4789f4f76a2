"""The batched solver's product with the nonzero coordinates of xbar, where its list can go wrong: partial
words of 32 coordinates, all, few or no coordinates at 0, the edge of n / 8, more coordinates than the list
or its words hold, no rows of A, a warm start.  First iterates match the oracle to 1e-10."""
import numpy as np
import pytest

import oracle
import qpgen
from tests.parity import close

pytestmark = pytest.mark.gpu


def instance(n, p, m, box, seed, phi="box", lam=0.0, linear=1.0):
    rng = np.random.default_rng(seed)
    A = qpgen.csr_bernoulli(rng, m, n, 0.3) if m else (np.zeros(1, np.int32), np.zeros(0, np.int32), np.zeros(0))
    x0 = rng.uniform(max(box[0], -1.0), min(box[1], 1.0), n)
    Ax = qpgen._csr_matvec(*A, x0) if m else np.zeros(0)
    l = Ax - 0.5
    u = Ax + 0.5
    if m:
        l[0] = u[0] = Ax[0]
    terms = [qpgen.QTerm("dense_factor", p=p, dense=rng.standard_normal((p, n)) / np.sqrt(n)),
             qpgen.QTerm("diag", dense=rng.uniform(0.05, 0.5, n))]
    return qpgen.QP(n, m, *A, linear * rng.standard_normal(n), l, u, np.full(n, box[0]), np.full(n, box[1]),
                    qpgen._PHI_NAMES[phi], lam, terms)


def batch():
    return [instance(31, 5, 2, (0.0, 0.1), 1), instance(32, 6, 3, (-1.0, 1.0), 2), instance(33, 7, 1, (0.0, 5.0), 3),
            instance(97, 9, 0, (0.0, 1.0), 4), instance(640, 20, 5, (0.0, 0.1), 5, linear=0.01),
            instance(800, 33, 11, (0.0, 1.0), 6, phi="l1_box", lam=0.8), instance(1601, 40, 4, (-5.0, 5.0), 7, phi="l1", lam=1.5),
            instance(5200, 8, 3, (0.0, 0.5), 8), instance(5200, 12, 2, (0.0, 0.5), 9, linear=-1.0),
            instance(16_400, 5, 2, (0.0, 0.2), 10), qpgen.portfolio(3, n=1237), qpgen.portfolio(4, n=257)]


@pytest.mark.parametrize("kw", [{}, {"autotune": 0}, {"batch_team": 64}, {"batch_team": 512}], ids=str)
def test_first_iterates(kw):
    import paper_2507_02470_gb300 as p
    p.build()
    probs = batch()
    refs = [oracle.solve(q, tol=1e-30, max_iter=60) for q in probs]
    warm = [None] * len(probs)
    warm[4] = np.linspace(0.0, 0.1, probs[4].n)
    refs[4] = oracle.solve(probs[4], tol=1e-30, max_iter=60, x0=warm[4], lambda_A=refs[4].lambda_A, lambda_Q=refs[4].lambda_Q)
    with p.BatchSolver(probs, x0=warm, lambda_A=[r.lambda_A for r in refs], lambda_Q=[r.lambda_Q for r in refs], **kw) as b:
        b.solve(tol=1e-30, max_iter=60)
        for i, r in enumerate(refs):
            x, y, z, k = b.get(i)
            assert k["iters"] == 60
            for a, w in zip((x, y, z), (r.x, r.y, r.z)):
                assert close(a, w) <= 1e-10, (i, probs[i].n)
