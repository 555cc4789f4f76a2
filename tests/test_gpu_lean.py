"""Problems that fit the device memory without the forms that take more of it than they need (the digits of a QAP term's
tensor-core product, the explicit entries of B^T B that factor_inline = 2 asks for) are created and solved
without them."""
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


def capped(base, cap):
    """The allocator of the binding, out of memory beyond `cap` bytes."""
    class Capped(base):
        def __init__(self):
            super().__init__()
            self.held, self.inner = {}, (self.alloc, self.free)

            def alloc(nbytes, ctx, stream):
                if sum(self.held.values()) + nbytes > cap:
                    return None
                p = self.inner[0](nbytes, ctx, stream)
                if p:
                    self.held[p] = nbytes
                return p

            def free(ptr, nbytes, ctx, stream):
                self.held.pop(ptr, None)
                self.inner[1](ptr, nbytes, ctx, stream)
            self.alloc, self.free = type(self.alloc)(alloc), type(self.free)(free)
    return Capped


def qap(d):
    qp = qpgen.qap_relaxation(d, seed=d)
    e = np.zeros(0, np.int32)
    return qpgen.QP(qp.n, 0, np.zeros(1, np.int32), e, np.zeros(0), -np.ones(qp.n), np.zeros(0), np.zeros(0),
                    np.zeros(qp.n), np.ones(qp.n), 0, 0.0, qp.qterms)


def factor():
    rng = np.random.default_rng(3)
    n, p = 9000, 2000
    rp, ci, v = qpgen.csr_k_per_row(rng, p, n, 40)
    e = np.zeros(0, np.int32)
    return qpgen.QP(n, 0, np.zeros(1, np.int32), e, np.zeros(0), -np.ones(n), np.zeros(0), np.zeros(0), np.zeros(n),
                    np.ones(n), 0, 0.0, [qpgen.QTerm("factor", p=p, rowptr=rp, colidx=ci, vals=v)])


@pytest.mark.parametrize("qp,more,less", [(qap(40), {}, {"autotune": 0}),
                                          (factor(), {"factor_inline": 2, "tiled_factor": 0},
                                           {"factor_inline": 0, "tiled_factor": 0})], ids=["qap", "factor"])
def test_created_without(pkg, monkeypatch, qp, more, less):
    from paper_2507_02470_gb300 import _lib as L
    with pkg.Solver(qp, torch_alloc=True, **more) as s:
        most = s.memory_stats()["hook_bytes"]
    with pkg.Solver(qp, torch_alloc=True, **less) as s:
        least = s.memory_stats()["hook_bytes"]
    assert least < most
    ref = oracle.solve(qp, tol=1e-30, max_iter=40)
    base = L._TorchAllocator
    monkeypatch.setattr(L, "_TorchAllocator", capped(base, least))
    with pkg.Solver(qp, torch_alloc=True, lambda_Q=ref.lambda_Q, **more) as s:
        s.solve(tol=1e-30, max_iter=40)
        assert close(s.get()[0], ref.x) <= 1e-10
        assert s.memory_stats()["hook_bytes"] <= least
    monkeypatch.setattr(L, "_TorchAllocator", capped(base, least // 2))
    with pytest.raises(pkg.HPRQPError) as e:
        pkg.Solver(qp, torch_alloc=True, **more)
    assert e.value.status == 7                          # HPRQP_OOM
