"""predict holds no memory for the decoder's product, which stays on chip: beyond its results, the BF16 members and
the network's output it takes less than the D x B FP32 product alone would."""
import numpy as np
import pytest

import qpgen

pytestmark = pytest.mark.gpu


def test_predict_takes_no_product():
    torch = pytest.importorskip("torch")
    import paper_2507_02470_gb300 as p
    p.build()
    from paper_2507_02470_gb300 import learned as L
    base = qpgen.param_family_base(n=40_000, m=20_000, seed=5)
    B, D = 64, base.n + base.m
    ws = L.LearnedWarmStart(base.n, base.m, base.L, base.U, base.l, base.u, d0=64, hidden=(64,), r=16, seed=1,
                            max_batch=B, chunk=B)
    ws.mu = torch.zeros(D, dtype=torch.float64, device="cuda")
    ws.fmean, ws.fistd = (torch.full((64,), v, dtype=torch.float32, device="cuda") for v in (0.0, 1.0))
    rng = np.random.default_rng(0)
    C = torch.from_numpy(rng.standard_normal((B, base.n))).cuda()
    U = torch.from_numpy(rng.standard_normal((B, base.m))).cuda()
    ws.predict(C, U)
    torch.cuda.synchronize()
    torch.cuda.reset_peak_memory_stats()
    before = torch.cuda.memory_allocated()
    Z, sig = ws.predict(C, U)
    peak = torch.cuda.max_memory_allocated() - before
    results = 8 * B * D + 2 * B * ws.Dp            # Z0, the members as BF16
    assert peak - results < 4 * B * D // 2, (peak, results)
    ws.close()
