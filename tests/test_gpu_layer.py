"""The network's products with their epilogues in one launch (K-splits of a tile as one cluster) at the
sizes where the split rows, the 4 x 4 pieces and the joined kernels can go wrong: widths and batches off
their multiples, one to sixteen K-splits, one layer, more splits than rows of four.  Forward values and
gradients lie within the FP32 accumulation and BF16 rounding bounds of the exact products of the same
BF16 operands."""
import numpy as np
import pytest

from oracle import learned as OL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import paper_2507_02470_gb300 as p
    p.build()
    from paper_2507_02470_gb300 import learned as L
    return torch, p, L


@pytest.mark.parametrize("dims,B", [((8, 1), 1), ((70, 5), 3), ((64, 33, 7), 65), ((513, 130, 129), 31), ((1030, 257), 130),
                                    ((1024, 100), 256), ((24, 640, 9), 200), ((100, 60, 40, 20), 513)])
def test_layers(env, dims, B):
    torch, p, L = env
    rng = np.random.default_rng(sum(dims) + B)
    net = L.MLP(dims, B, stream=torch.cuda.current_stream())
    W = [rng.standard_normal((dims[i + 1], dims[i])) / np.sqrt(dims[i]) for i in range(len(dims) - 1)]
    b = [rng.standard_normal(dims[i + 1]) for i in range(len(dims) - 1)]
    for i in range(len(W)):
        net.set_layer(i, W[i], b[i])
    X = OL.bf16_round(rng.standard_normal((B, dims[0])))
    Xt = torch.zeros(B, L.round8(dims[0]), dtype=torch.bfloat16, device="cuda")
    Xt[:, :dims[0]] = torch.from_numpy(X).cuda()
    Y = net.forward(Xt).cpu().double().numpy()
    dY = rng.standard_normal((B, dims[-1])).astype(np.float32)
    net.backward(torch.from_numpy(dY).cuda())
    Wb = [OL.bf16_round(w) for w in W]
    bf = [v.astype(np.float32).astype(np.float64) for v in b]
    U32, U16 = 2.0 ** -24, 2.0 ** -8
    h, err, hs, errs = X, np.zeros_like(X), [X], [np.zeros_like(X)]
    for i in range(len(W)):
        K = dims[i]
        mag = (np.abs(h) + err) @ np.abs(Wb[i]).T
        z = h @ Wb[i].T + bf[i]
        err = err @ np.abs(Wb[i]).T + 4 * K * U32 * mag + 2 * U32 * (mag + np.abs(bf[i]))
        if i + 1 < len(W):
            h = OL.bf16_round(np.maximum(z, 0.0))
            err = err + U16 * (2 * np.abs(h) + err)
            hs.append(h)
            errs.append(err)
    assert np.all(np.abs(Y - z) <= err + 1e-30)
    dZ, ez = OL.bf16_round(dY.astype(np.float64)), np.zeros_like(dY, dtype=np.float64)
    for i in range(len(W) - 1, -1, -1):
        gW, gb = net.get_grad(i)
        a, x = np.abs(dZ) + ez, np.abs(hs[i]) + errs[i]
        assert np.all(np.abs(gW - dZ.T @ hs[i]) <= ez.T @ x + np.abs(dZ).T @ errs[i] + 4 * B * U32 * (a.T @ x) + 1e-30)
        assert np.all(np.abs(gb - dZ.sum(0)) <= ez.sum(0) + 4 * B * U32 * a.sum(0) + 1e-30)
        if i == 0:
            break
        K = dims[i + 1]
        dX = dZ @ Wb[i]
        e = ez @ np.abs(Wb[i]) + 4 * K * U32 * (a @ np.abs(Wb[i]))
        unsure = hs[i] <= errs[i]                # the ReLU of the layer below may be on either side
        dZ = OL.bf16_round(dX * (hs[i] > 0))
        ez = np.where(unsure, np.abs(dX) + e + U16 * (np.abs(dX) + e), e + U16 * (2 * np.abs(dZ) + e))
    net.adam(lr=1e-3)
    for i in range(len(W)):
        gW, gb = net.get_grad(i)
        w1, b1 = net.get_layer(i)
        # Adam's first step: -lr g / (|g| + eps)
        for new, old, g in ((w1, W[i].astype(np.float32), gW), (b1, b[i].astype(np.float32), gb)):
            want = old - 1e-3 * g / (np.abs(g) + 1e-8)
            assert np.max(np.abs(new - want)) <= 1e-6 + 1e-5 * max(1.0, float(np.max(np.abs(old))))
    L.check()
