"""The network's products where the device holds no cluster of sixteen blocks (hprqp_mlp_set_cluster stands in for
such a device): forward values and gradients lie within the rounding of the FP32 sums, whose order alone
changes, and the full cluster gives its bits again afterwards."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,B", [((1030, 257), 130), ((513, 130, 129), 31), ((4096, 64), 16)])
def test_fewer_blocks(dims, B):
    torch = pytest.importorskip("torch")
    import paper_2507_02470_gb300 as p
    p.build()
    from paper_2507_02470_gb300 import learned as L
    rng = np.random.default_rng(B)
    net = L.MLP(dims, B)
    for i in range(len(dims) - 1):
        net.set_layer(i, rng.standard_normal((dims[i + 1], dims[i])) / np.sqrt(dims[i]), np.zeros(dims[i + 1]))
    X = torch.zeros(B, L.round8(dims[0]), dtype=torch.bfloat16, device="cuda")
    X[:, :dims[0]] = torch.from_numpy(rng.standard_normal((B, dims[0]))).cuda()
    dY = torch.from_numpy(rng.standard_normal((B, dims[-1])).astype(np.float32)).cuda()

    def run(most):
        net.set_cluster(most)
        Y = net.forward(X).cpu().numpy()
        net.backward(dY)
        return [Y] + [net.get_grad(i)[0] for i in range(len(dims) - 1)]

    want = run(0)
    for most in (8, 5, 2, 1):
        for a, b in zip(run(most), want):
            # a BF16 value on the edge of two may fall to either side in the layer below: 2^-8 of the norm
            tol = 2.0 ** -8 if len(dims) > 2 else max(dims) * 2.0 ** -24
            assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), most
    for a, b in zip(run(0), want):
        assert np.array_equal(a, b)
    for bad in (-1, 17):
        with pytest.raises(Exception):
            net.set_cluster(bad)
    L.check()
    net.close()
