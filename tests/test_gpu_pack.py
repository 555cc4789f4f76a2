"""The copy-rate BF16 casts and the decoder fused into its product, at the sizes where their
pairing and tiling can go wrong: odd columns, rows off a pair's alignment, values at the edges of
FP32's range, partial tiles of rows and columns.  The casts match the oracle's rounding bit for
bit; the decoder lies within the FP32 accumulation bound of the exact product, clipped alike."""
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


EDGES = [0.0, -0.0, 1.0, -1.0, 2.0 ** -126, 2.0 ** -127, -2.0 ** -149, 2.0 ** -150, 1e-300, 5e-324, 3.4e38, 3.3895e38,
         3.3961775e38, 1e300, -1e300, np.inf, -np.inf, np.nan, 1 + 2.0 ** -8, 1 + 3 * 2.0 ** -9, 1 + 2.0 ** -8 + 2.0 ** -40,
         1.00390625 - 2.0 ** -30, 2.0 - 2.0 ** -24, 2.0 - 2.0 ** -25, 2.0 - 2.0 ** -53]


def bits(t):
    import torch
    return t.view(torch.int16).cpu().numpy().view(np.uint16)


def rounded(a):
    """The contract: non-finite to 0, FP64 -> FP32 -> BF16, ties to even."""
    with np.errstate(over="ignore"):
        f = np.where(np.isfinite(a), a, 0.0).astype(np.float32)
    b = f.view(np.uint32)
    out = ((b.astype(np.uint64) + 0x7FFF + ((b >> 16) & 1)) >> 16).astype(np.uint16)
    return out


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("rows,cols,pad,shift", [(1, 1, 0, 0), (3, 25, 0, 1), (2, 2047, 1, 0), (5, 2049, 0, 0), (1, 6001, 3, 1)])
def test_cast_bits(env, dtype, rows, cols, pad, shift):
    torch, p, L = env
    rng = np.random.default_rng(rows * 100 + cols)
    a = rng.standard_normal((rows, cols)) * np.exp2(rng.integers(-140, 120, (rows, cols)))
    k = min(cols, len(EDGES))
    a[0, :k] = EDGES[:k]
    with np.errstate(over="ignore"):
        a = a.astype(dtype)
    buf = torch.zeros(rows * (cols + pad) + shift, dtype=getattr(torch, dtype), device="cuda")
    x = buf[shift:].reshape(rows, cols + pad)[:, :cols]
    x.copy_(torch.from_numpy(a))
    ld = L.round8(cols) + 8
    got = bits(L.cast_bf16(x, ld=ld))
    assert np.array_equal(got[:, :cols], rounded(a.astype(np.float64)))
    assert not got[:, cols:].any()


@pytest.mark.parametrize("n,m", [(7, 3), (8, 0), (1, 2050), (2047, 5), (3001, 1500)])
def test_pack_is_the_cast_of_the_joined_rows(env, n, m):
    torch, p, L = env
    rng = np.random.default_rng(n + m)
    C, U = rng.standard_normal((3, n + 1)), rng.standard_normal((3, m + 2))
    c, u = torch.from_numpy(C).cuda()[:, :n], torch.from_numpy(U).cuda()[:, :m]
    ws = L.LearnedWarmStart(n, m, np.zeros(n), np.ones(n), np.zeros(m), np.ones(m), d0=8, hidden=(8,), r=8, max_batch=4)
    got = ws._pack(c, u)
    want = ws._pack(C[:, :n], U[:, :m])        # host rows: joined in FP64, then cast
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    assert np.array_equal(bits(got)[:, :n + m], rounded(np.concatenate([C[:, :n], U[:, :m]], axis=1)))


@pytest.mark.parametrize("D,B,r", [(1, 1, 1), (127, 3, 8), (129, 64, 70), (300, 65, 256), (1000, 130, 64)])
def test_fused_decoder(env, D, B, r):
    torch, p, L = env
    from paper_2507_02470_gb300._lib import lib
    import ctypes as C
    rng = np.random.default_rng(D + B)
    phi = torch.zeros(D, L.round8(r), dtype=torch.bfloat16, device="cuda")
    phi[:, :r] = torch.from_numpy(rng.standard_normal((D, r))).cuda()
    O = torch.from_numpy(rng.standard_normal((B, r + 2)).astype(np.float32)).cuda()
    mu, lo, hi = rng.standard_normal(D), np.full(D, -1.0), np.full(D, np.inf)
    lo[::3], hi[::2] = -np.inf, 0.25
    dev = [torch.from_numpy(v).cuda() for v in (mu, lo, hi)]
    Z = torch.full((B, D + 3), float("nan"), dtype=torch.float64, device="cuda")
    sig = torch.empty(B, dtype=torch.float64, device="cuda")
    work = torch.empty(D * B, dtype=torch.float32, device="cuda")
    alpha = np.float32(0.37)
    st = lib().hprqp_ws_decode(phi.data_ptr(), phi.stride(0), D, r, O.data_ptr(), O.stride(0), B, C.c_float(alpha),
                               C.c_float(0.1), C.c_float(2.0), *[t.data_ptr() for t in dev], work.data_ptr(),
                               Z.data_ptr(), Z.stride(0), sig.data_ptr(), None)
    assert st == 0
    torch.cuda.synchronize()
    L.check()
    ell = OL.bf16_round(O.cpu().numpy().astype(np.float64)[:, 1:1 + r])
    P = phi[:, :r].double().cpu().numpy()
    z = mu + float(alpha) * (ell @ P.T)
    bound = float(alpha) * 4 * r * 2.0 ** -24 * (np.abs(ell) @ np.abs(P).T) + 1e-15 * (1 + np.abs(z))
    got = Z.cpu().numpy()
    assert np.all(np.abs(got[:, :D] - np.minimum(np.maximum(z, lo), hi)) <= bound)
    assert np.isnan(got[:, D:]).all()
