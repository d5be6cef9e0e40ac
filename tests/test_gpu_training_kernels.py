"""Training kernels at the edges of their tiles: forward, per-segment maximum and backward against
torch on the CPU."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_01448_gb300 import build
    build.build()
    import paper_1812_01448_gb300 as ue
    from paper_1812_01448_gb300 import learned
    rng = np.random.default_rng(2)
    p = learned.init_params(1)
    p[:768] += 0.1 * rng.standard_normal(768).astype(np.float32)
    p[-65:-1] = 0.2 * rng.standard_normal(64)
    return torch, ue, torch.from_numpy(p.astype(np.float32))


def _layers(torch, p, X, bf16):
    r = (lambda t: t.to(torch.bfloat16).double()) if bf16 else (lambda t: t.double())
    W1, b1, W2, b2, w3, b3 = torch.split(p, [768, 64, 4096, 64, 64, 1])
    x, W1, W2 = r(X), r(W1).reshape(64, 12), r(W2).reshape(64, 64)
    a1 = x @ W1.T + b1.double()
    h1 = r(torch.relu(a1).float())
    a2 = h1 @ W2.T + b2.double()
    return x, W2, a1, h1, a2, torch.relu(a2) @ w3.double() + b3.double()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 129, 152 * 128 - 1, 152 * 128 + 1, 700_003])
@pytest.mark.parametrize("shift", [0, 1])
def test_forward(lib, n, shift):
    """1e-3: the h1 that lie within an accumulation error of a BF16 midpoint may round the other
    way (2^-8 of a value, times a weight product below 0.2); the rest agrees to FP32."""
    torch, ue, p = lib
    flat = torch.randn(n * 12 + 1, generator=torch.Generator().manual_seed(n))
    X = flat[shift:shift + n * 12].reshape(n, 12)     # shift 1: rows off the 8-byte boundary
    Xd = flat.cuda()[shift:shift + n * 12].reshape(n, 12)
    z = torch.full((n + 1,), 7.0, device="cuda")
    ue.mlp_forward(p.cuda(), Xd, z, bf16=True)
    ref = _layers(torch, p, X, True)[-1]
    err = (z[:n].cpu().double() - ref).abs()
    assert err.max() < 1e-3 * ref.abs().max() + 1e-3 and err.median() < 2e-6
    assert z[n] == 7.0


@pytest.mark.parametrize("n", [32_767, 32_768, 32_895, 152 * 512 - 1, 152 * 512 + 1, 4 * 152 * 512 + 129])
def test_forward_of_many_rows(lib, n):
    """Around the rows from which layer 2 runs on tcgen05, and around its tiles: against torch, and
    against the same rows at an address that keeps the other kernel.  1e-5: both sum 64 products in FP32
    (a few 2^-24 of terms below 1) from the same BF16 h1.  Rows with a NaN or an infinity agree too."""
    torch, ue, p = lib
    flat = torch.randn(n * 12, generator=torch.Generator().manual_seed(n))
    X = flat.reshape(n, 12)
    X[7, 3], X[130, 0], X[131, 5], X[n - 1, 11] = float("nan"), float("inf"), -float("inf"), float("nan")
    off = torch.empty(n * 12 + 1, device="cuda")
    off[1:] = flat.cuda()
    z, y = torch.full((n + 1,), 7.0, device="cuda"), torch.full((n + 1,), 7.0, device="cuda")
    ue.mlp_forward(p.cuda(), X.cuda(), z, bf16=True)
    ue.mlp_forward(p.cuda(), off[1:].reshape(n, 12), y, bf16=True)
    assert z[n] == 7.0 and y[n] == 7.0
    assert torch.equal(z.isnan(), y.isnan()) and torch.equal(z.isinf(), y.isinf())
    f = z.isfinite()
    assert f.sum() >= n - 4
    assert (z[f] - y[f]).abs().max() < 1e-5
    ok = torch.isfinite(X).all(1)
    err = (z[:n].cpu().double() - _layers(torch, p, X, True)[-1])[ok].abs()
    assert err.max() < 4e-3 and err.median() < 2e-6


@pytest.mark.parametrize("sizes", [[1], [0, 3, 0], [4095, 4096, 4097, 1], [512, 511, 513, 20_000]])
def test_segment_argmax(lib, sizes):
    torch, ue, _ = lib
    off = np.concatenate([[0], np.cumsum(sizes)])
    rng = np.random.default_rng(len(sizes))
    z = rng.integers(0, 50, off[-1]).astype(np.float32)          # many ties: the first row wins
    base = rng.integers(0, 3, off[-1]).astype(np.float32)
    if off[-1] > 10:
        z[5] = np.nan
        base[7] = -np.inf
    best, arg = torch.zeros(len(sizes), device="cuda"), torch.zeros(len(sizes), dtype=torch.int64, device="cuda")
    ue.seg_argmax(torch.from_numpy(z).cuda(), torch.from_numpy(base).cuda(), torch.from_numpy(off).cuda(), best, arg)
    for s, (a, b) in enumerate(zip(off[:-1], off[1:])):
        t = np.where(np.isnan(z[a:b] + base[a:b]), -np.inf, z[a:b] + base[a:b])
        if b == a:
            assert best[s] == -np.inf and arg[s] == -1
        else:
            assert best[s] == t.max() and arg[s] == a + int(np.argmax(t))


@pytest.mark.parametrize("m", [1, 3, 4, 5, 1217, 2500])
@pytest.mark.parametrize("bf16", [False, True])
def test_backward(lib, m, bf16):
    """Sums of m FP32 products against FP64: m 2^-24 of the sum of magnitudes at most, and the
    chains of 64 before them as much again."""
    torch, ue, p = lib
    g = torch.Generator().manual_seed(m)
    X = torch.randn(3000, 12, generator=g)
    rows = torch.randint(0, 3000, (m,), generator=g)
    dz = torch.randn(m, generator=g)
    grad, work = torch.zeros(p.shape[0], device="cuda"), torch.zeros(m, p.shape[0], device="cuda")
    ue.mlp_backward(p.cuda(), X.cuda(), rows.cuda(), dz.cuda(), grad, work, bf16=bf16)
    x, W2, a1, h1, a2, _ = _layers(torch, p, X[rows], bf16)
    d = dz.double()[:, None]
    d2 = torch.where(a2 > 0, d * p[-65:-1].double(), 0.0)
    d1 = torch.where(a1 > 0, d2 @ W2, 0.0)

    def flat(e1, e2, x, h1, h2, d):
        return torch.cat([(e1.T @ x).ravel(), e1.sum(0), (e2.T @ h1).ravel(), e2.sum(0), h2.sum(0), d.sum().reshape(1)])
    ref = flat(d1, d2, x, h1, d * torch.relu(a2), d)
    size = flat(d1.abs(), d2.abs(), x.abs(), h1.abs(), (d * torch.relu(a2)).abs(), d.abs())
    # a unit whose a2 or h1 lies within rounding of a switch may differ: none does for these seeds
    err = (grad.cpu().double() - ref).abs()
    assert (err <= (m + 128) * 2.0 ** -24 * size + (2e-3 if bf16 else 1e-5) * size.max() / m ** 0.5).all()
