"""The training kernels' forms for few rows, few triangles and many segments, at the lines between the forms."""
import numpy as np
import pytest

import meshgen
from oracle import relax
from test_gpu_training_kernels import _layers, lib  # noqa: F401
from test_oracle_relax import _scramble

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_seg", [304, 305, 608, 609, 2432, 2433, 2440, 20_001])
def test_argmax_of_many_segments(lib, n_seg):  # noqa: F811
    """512 and 256 threads a segment, 128 (two segments a block) and a warp each (eight), with empty segments,
    segments of one row and of several passes, ties, NaN and infinities."""
    torch, ue, _ = lib
    rng = np.random.default_rng(n_seg)
    sizes = rng.choice([0, 1, 7, 31, 32, 33, 255, 256, 257, 300, 1025], n_seg)
    sizes[n_seg // 2] = 9001
    off = np.concatenate([[0], np.cumsum(sizes)])
    z = rng.integers(0, 40, off[-1]).astype(np.float32)
    base = rng.integers(0, 3, off[-1]).astype(np.float32)
    z[rng.integers(0, off[-1], 50)] = np.nan
    base[rng.integers(0, off[-1], 50)] = -np.inf
    z[rng.integers(0, off[-1], 5)] = np.inf
    best = torch.full((n_seg + 1,), 7.0, device="cuda")
    arg = torch.full((n_seg + 1,), 7, dtype=torch.int64, device="cuda")
    ue.seg_argmax(torch.from_numpy(z).cuda(), torch.from_numpy(base).cuda(), torch.from_numpy(off).cuda(), best[:n_seg], arg[:n_seg])
    with np.errstate(invalid="ignore"):
        t = z + base
    t[np.isnan(t)] = -np.inf
    want_b, want_a = np.full(n_seg, -np.inf, np.float32), np.full(n_seg, -1, np.int64)
    for s in range(n_seg):
        seg = t[off[s]:off[s + 1]]
        if seg.size and seg.max() > -np.inf:
            want_b[s], want_a[s] = seg.max(), off[s] + int(np.argmax(seg))
    assert np.array_equal(best.cpu().numpy()[:n_seg], want_b) and np.array_equal(arg.cpu().numpy()[:n_seg], want_a)
    assert float(best[n_seg]) == 7.0 and int(arg[n_seg]) == 7


@pytest.mark.parametrize("n", [1, 15, 17, 64, 65, 32_767, 49_999, 50_000, 50_001])
@pytest.mark.parametrize("shift", [1, 2])
def test_forward_off_the_alignment(lib, n, shift):  # noqa: F811
    """Around the line between the network in shared memory and in registers; bounds as for the other
    forms: an h1 that lies within an accumulation error of a BF16 midpoint may round the other way."""
    torch, ue, p = lib
    flat = torch.randn(n * 12 + 2, generator=torch.Generator().manual_seed(n))
    X = flat[shift:shift + n * 12].reshape(n, 12)
    z = torch.full((n + 1,), 7.0, device="cuda")
    ue.mlp_forward(p.cuda(), flat.cuda()[shift:shift + n * 12].reshape(n, 12), z[:n], bf16=True)
    ref = _layers(torch, p, X, True)[-1]
    err = (z[:n].cpu().double() - ref).abs()
    assert err.max() < 1e-3 * ref.abs().max() + 1e-3 and err.median() < 2e-6
    assert z[n] == 7.0


@pytest.mark.parametrize("m", [1, 2, 4, 5, 8])
def test_backward_of_one_block_and_two(lib, m):  # noqa: F811
    """One block writes the gradient itself; the sum over several blocks' shares adds the same rows."""
    torch, ue, p = lib
    g = torch.Generator().manual_seed(m)
    X, rows = torch.randn(50, 12, generator=g).cuda(), torch.randint(0, 50, (m,), generator=g).cuda()
    dz, k = torch.randn(m, generator=g).cuda(), p.shape[0]
    grad, part, work = torch.full((k,), 7.0, device="cuda"), torch.zeros(k, device="cuda"), torch.full((m * k,), 3.0, device="cuda")
    ue.mlp_backward(p.cuda(), X, rows, dz, grad, work)
    total = torch.zeros(k, dtype=torch.float64)
    size = torch.zeros(k, dtype=torch.float64)
    for i in range(m):
        ue.mlp_backward(p.cuda(), X, rows[i:i + 1], dz[i:i + 1], part, work)
        total += part.cpu().double()
        size += part.cpu().double().abs()
    # the same products, at most m + 1 FP32 additions each
    assert ((grad.cpu().double() - total).abs() <= (m + 1) * 2.0 ** -24 * size).all()


@pytest.mark.parametrize("points", [60, 180, 195, 205, 230])
def test_relaxation_around_the_line_for_host_marks(lib, points):  # noqa: F811
    """384 triangles: below, the flips' neighbours and marks are made on the host."""
    _, ue, _ = lib
    ms = meshgen.random_delaunay(points, seed=points)
    tris = _scramble(ms.xy, relax.orient_ccw(ms.xy, ms.tris), points // 3, seed=3).astype(np.int32)
    h = np.full(len(ms.xy), 1.2 / points ** 0.5)
    x, t, k = ue.mesh_relax(ms.xy, tris, 6, flip_every=2, h_nodes=h)
    y, u, f = ms.xy, tris, 0
    for _ in range(3):
        y, u, _ = ue.mesh_relax(y, u, 2, flip_every=0, h_nodes=h)
        u, n = ue.mesh_flip(y, u)
        f += n
    assert k == f > 0 and np.array_equal(t, u) and np.array_equal(x, y)
