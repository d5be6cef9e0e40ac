"""ue_modes after a fixed number of products against the same block iteration in numpy (QR after
every product), for every block width class: the library's Cholesky QR comes after several."""
import numpy as np
import pytest

import meshgen
from oracle import mesh as om, operators, spectral

pytestmark = pytest.mark.gpu


def _splitmix(x):
    with np.errstate(over="ignore"):
        z = x + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


@pytest.mark.parametrize("n_modes", [1, 3, 5, 8, 11, 16, 24])
@pytest.mark.parametrize("iters", [1, 2, 37])
def test_block_iteration_matches_numpy(n_modes, iters):
    """Ritz values to 1e-10: the span differs by rounding only (bases conditioned to 100, so
    Gram matrices to 1e4: at most 32 * 1e4 * 2^-53 = 4e-11, and Ritz values err to second order)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_01448_gb300 import build
    build.build()
    import paper_1812_01448_gb300 as ue
    ms = meshgen.graded_square(0.05, 0.12, grade=0.3, seed=5, holes=[meshgen.polygon_triangle((0.5, 0.5), 0.3)])
    ops = operators.Operators(om.canonicalize(ms.xy, ms.tris))
    n, m = ms.n_tris, min(32, 2 * n_modes)
    key = np.uint64(7 << 32) + np.arange(n * m, dtype=np.uint64)
    V = ((_splitmix(key) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 * 2 - 1).reshape(n, m)
    rs = np.sqrt(ops.w_B)[:, None]
    V = np.linalg.qr(rs * V)[0]
    for _ in range(iters):
        V = np.linalg.qr(rs * spectral.apply_K(ops, V / rs))[0]
    lam = np.linalg.eigvalsh(V.T @ (rs * spectral.apply_K(ops, V / rs)))[::-1]
    mesh = ue.Mesh(ms.xy, ms.tris)
    mesh.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=1e-4)
    w, B = mesh.modes(n_modes, iters=iters, seed=7, vectors=True)
    mesh.close()
    assert np.abs(w / np.sqrt(lam[:n_modes]) - 1).max() < 1e-10
    G = (B * ops.w_B) @ B.T
    assert np.abs(G - np.eye(n_modes)).max() < 1e-10
