"""ue_mesh_relax's device lists and marks against the host's flips and the oracle, at the edges of the
device path: nodes of more triangles than one thread sorts, edges of more than two triangles."""
import numpy as np
import pytest

import meshgen
from oracle import relax
from test_oracle_relax import _scramble

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ue():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_01448_gb300 import build
    build.build()
    import paper_1812_01448_gb300 as ue
    return ue


def _mesh(kind):
    rng = np.random.default_rng(4)
    if kind.startswith("wheel"):           # a hub of n triangles, its rim the boundary
        n = int(kind[5:])
        a = 2 * np.pi * np.arange(n) / n
        xy = np.concatenate([[[0.11, -0.07]], np.stack([np.cos(a), np.sin(a)], 1)])
        k = np.arange(n)
        return xy, np.stack([np.zeros(n, int), 1 + k, 1 + (k + 1) % n], 1).astype(np.int32)
    ms = meshgen.random_delaunay(300, seed=6)
    tris = _scramble(ms.xy, relax.orient_ccw(ms.xy, ms.tris), 120, seed=3).astype(np.int32)
    if kind == "shuffled":                 # corners rotated, some turned over, triangles in any order
        tris = np.stack([np.roll(r, i % 3) for i, r in enumerate(tris)])
        tris[::7] = tris[::7, ::-1]
        return ms.xy, np.ascontiguousarray(tris[rng.permutation(len(tris))])
    if kind == "doubled":                  # a part of the triangles twice: up to four on an edge
        return ms.xy, np.concatenate([tris, tris[40:90]])
    return ms.xy, tris


@pytest.mark.parametrize("kind", ["scrambled", "shuffled", "doubled", "wheel32", "wheel33", "wheel200"])
def test_relaxation_is_steps_and_host_flips_in_turn(ue, kind):
    """Rows, corners and positions bit for bit those of one call per step with the flips between
    them made by ue_mesh_flip; positions without flips against the oracle's."""
    xy, tris = _mesh(kind)
    h = np.full(len(xy), 0.06)
    x, t, k = ue.mesh_relax(xy, tris, 6, flip_every=2, h_nodes=h)
    y, u, f = xy, tris, 0
    for _ in range(3):
        y, u, _ = ue.mesh_relax(y, u, 2, flip_every=0, h_nodes=h)
        u, n = ue.mesh_flip(y, u)
        f += n
    assert np.array_equal(t, u) and k == f
    assert np.array_equal(x, y)
    if not kind.startswith("wheel"):
        assert k > 0
    # 20 steps: sums of up to 400 pulls a few ulps apart, damped from step to step
    z, _, _ = ue.mesh_relax(xy, tris, 20, flip_every=0, h_nodes=h)
    o, _, _ = relax.relax(xy, tris, 20, h_nodes=h)
    assert np.abs(z - o).max() < 1e-10 * 0.06
