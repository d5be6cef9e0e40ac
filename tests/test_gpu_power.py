"""The power iteration of ue_geometry_build against the same iteration in numpy, at the edges of
its launch shapes and of the segments between rescalings."""
import numpy as np
import pytest

from test_gpu_modes_block import _splitmix
from test_gpu_resident import _lattice

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


def _reference(m, iters, seed):
    """S-normalised power iteration from the library's tables and geometry (caller order)."""
    g, t = m.geometry(), m.tables()
    perm = t["perm_tri"]
    S = g["S"][perm]
    c = (g["elen"] / g["d"])[t["edge_caller"]]
    R, L = t["edge_tri"].T
    v = (_splitmix(np.uint64(seed << 32) + perm.astype(np.uint64)) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 * 2 - 1
    for _ in range(iters):
        v /= np.sqrt(np.dot(S * v, v))
        f = c * (v[R] - v[L])
        w = (np.bincount(R, f, m.n_tris) - np.bincount(L, f, m.n_tris)) / S
        rho = np.sqrt(np.dot(S * v, w))
        v = w
    return rho


@pytest.mark.parametrize("n_t,iters", [(2, 3), (33, 99), (1024, 100), (1025, 101), (2048, 200), (2049, 201),
                                       (4865, 1), (4865, 350), (155_649, 30), (311_297, 30), (622_593, 110)])
def test_power_iteration_matches_numpy(ue, n_t, iters):
    """1e-11: each product rounds to a few 2^-53 of |K||v|, and the quotient errs to second order."""
    xy, tris, h = _lattice(n_t, 11)
    m = ue.Mesh(xy, tris)
    m.geometry_build(power_iters=iters, power_seed=9)
    _, rho, src = m.get_dt()
    ref = _reference(m, iters, 9)
    m.close()
    assert src == 1 and abs(rho / ref - 1) < 1e-11


def test_power_iteration_with_scattered_neighbours(ue):
    """The caller's order kept and random: more remote neighbours than a CTA lists."""
    xy, tris, h = _lattice(400_000, 5, shuffle=True)
    m = ue.Mesh(xy, tris, reorder=ue.UE_REORDER_NONE)
    m.geometry_build(power_iters=40, power_seed=9)
    _, rho, _ = m.get_dt()
    ref = _reference(m, 40, 9)
    m.close()
    assert abs(rho / ref - 1) < 1e-11
