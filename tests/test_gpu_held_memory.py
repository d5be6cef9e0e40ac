"""Calls that take work space leave the device's free memory as it was, but for 64 MB at most."""
import random

import pytest

import meshgen

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


def _used():
    import torch
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_repeated_calls_hold_bounded_memory(ue):
    ms = meshgen.plasma_square_mesh(60000, seed=6)
    before = _used()
    m = ue.Mesh(ms.xy, ms.tris)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h)
    m.modes(24, iters=2)                  # kernels loaded
    m.modes_low(2, iters=1, degree=2)
    m.geometry()
    built = _used()
    rng = random.Random(7)
    for i in range(150):
        m.modes(rng.randint(1, 24), iters=1, vectors=True)
        if i % 10 == 0:
            m.modes_low(rng.randint(1, 16), iters=1, degree=2)
            m.geometry()
            m.set_plasma(1.0 + ms.xy[:, 0], 0.5)
    # 64 MB of returned work space, a chunk for the medium's arrays
    assert _used() - built <= (64 + 16) << 20
    for _ in range(3):
        m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h)
    rebuilt = _used()
    assert rebuilt - built <= 16 << 20
    m.close()
    assert _used() - before <= 16 << 20      # what loading kernels took
