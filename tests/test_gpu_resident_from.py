"""From how many steps on a blocked mesh's calls run resident, and that both forms leave the same bits."""
import numpy as np
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


# triangles, tile size, depth, source -> fewest steps (None: never); the largest tile with its rings has
# 894, 606, 1,923, 2,301, 1,929 (depth 5), 2,324, 687 (256 tiles) and 1,104 triangles; slots hold 2,048 or 3,072
CASES = [(6_000, 500, 8, False, None), (6_000, 500, 8, True, 64), (6_000, 500, 4, False, 64), (6_000, 500, 3, False, 30),
         (6_000, 1_900, 8, False, None), (22_000, 1_900, 8, False, 64), (22_000, 1_900, 8, True, 32),
         (22_000, 1_900, 5, False, 64), (4_000, 2_100, 8, False, None), (60_000, 300, 8, False, 32),
         (60_000, 700, 8, False, None)]


@pytest.mark.parametrize("n_t,tile,depth,source,least", CASES)
@pytest.mark.parametrize("watchdog", [0, 40])
def test_the_shortest_resident_call(ue, n_t, tile, depth, source, least, watchdog):
    ms = meshgen.plasma_square_mesh(n_t, seed=4)
    ids, amp = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.35, ms.h)
    calls = [31, 64, 63, 256, 20, 300, least or 32, (least or 32) - 1]
    out = []
    for flag in (0, ue.UE_VARIANT_NO_RESIDENT):
        m = ue.Mesh(ms.xy, ms.tris, reorder=ue.UE_REORDER_KD, tile_tris=tile)
        m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h, variant=ue.UE_VARIANT_BLOCKED | flag, block_depth=depth,
                         watchdog_every=watchdog)
        if source:
            m.set_source(ids, amp, 1.0 / ms.h, 0.0, 0.3)
        m.write_fields(B=np.sin(7 * ms.xy[ms.tris].mean(axis=1)[:, 0]))
        m.step_prepare()
        runs = 0
        for n in calls:
            m.step_n(n)
            runs += bool(least) and n >= least and not flag
            assert m.stats()["resident_launches"] == runs
        assert m.check()[0]
        out.append(m.read_fields()[:2] + (m.get_step(),))
        m.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
