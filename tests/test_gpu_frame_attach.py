"""A frame attached, changed or taken off after the build takes effect at the next build: until then the
mesh steps as it was built, in the resident launch as in single launches."""
import math

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


def _run(ue, ms, chunk, built, then, replan, variant):
    tiled = variant == ue.UE_VARIANT_BLOCKED
    m = ue.Mesh(ms.xy, ms.tris, **(dict(reorder=ue.UE_REORDER_GREEDY, tile_tris=256) if tiled else {}))
    m.frame_attach(built)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h, graph_chunk=chunk, variant=variant, block_depth=4)
    c = ms.xy[ms.tris].mean(axis=1)
    m.write_fields(B=np.sin(5 * c[:, 0]) * np.cos(3 * c[:, 1]))
    m.frame_attach(then)
    if replan:
        ids, amp = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.35, ms.h)
        m.set_source(ids, amp, 40 * math.pi, 0.0, 0.05)
    m.step_n(70)
    assert m.check()[0]
    out = list(m.read_fields()[:2])
    if built:
        m.frame_attach(built)      # the layout of what frame_fields returns
        out += list(m.frame_fields())
    m.close()
    return out


@pytest.mark.parametrize("h", [1 / 16, 1 / 64])      # one CTA, several
@pytest.mark.parametrize("built,then", [(0, 6), (6, 0), (6, 9)])
@pytest.mark.parametrize("replan", [False, True])
@pytest.mark.parametrize("variant", [1, 2])
def test_frame_changes_wait_for_the_next_build(ue, h, built, then, replan, variant):
    ms = meshgen.graded_square(h, h, grade=0.0, holes=(), seed=5)
    a, b = (_run(ue, ms, chunk, built, then, replan, variant) for chunk in (32, -1))
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
