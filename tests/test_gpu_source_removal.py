"""A source that is taken off again: every launch form steps as a mesh that never had one."""
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


@pytest.mark.parametrize("opt", [dict(variant=1), dict(variant=257), dict(variant=3), dict(variant=2), dict(variant=258),
                                 dict(variant=258, tb_kernel=1), dict(variant=258, tb_threads=1024)])
@pytest.mark.parametrize("tile", [64, 256, 8192])
@pytest.mark.parametrize("plasma", [False, True])
def test_a_source_taken_off(ue, opt, tile, plasma):
    ms = meshgen.graded_square(1 / 28, 1 / 28, grade=0.0, holes=(), seed=5)
    ids, amp = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.3, ms.h)
    out = []
    for source in (False, True):
        m = ue.Mesh(ms.xy, ms.tris, reorder=ue.UE_REORDER_GREEDY, tile_tris=tile)
        m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h, graph_chunk=16, block_depth=4, **opt)
        if plasma:
            m.set_plasma(1.0 + ms.xy[:, 0], 0.5)
        if source:
            m.set_source(ids, amp, 20.0, 0.0, 0.3)
            m.step_n(37)
            m.set_source(ids[:0], amp[:0], 20.0, 0.0, 0.3)
        m.write_fields(E=np.zeros(m.n_edges), B=np.sin(7 * ms.xy[ms.tris].mean(axis=1)[:, 0]), j=np.zeros(m.n_edges))
        m.step_n(37)
        assert m.check()[0]
        out.append(m.read_fields(j=True))
        m.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
