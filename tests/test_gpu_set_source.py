"""ue_set_source again and again on one mesh: the device arrays, the resident plan and the tiles' records
follow the last call; a call without memory leaves no source."""
import numpy as np
import pytest

import meshgen
from test_gpu_memory_limits import Limited, _load

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


FORMS = [dict(), dict(precision=1), dict(variant=257), dict(variant=2, block_depth=4), dict(variant=258, block_depth=4),
         dict(variant=258, block_depth=4, tb_kernel=1)]


def _build(ue, ms, m, frame, opt):
    m.frame_attach(frame)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h, graph_chunk=32, **opt)


def _go(ms, m, n=40):
    m.set_step(3)
    m.write_fields(E=np.zeros(m.n_edges), B=np.sin(7 * ms.xy[ms.tris].mean(axis=1)[:, 0]))
    m.step_n(n)
    assert m.check()[0]
    return m.read_fields()[:2]


@pytest.mark.parametrize("opt", FORMS)
@pytest.mark.parametrize("frame", [0, 5])
def test_sources_in_turn(ue, opt, frame):
    ms = meshgen.graded_square(1 / 40, 1 / 40, grade=0.0, holes=(), seed=5)
    lines = [meshgen.source_line_amplitudes(ms.xy, ms.tris, x, ms.h) for x in (0.3, 0.7, 0.5)]
    lines[1] = tuple(a[:1] for a in lines[1])               # a single edge
    load = dict(reorder=ue.UE_REORDER_GREEDY, tile_tris=256)
    m = ue.Mesh(ms.xy, ms.tris, **load)
    _build(ue, ms, m, frame, opt)
    none = _go(ms, m)
    for i, (ids, amp) in enumerate(lines + [lines[0]]):
        m.set_source(ids, amp, 20.0 + i, 0.0, 0.3)
        got = _go(ms, m)
        f = ue.Mesh(ms.xy, ms.tris, **load)
        _build(ue, ms, f, frame, {**opt, "variant": 257, "block_depth": 1, "tb_kernel": 0})   # launches, graphs
        f.set_source(ids, amp, 20.0 + i, 0.0, 0.3)
        for a, b in zip(got, _go(ms, f)):
            assert np.array_equal(a, b)
        f.close()
        assert not np.array_equal(got[0], none[0])
    m.set_source(lines[0][0][:0], lines[0][1][:0], 20.0, 0.0, 0.3)
    for a, b in zip(_go(ms, m), none):
        assert np.array_equal(a, b)
    m.close()


@pytest.mark.parametrize("variant", [1, 2, 257, 258])
@pytest.mark.parametrize("frame", [0, 5])
def test_no_memory_leaves_no_source(ue, variant, frame):
    ms = meshgen.graded_square(1 / 40, 1 / 40, grade=0.0, holes=(), seed=5)
    ids, amp = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.3, ms.h)
    lim = Limited()
    m = _load(ue, ms, lim, reorder=ue.UE_REORDER_GREEDY, tile_tris=256)
    _build(ue, ms, m, frame, dict(variant=variant, block_depth=4))
    none = _go(ms, m)
    m.set_source(ids, amp, 20.0, 0.0, 0.3)
    with_source = _go(ms, m)
    lim.block = 0
    with pytest.raises(ue.UEError) as e:
        m.set_source(ids, amp, 30.0, 0.0, 0.3)
    assert e.value.code == -6
    lim.block = 1 << 62
    for a, b in zip(_go(ms, m), none):
        assert np.array_equal(a, b)
    m.set_source(ids, amp, 20.0, 0.0, 0.3)
    for a, b in zip(_go(ms, m), with_source):
        assert np.array_equal(a, b)
    m.close()
    assert lim.used == 0
