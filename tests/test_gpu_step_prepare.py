"""ue_step_prepare makes what the next long call will use and nothing else: graphs where the mesh replays
them (also where the resident step is declined), none where it steps resident.  Captures of thousands
of launches take tens of milliseconds, so host times tell which was made."""
import time

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


def _mesh(ue, ms, variant, **opt):
    m = ue.Mesh(ms.xy, ms.tris, reorder=ue.UE_REORDER_KD, tile_tris=256)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h, variant=variant, **opt)
    m.write_fields(B=np.sin(7 * ms.xy[ms.tris].mean(axis=1)[:, 0]))
    return m


def _host_time(f):
    import torch
    torch.cuda.synchronize()
    t = time.perf_counter()
    f()
    t = time.perf_counter() - t
    torch.cuda.synchronize()
    return t


def test_a_declined_resident_step_is_prepared_as_graphs(ue):
    """With the watchdog on, a graph chunk longer than a resident launch: the chunk's graph is replayed."""
    ms = meshgen.plasma_square_mesh(5000, seed=4)
    first, out = {False: [], True: []}, []
    for _ in range(3):
        for prepare in (False, True):
            m = _mesh(ue, ms, ue.UE_VARIANT_PLAIN, graph_chunk=2048, watchdog_every=2048)
            if prepare:
                m.step_prepare()
            first[prepare].append(_host_time(lambda: m.step_n(2048)))
            assert m.check()[0] and m.stats()["resident_launches"] == 0
            out.append(m.read_fields()[:2])
            m.close()
    m = _mesh(ue, ms, ue.UE_VARIANT_PLAIN, graph_chunk=-1)
    m.step_n(2048)
    for E, B in out:
        assert np.array_equal(E, m.read_fields()[0]) and np.array_equal(B, m.read_fields()[1])
    m.close()
    assert min(first[True]) < 0.5 * min(first[False])      # nothing left to capture


@pytest.mark.parametrize("variant", [1, 2])
def test_a_resident_mesh_prepares_no_graph(ue, variant):
    ms = meshgen.plasma_square_mesh(5000, seed=4)
    t = {}
    for flag in (0, ue.UE_VARIANT_NO_RESIDENT):
        t[flag] = []
        for _ in range(3):
            m = _mesh(ue, ms, variant | flag, graph_chunk=2000, block_depth=1)
            t[flag].append(_host_time(m.step_prepare))
            m.step_n(2000)
            assert (m.stats()["resident_launches"] > 0) == (flag == 0)
            m.close()
    assert min(t[0]) < 0.2 * min(t[ue.UE_VARIANT_NO_RESIDENT])
