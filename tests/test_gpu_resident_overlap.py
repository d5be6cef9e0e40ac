"""Resident launches beside each other and beside other work: meshes on streams of their own, from threads of
their own, end with the bits that each has alone."""
import threading

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


SIZES = [(400, 0), (6_000, 0), (6_000, 1), (150_000, 0), (120_000, 0), (120_000, 1)]   # triangles, precision


def _mesh(ue, i):
    n_t, prec = SIZES[i]
    ms = meshgen.plasma_square_mesh(n_t, seed=20 + i)
    m = ue.Mesh(ms.xy, ms.tris)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h, graph_chunk=32, precision=prec, watchdog_every=32)
    ids, amp = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.35, ms.h)
    m.set_source(ids, amp, 1.0 / ms.h, 0.0, 0.3)
    m.write_fields(B=np.sin(7 * ms.xy[ms.tris].mean(axis=1)[:, 0]))
    return m


@pytest.mark.parametrize("threads", [False, True])
def test_meshes_on_streams_of_their_own(ue, threads):
    import torch
    alone = []
    for i in range(len(SIZES)):
        m = _mesh(ue, i)
        for _ in range(8):
            m.step_n(50)
        alone.append(m.read_fields()[:2])
        m.close()
    meshes = [_mesh(ue, i) for i in range(len(SIZES))]
    streams = [torch.cuda.Stream() for _ in meshes]
    torch.cuda.synchronize()
    errors = []

    def run(m, s):
        try:
            for _ in range(8):
                m.step_n(50, s)
        except Exception as e:   # reported by the main thread
            errors.append(e)
    a = torch.randn(4096, 4096, device="cuda", dtype=torch.bfloat16)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        for _ in range(50):
            b = a @ a
    if threads:
        ts = [threading.Thread(target=run, args=x) for x in zip(meshes, streams)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    else:
        for _ in range(8):
            for m, s in zip(meshes, streams):
                m.step_n(50, s)
    torch.cuda.synchronize()
    assert not errors and bool(torch.isfinite(b.float()).all())
    for m, (E, B) in zip(meshes, alone):
        assert m.check()[0] and m.stats()["resident_launches"] == 8
        got = m.read_fields()[:2]
        assert np.array_equal(got[0], E) and np.array_equal(got[1], B)
        m.close()
