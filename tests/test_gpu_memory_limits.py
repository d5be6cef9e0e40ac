"""Where the allocator refuses memory that only the faster paths take, the calls go through as without
them: no resident step, the power iteration by edges and triangles, the same results."""
import ctypes as C

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


class Limited:
    """Allocator callbacks over torch tensors: at most `limit` bytes at once, no block above `block`."""

    def __init__(self):
        import torch
        from paper_1812_01448_gb300 import _native as N
        self.limit = self.block = 1 << 62
        self.live, self.used, self.most = {}, 0, 0

        def alloc(nbytes, stream, ctx):
            if nbytes > self.block or self.used + nbytes > self.limit:
                return None
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            self.live[t.data_ptr()] = t
            self.used += nbytes
            self.most = max(self.most, self.used)
            return t.data_ptr()

        def free(ptr, stream, ctx):
            self.used -= self.live.pop(ptr).numel()

        self.alloc, self.free = N.ALLOC_FN(alloc), N.FREE_FN(free)


def _load(ue, ms, lim, **load):
    from paper_1812_01448_gb300 import _native as N
    xy, t = np.ascontiguousarray(ms.xy), np.ascontiguousarray(ms.tris, dtype=np.int32)
    h, o = C.c_void_p(), ue.options(**load)
    N.check(N.lib().ue_mesh_load(xy.ctypes.data_as(N.PD), xy.shape[0], t.ctypes.data_as(N.PI32), t.shape[0], C.byref(o),
                                 lim.alloc, lim.free, None, C.byref(h)), "ue_mesh_load")
    return ue.Mesh._wrap(h, keep=(lim,))


def _steps(ue, ms, m, **opt):
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h, graph_chunk=32, **opt)
    ids, amp = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.35, ms.h)
    m.set_source(ids, amp, 20.0, 0.0, 0.3)
    m.write_fields(B=np.sin(7 * ms.xy[ms.tris].mean(axis=1)[:, 0]))
    m.step_n(70)
    return m.read_fields()[:2]


@pytest.mark.parametrize("n_t", [600, 6000])
@pytest.mark.parametrize("opt", [dict(), dict(precision=1), dict(watchdog_every=32)])
def test_a_build_without_room_for_the_resident_step(ue, n_t, opt):
    ms = meshgen.plasma_square_mesh(n_t, seed=6)
    lim = Limited()
    m = _load(ue, ms, lim)
    ref = _steps(ue, ms, m, variant=ue.UE_VARIANT_NO_RESIDENT, **opt)
    without = lim.most
    m.close()
    assert lim.used == 0
    for room in (0, 64, 4 * n_t, 24 * n_t):    # none, the control words, some of the arrays
        lim = Limited()
        m = _load(ue, ms, lim)
        # the source's table of g(t) is sized for a resident launch when one was planned
        lim.limit = without + 8 * 1024 + room
        got = _steps(ue, ms, m, **opt)
        assert m.check()[0] and m.stats()["resident_launches"] == 0
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)
        lim.limit = 1 << 62                    # room again: the next build steps resident
        got = _steps(ue, ms, m, **opt)
        assert m.stats()["resident_launches"] > 0
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)
        m.close()
        assert lim.used == 0


@pytest.mark.parametrize("frame", [0, 6])
def test_a_later_call_takes_the_resident_step_s_room(ue, frame):
    """Modes, a medium and sources after a build that left no room: the resident step makes way."""
    ms = meshgen.graded_square(1 / 48, 1 / 48, grade=0.0, holes=(), seed=5)
    dens = 10.0 + ms.xy[:, 0]
    ids, amp = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.35, ms.h)
    out = []
    for limited in (False, True):
        lim = Limited()
        m = _load(ue, ms, lim)
        m.frame_attach(frame)
        m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h, graph_chunk=32)
        m.write_fields(B=np.sin(7 * ms.xy[ms.tris].mean(axis=1)[:, 0]))
        m.step_n(64)
        assert m.stats()["resident_launches"] == 1
        if limited:
            lim.limit = lim.used + 64
        om = m.modes(1, iters=4) if not frame else None
        m.set_plasma(dens, 0.5)
        m.set_source(ids, amp, 20.0, 0.0, 0.3)
        m.step_n(64)
        assert m.check()[0] and m.stats()["resident_launches"] == (1 if limited else 2)
        out.append((om,) + tuple(m.read_fields(j=True)))
        m.close()
        assert lim.used == 0
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_power_iteration_on_the_smaller_work_space(ue):
    ms = meshgen.plasma_square_mesh(6000, seed=6)
    lim = Limited()
    m = _load(ue, ms, lim)
    m.geometry_build()
    rho = m.get_dt()[1]
    lim.block = 8 * 9 * m.n_tris         # between the two work spaces, 12 and 6 doubles per triangle
    m.geometry_build()
    small = m.get_dt()[1]
    m.close()
    # the same 200 products with other roundings, a few ulp of the iterate each
    assert abs(small / rho - 1) <= 1e-12 and lim.used == 0
