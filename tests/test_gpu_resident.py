"""The resident step (one cooperative launch for many steps) against the plain launches, bit for
bit: every medium, precision and order it takes, at the edges of its launch shapes."""
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


def _lattice(n_t, seed, shuffle=False):
    """About n_t triangles: a strip of equilateral rows cut to exactly n_t, jittered, the caller's
    triangle order shuffled on request."""
    rows = max(1, int(math.sqrt(n_t / 2)))
    cols = -(-n_t // (2 * rows))
    r, c = np.meshgrid(np.arange(rows + 1), np.arange(cols + 1), indexing="ij")
    xy = np.stack([(c + 0.5 * r).ravel(), (math.sqrt(3) / 2 * r).ravel()], axis=1).astype(np.float64)
    w = cols + 1
    p = (np.arange(rows)[:, None] * w + np.arange(cols)[None, :]).ravel()
    tris = np.stack([np.stack([p, p + 1, p + w], 1), np.stack([p + 1, p + w + 1, p + w], 1)], 1).reshape(-1, 3)[:n_t]
    rng = np.random.default_rng(seed)
    xy = (xy + rng.uniform(-0.08, 0.08, xy.shape)) / max(rows, cols)
    if shuffle:
        tris = tris[rng.permutation(len(tris))]
    used = np.zeros(len(xy), bool)
    used[tris.ravel()] = True
    return xy[used], (np.cumsum(used) - 1)[tris].astype(np.int32), 1.0 / max(rows, cols)


def _run(ue, xy, tris, h, steps, chunk, load=None, plasma=False, source=True, frame=0, calls=1, **opt):
    m = ue.Mesh(xy, tris, **(load or {}))
    if frame:
        m.frame_attach(frame)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.1 * h, graph_chunk=chunk, **opt)
    w0 = 2.0 / h
    if source:
        ids, amp = meshgen.source_line_amplitudes(xy, tris, float(xy[:, 0].mean()), h)
        if ids.size:
            m.set_source(ids, amp, w0, 0.0, 0.3)
    if plasma:
        m.set_plasma((0.3 / h) ** 2 * (1 + xy[:, 0]), 0.5)
    rng = np.random.default_rng(3)
    B, E, j = rng.standard_normal(m.n_tris), rng.standard_normal(m.n_edges), rng.standard_normal(m.n_edges)
    m.write_fields(E, B, j if plasma else None)
    m.set_step(7)
    for _ in range(calls):
        m.step_n(steps)
    assert m.check()[0]
    out = list(m.read_fields(j=plasma))[:3 if plasma else 2]
    if frame:
        out += list(m.frame_fields())
    out += [m.get_step(), m.energy(), m.stats()["kernel_launches"]]
    m.close()
    return out


def _same(a, b):
    for x, y in zip(a[:-1], b[:-1]):
        assert np.array_equal(x, y)
    assert a[-1] < b[-1]      # the resident calls launch fewer kernels


@pytest.mark.parametrize("n_t", [1, 2, 33, 1024, 1025, 2048, 2049, 2081, 4865])
@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("plasma", [False, True])
def test_resident_is_bit_identical_to_plain(ue, n_t, fp64, plasma):
    xy, tris, h = _lattice(n_t, n_t)
    kw = dict(plasma=plasma, calls=2, precision=ue.UE_PREC_FP64 if fp64 else ue.UE_PREC_FP32)
    _same(_run(ue, xy, tris, h, 45, 32, **kw), _run(ue, xy, tris, h, 45, -1, **kw))


@pytest.mark.parametrize("n_t", [155_648, 155_649, 311_297, 622_592, 622_593, 1_245_184, 1_245_185])
@pytest.mark.parametrize("plasma", [False, True])
def test_resident_at_the_edges_of_its_shapes(ue, n_t, plasma):
    """152 CTAs of 1,024, 2,048, 4,096 and, without a current, 8,192 triangles (which of the
    largest run resident depends on how many neighbours of a CTA lie in others)."""
    xy, tris, h = _lattice(n_t, 5)
    kw = dict(plasma=plasma)
    a, b = _run(ue, xy, tris, h, 33, 32, **kw), _run(ue, xy, tris, h, 33, -1, **kw)
    for x, y in zip(a[:-1], b[:-1]):
        assert np.array_equal(x, y)
    assert a[-1] < b[-1] if n_t <= (622_592 if plasma else 622_593) else True
    assert a[-1] >= b[-1] if n_t > (622_592 if plasma else 1_245_184) else True


def test_resident_fp64_with_two_slots(ue):
    xy, tris, h = _lattice(200_001, 5)
    kw = dict(plasma=True, precision=ue.UE_PREC_FP64)
    _same(_run(ue, xy, tris, h, 33, 32, **kw), _run(ue, xy, tris, h, 33, -1, **kw))


@pytest.mark.parametrize("n_t,shuffle", [(155_648, False), (155_649, False), (311_296, False), (7_000, True),
                                         (60_000, True), (280_000, True)])
@pytest.mark.parametrize("plasma", [False, True])
def test_resident_fp64_edges_apart(ue, n_t, shuffle, plasma):
    """FP64 at the edges of its shapes, and with nearly every edge between two CTAs (up to a full list of
    remote neighbours, and past it, where the launches stay): fields bit for bit, a watchdog's energy."""
    xy, tris, h = _lattice(n_t, 5, shuffle=shuffle)
    kw = dict(plasma=plasma, precision=ue.UE_PREC_FP64, load=dict(reorder=ue.UE_REORDER_NONE) if shuffle else None)
    a = _run(ue, xy, tris, h, 33, 32, watchdog_every=16, **kw)
    b = _run(ue, xy, tris, h, 33, -1, **kw)
    for x, y in zip(a[:-1], b[:-1]):
        assert np.array_equal(x, y)
    m = ue.Mesh(xy, tris, **(kw["load"] or {}))
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.1 * h, graph_chunk=32, watchdog_every=32, precision=ue.UE_PREC_FP64)
    m.write_fields(B=np.cos(np.arange(m.n_tris)))
    m.step_n(64)
    W = m.check()[1]
    # the same positive terms in another order
    assert abs(W / m.energy() - 1) <= 4 * n_t * 1.2e-16
    m.close()


@pytest.mark.parametrize("n_t", [7_000, 400_000])
def test_resident_with_scattered_neighbours(ue, n_t):
    """The caller's order kept and random: nearly every neighbour is in another CTA; the larger
    mesh has more than a CTA lists and keeps its launches."""
    xy, tris, h = _lattice(n_t, 5, shuffle=True)
    kw = dict(plasma=True, load=dict(reorder=ue.UE_REORDER_NONE))
    a, b = _run(ue, xy, tris, h, 40, 32, **kw), _run(ue, xy, tris, h, 40, -1, **kw)
    for x, y in zip(a[:-1], b[:-1]):
        assert np.array_equal(x, y)
    assert (a[-1] < b[-1]) == (n_t < 10_000)


@pytest.mark.parametrize("tiled", [False, True])
@pytest.mark.parametrize("plasma", [False, True])
@pytest.mark.parametrize("frame,order", [(1, 3), (16, 3), (5, 1)])
def test_resident_with_a_frame(ue, tiled, plasma, frame, order):
    ms = meshgen.graded_square(0.05, 0.05, holes=[meshgen.polygon_triangle((0.5, 0.5), 0.3)], seed=4)
    kw = dict(plasma=plasma, frame=frame)
    plain = _run(ue, ms.xy, ms.tris, 0.05, 70, -1, load=dict(reorder=ue.UE_REORDER_GREEDY_RINGS, tile_tris=200) if tiled else None, **kw)
    if tiled:
        kw.update(load=dict(reorder=ue.UE_REORDER_GREEDY_RINGS, tile_tris=200), variant=ue.UE_VARIANT_BLOCKED, block_depth=4)
    _same(_run(ue, ms.xy, ms.tris, 0.05, 70, 32, **kw), plain)


def test_resident_batch_and_watchdog(ue):
    """A batch of meshes with their own sources, and the watchdog's checks at the same steps."""
    out, energy = [], []
    for chunk in (32, -1):
        meshes = []
        for n_t in (300, 4097, 2500):
            xy, tris, h = _lattice(n_t, n_t)
            m = ue.Mesh(xy, tris)
            m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.1 * h, graph_chunk=chunk, watchdog_every=32)
            ids, amp = meshgen.source_line_amplitudes(xy, tris, float(xy[:, 0].mean()), h)
            m.set_source(ids, amp, 1.0 / h, 0.0, 0.3)
            meshes.append(m)
        b = ue.batch_create(meshes)
        b.write_fields(B=np.cos(np.arange(b.n_tris)))
        b.step_n(64)
        ok, W, flag = b.check()
        E, B, _ = b.read_fields()
        assert ok and flag == 0
        out.append((E, B))
        energy.append(W)
        b.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
    assert abs(energy[0] / energy[1] - 1) < 1e-13      # the same terms, summed in another order


@pytest.mark.parametrize("every", [1, 32, 40, 100])
@pytest.mark.parametrize("n_t", [500, 5000])
def test_resident_watchdog_checks_at_the_same_steps(ue, every, n_t):
    """The energy at the last check over calls that end inside and between the checks' steps, and a
    run above the stability bound flagged."""
    xy, tris, h = _lattice(n_t, 3)
    calls, unit = (70, 32, 110, 45, 2000), 32
    # the launches' checks: at the ends of the graph chunks and of the call, once `every` is reached
    ends, since, at, last = [], 0, 0, 0
    for n in calls:
        for part in [unit] * (n // unit) + ([n % unit] if n % unit else []):
            at, since = at + part, since + part
            if since >= every:
                since, last = 0, at
        ends.append((at, last))
    m = ue.Mesh(xy, tris)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.1 * h, graph_chunk=unit, watchdog_every=every)
    m.write_fields(B=np.cos(np.arange(m.n_tris)))
    r = ue.Mesh(xy, tris)
    r.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.1 * h, graph_chunk=-1)
    r.write_fields(B=np.cos(np.arange(r.n_tris)))
    stepped, ref = 0, 0.0
    for n, (_, last) in zip(calls, ends):
        m.step_n(n)
        if last > stepped:
            r.step_n(last - stepped)
            stepped, ref = last, r.energy()
        ok, W, flag = m.check()
        assert ok and flag == 0
        # the same positive terms summed in another order, fewer than n_t + n_ei additions deep
        assert abs(W - ref) <= 4 * n_t * 2.3e-16 * ref
    m.close()
    r.close()
    # a step above the stability bound is flagged inside the launch
    m = ue.Mesh(xy, tris)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.8 * h, graph_chunk=unit, watchdog_every=every, watchdog_growth=10.0)
    m.write_fields(B=np.cos(np.arange(m.n_tris)))
    m.step_n(960)
    ok, _, flag = m.check()
    m.close()
    assert not ok and flag in (1, 2)


def test_resident_wait_that_runs_out_is_reported(ue):
    """One CTA that never publishes (test hook): the others' waits end after about a second,
    UE_ERR_TIMEOUT is reported, and the rebuilt mesh steps normally."""
    xy, tris, h = _lattice(5000, 2)
    m = ue.Mesh(xy, tris)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.1 * h, graph_chunk=32, test_skip_cta=1)
    m.write_fields(B=np.ones(m.n_tris))
    m.step_n(32)
    ok, _, flag = m.check()
    m.close()
    assert not ok and flag == 3
    _same(_run(ue, xy, tris, h, 40, 32), _run(ue, xy, tris, h, 40, -1))
