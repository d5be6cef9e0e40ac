"""The launch forms that meshes beyond the chip step by, on small meshes kept from the resident step
(UE_VARIANT_NO_RESIDENT): graph replay, the blocked kernels on every tiler, frame regions and merged
batches, each against single plain launches bit for bit, with the kernel that ran named."""
import math

import numpy as np
import pytest

import meshgen
from oracle import leapfrog as lf, mesh as om, operators, spectral

pytestmark = pytest.mark.gpu

STEP_BY_STEP = -1     # graph_chunk: no graph


@pytest.fixture(scope="module")
def ue():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_01448_gb300 import build
    build.build()
    import paper_1812_01448_gb300 as ue
    return ue


@pytest.fixture(scope="module")
def square():
    ms = meshgen.plasma_square_mesh(20000, seed=1003)
    w0 = 2 * math.pi * 20
    ids, amp = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.35, ms.h)
    return ms, w0, meshgen.plasma_density_nodes(ms.xy, w0), (ids, amp)


@pytest.fixture(scope="module")
def holed():
    ms = meshgen.graded_square(1 / 32, 1 / 32, grade=0.0, holes=[meshgen.polygon_triangle((0.5, 0.5), 0.2)], seed=5)
    return ms, meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.35, ms.h)


def _run(ue, ms, src, w0, steps, variant, chunk=0, plasma=None, frame=0, reorder=1, tile=2048, prepare=False,
         resident=False, kernel_used=None, **opt):
    m = ue.Mesh(ms.xy, ms.tris, reorder=reorder, tile_tris=tile)
    m.frame_attach(frame)
    flag = 0 if resident else ue.UE_VARIANT_NO_RESIDENT
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.02 * ms.h, variant=variant | flag, graph_chunk=chunk, **opt)
    if prepare:
        m.step_prepare()
    if plasma is not None:
        m.set_plasma(plasma, 0.01 * w0)
    m.set_source(*src, w0, 0.0, 0.05)
    if kernel_used is not None:
        assert m.stats()["tb_kernel_used"] in kernel_used
    m.write_fields(B=np.sin(7 * ms.xy[ms.tris].mean(axis=1)[:, 0]))
    if prepare:
        m.step_prepare()
    m.step_n(steps)
    out = [a for a in m.read_fields(j=plasma is not None) if a is not None]
    if frame:
        out += list(m.frame_fields())
    out.append(m.get_step())
    assert (m.stats()["resident_launches"] > 0) == resident
    m.close()
    assert np.linalg.norm(out[0]) > 0
    return out


def _same(a, b):
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("plasma", [False, True])
@pytest.mark.parametrize("frame", [0, 6])
@pytest.mark.parametrize("fp64", [0, 1])
def test_plain_graphs(ue, holed, plasma, frame, fp64):
    ms, src = holed
    w0 = 2 * math.pi * 20
    kw = dict(plasma=meshgen.plasma_density_nodes(ms.xy, w0) if plasma else None, frame=frame, precision=fp64)
    ref = _run(ue, ms, src, w0, 100, ue.UE_VARIANT_PLAIN, chunk=STEP_BY_STEP, **kw)
    _same(_run(ue, ms, src, w0, 100, ue.UE_VARIANT_PLAIN, chunk=32, **kw), ref)
    _same(_run(ue, ms, src, w0, 100, ue.UE_VARIANT_PLAIN, chunk=32, prepare=True, **kw), ref)
    _same(_run(ue, ms, src, w0, 100, ue.UE_VARIANT_PLAIN, chunk=32, resident=True, **kw), ref)


@pytest.mark.parametrize("tile,k,steps,threads", [(512, 4, 70, 0), (1024, 8, 40, 0), (2048, 3, 64, 0), (1500, 6, 61, 1024),
                                                  (64, 5, 31, 0), (64, 10, 47, 0), (1024, 10, 43, 0)])
@pytest.mark.parametrize("tiler", ["KD", "GREEDY", "GREEDY_RINGS"])
@pytest.mark.parametrize("kernel", ["split", "fused"])
@pytest.mark.parametrize("plasma", [False, True])
def test_blocked_graphs(ue, square, tile, k, steps, threads, tiler, kernel, plasma):
    """Graph replays of whole chunks, then single launches for the rest."""
    ms, w0, dens, src = square
    kw = dict(reorder=getattr(ue, "UE_REORDER_" + tiler), tile=tile, plasma=dens if plasma else None)
    ref = _run(ue, ms, src, w0, steps, ue.UE_VARIANT_PLAIN, chunk=STEP_BY_STEP, **kw)
    # the fused kernel takes vacuum media, 512 threads and at most 1,023 source records per tile
    # (tiles of 1,024 with a 10-ring halo may hold more)
    fused = kernel == "fused" and not plasma and threads != 1024
    used = {4} if fused and (tile, k) != (1024, 10) else {1, 2, 3, 4} if fused else {1, 2, 3}
    if tile == 64:
        used &= {3, 4}    # more tiles than SMs: a pipelined form
    kw.update(block_depth=k, tb_threads=threads, tb_kernel=ue.UE_TB_FUSED if kernel == "fused" else ue.UE_TB_SPLIT)
    got = _run(ue, ms, src, w0, steps, ue.UE_VARIANT_BLOCKED, kernel_used=used, **kw)
    _same(got, ref)
    if tile == 64 and k == 5:
        _same(_run(ue, ms, src, w0, steps, ue.UE_VARIANT_BLOCKED, kernel_used=used, prepare=True, **kw), ref)


@pytest.mark.parametrize("tile,k,steps", [(256, 4, 61), (128, 8, 50), (400, 3, 37), (256, 4, 45), (4096, 4, 70)])
@pytest.mark.parametrize("plasma", [False, True])
def test_blocked_graphs_with_a_frame(ue, holed, tile, k, steps, plasma):
    """Blocked tiles beside the region next to the frame; the last case has no blocked tile."""
    ms, src = holed
    w0 = 2 * math.pi * 20
    kw = dict(plasma=meshgen.plasma_density_nodes(ms.xy, w0) if plasma else None, frame=6,
              reorder=ue.UE_REORDER_GREEDY, tile=tile)
    ref = _run(ue, ms, src, w0, steps, ue.UE_VARIANT_PLAIN, chunk=STEP_BY_STEP, **kw)
    _same(_run(ue, ms, src, w0, steps, ue.UE_VARIANT_BLOCKED, block_depth=k, **kw), ref)
    _same(_run(ue, ms, src, w0, steps, ue.UE_VARIANT_BLOCKED, block_depth=k, prepare=True, **kw), ref)


def test_blocked_against_the_oracle(ue, square):
    ms, w0, dens, (ids, amp) = square
    ops = operators.Operators(om.canonicalize(ms.xy, ms.tris))
    rho, _ = spectral.power_iteration(ops, 200)
    pl = lf.Plasma(dens, 0.01 * w0)
    dt = spectral.stable_dt(rho, 0.5, pl.nbar(ops).max())
    m = ue.Mesh(ms.xy, ms.tris, reorder=ue.UE_REORDER_GREEDY_RINGS, tile_tris=1024)
    m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=dt, variant=ue.UE_VARIANT_BLOCKED | ue.UE_VARIANT_NO_RESIDENT, block_depth=4)
    m.set_plasma(dens, 0.01 * w0)
    m.set_source(ids, amp, w0, 0.1, 0.05)
    m.step_n(1001)
    got = m.read_fields(j=True)
    assert m.stats()["resident_launches"] == 0 and m.stats()["tb_kernel_used"] in (1, 2, 3)
    m.close()
    st = lf.run(ops, lf.initial_state(ops), dt, 1001, plasma=pl, source=lf.Source(ids, amp, w0, 0.1, 0.05))
    for a, b in zip(got, (ops.extend(st.E), st.B, ops.extend(st.j))):
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)


@pytest.mark.parametrize("variant,tiler,kernel", [("PLAIN", "RCM", 0), ("BLOCKED", "KD", 0), ("BLOCKED", "GREEDY_RINGS", 0),
                                                  ("BLOCKED", "GREEDY", 1)])
def test_batches(ue, variant, tiler, kernel):
    """A merged batch's launches and graphs against its meshes stepped alone, launch by launch."""
    singles, refs = [], []
    for i, sp in enumerate(meshgen.batch_specs(5, seed=31, n_min=1500, n_max=12000)):
        ms = meshgen.batch_mesh(sp)
        src = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.3, ms.h)
        for out, var, chunk in ((singles, getattr(ue, "UE_VARIANT_" + variant) | ue.UE_VARIANT_NO_RESIDENT, 32),
                                (refs, ue.UE_VARIANT_PLAIN, STEP_BY_STEP)):
            m = ue.Mesh(ms.xy, ms.tris, reorder=getattr(ue, "UE_REORDER_" + tiler), tile_tris=400)
            m.geometry_build(power_iters=60, variant=var, block_depth=3, graph_chunk=chunk, tb_kernel=kernel)
            m.set_source(*src, sp["omega0"], 0.0, 0.05)
            m.write_fields(B=np.cos(3.0 * ms.xy[ms.tris].mean(axis=1)[:, 1] + i))
            out.append(m)
    b = ue.batch_create(singles)
    for n in (17, 37, 64):        # launches, then graph chunks and a rest
        b.step_n(n)
        for m in refs:
            m.step_n(n)
    E, B, _ = b.read_fields()
    st = b.stats()
    assert st["resident_launches"] == 0
    if variant == "BLOCKED":
        assert st["tb_kernel_used"] in ({4} if kernel else {1, 3})
    Es, Bs = zip(*(m.read_fields()[:2] for m in refs))
    assert np.array_equal(E, np.concatenate(Es)) and np.array_equal(B, np.concatenate(Bs))
    for m in [b] + singles + refs:
        m.close()


@pytest.mark.parametrize("n_t,rows", [(1_245_184, 64), (622_593, 64)])
def test_the_largest_shapes_run_resident(ue, n_t, rows):
    """A strip, so that a CTA has few neighbours in others: the 16-slot shape, full and barely used."""
    cols = -(-n_t // (2 * rows))
    r, c = np.meshgrid(np.arange(rows + 1), np.arange(cols + 1), indexing="ij")
    rng = np.random.default_rng(2)
    xy = np.stack([(c + 0.5 * r).ravel(), (math.sqrt(3) / 2 * r).ravel()], 1) + rng.uniform(-0.08, 0.08, (r.size, 2))
    p = (np.arange(cols)[:, None] + np.arange(rows)[None, :] * (cols + 1)).ravel()
    w = cols + 1
    tris = np.stack([np.stack([p, p + 1, p + w], 1), np.stack([p + 1, p + w + 1, p + w], 1)], 1).reshape(-1, 3)[:n_t]
    used = np.zeros(len(xy), bool)
    used[tris] = True
    tris = (np.cumsum(used) - 1)[tris].astype(np.int32)
    out = []
    for flag in (0, ue.UE_VARIANT_NO_RESIDENT):
        m = ue.Mesh(xy[used], tris)
        m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.1, variant=ue.UE_VARIANT_PLAIN | flag, graph_chunk=32)
        m.write_fields(B=np.cos(np.arange(n_t)))
        m.step_n(33)
        assert m.check()[0] and m.stats()["resident_launches"] == (0 if flag else 1)
        out.append(m.read_fields()[:2])
        m.close()
    _same(*out)


def test_the_flag_alone_and_with_other_variants(ue, holed):
    ms, _ = holed
    m = ue.Mesh(ms.xy, ms.tris)
    with pytest.raises(ue.UEError):
        m.geometry_build(variant=ue.UE_VARIANT_PERSISTENT | ue.UE_VARIANT_NO_RESIDENT)
    m.geometry_build(variant=ue.UE_VARIANT_NO_RESIDENT)
    m.step_n(64)
    assert m.stats()["resident_launches"] == 0
    m.geometry_build()
    m.step_n(64)
    assert m.stats()["resident_launches"] == 1
    m.close()
