"""The batch tuner times the form that the whole batch will launch: a sample that fits the chip is kept from
the resident step when the batch does not fit."""
import numpy as np
import pytest

import meshgen
from paper_1812_01448_gb300 import tune

CANDS = (("plain", "kd", 400, 1, 512), ("persistent", "kd", 400, 1, 512), ("blocked", "kd", 400, 4, 512))


def _items(n, n_min, n_max):
    items = []
    for sp in meshgen.batch_specs(n, seed=77, n_min=n_min, n_max=n_max):
        ms = meshgen.batch_mesh(sp)
        ids, amp = meshgen.source_line_amplitudes(ms.xy, ms.tris, 0.3, ms.h)
        items.append((ms, ids, amp, sp["omega0"]))
    return items


@pytest.mark.parametrize("over", [False, True])
def test_the_sample_is_timed_as_the_batch_runs(monkeypatch, over):
    items = _items(4, 600, 1500)
    total = sum(ms.n_tris for ms, *_ in items)
    seen = []

    def fake_time(sub, variant, tile, depth, threads, **kw):
        seen.append((variant, kw["resident"]))
        return 1e9
    monkeypatch.setattr(tune, "time_batch", fake_time)
    monkeypatch.setattr(tune, "resident_capacity", lambda: total - 1 if over else total)
    _, table = tune.autotune_batch(items, candidates=CANDS, sample=2)
    assert table["resident"] is (not over) and table["sample_meshes"] == 2
    assert seen == [(c[0], not over) for c in CANDS]


@pytest.mark.gpu
def test_time_batch_keeps_the_launches(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_01448_gb300 import build
    build.build()
    import paper_1812_01448_gb300 as ue
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert ue.resident_capacity() == sms * 8192 and ue.resident_capacity(ue.UE_PREC_FP64) == sms * 2048
    items, runs = _items(3, 1500, 4000), []

    def create(meshes, stream=None):
        b = ue.batch_create(meshes, stream)
        close = b.close

        def counted():
            if b._h:
                runs.append(b.stats()["resident_launches"])
            close()
        b.close = counted
        return b
    monkeypatch.setattr(tune, "batch_create", create)
    for variant in ("plain", "blocked", "persistent"):
        for resident in (True, False):
            rate = tune.time_batch(items, variant, 400, 4, 512, steps=64, warmup=32, resident=resident)
            assert rate > 0 and np.isfinite(rate)
            assert (runs[-1] > 0) == (resident and variant != "persistent")
