"""Float32 field transfers of a batch: the same fields as the double transfers."""
import numpy as np
import pytest

import meshgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pin", [False, True])
def test_float32_transfers_of_a_batch(pin):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_01448_gb300 import build
    build.build()
    import paper_1812_01448_gb300 as ue
    meshes = []
    for n in (9, 12):
        ms = meshgen.equilateral_lattice(n, 0.1, jitter=0.1, seed=n)
        m = ue.Mesh(ms.xy, ms.tris)
        m.geometry_build(dt_mode=ue.UE_DT_GIVEN, dt=0.01)
        meshes.append(m)
    b = ue.batch_create(meshes)
    mem = lambda n: (torch.zeros(n, dtype=torch.float32).pin_memory() if pin else torch.zeros(n)).numpy()  # noqa: E731
    E, B = mem(b.n_edges), mem(b.n_tris)
    E[:] = np.sin(np.arange(b.n_edges))
    B[:] = np.cos(np.arange(b.n_tris))
    b.write_fields_f32(E=E, B=B)      # the batch's first transfer of any kind
    E32, B32, _ = b.read_fields_f32(out={"E": mem(b.n_edges), "B": mem(b.n_tris)})
    E64, B64, _ = b.read_fields()
    b.close()
    assert np.array_equal(B32, B) and np.array_equal(B64, B.astype(np.float64))
    assert np.array_equal(E32, E64.astype(np.float32))
    inside = E64 != 0
    assert inside.any() and np.abs(E64[inside] / E[inside] - 1).max() < 2e-7
