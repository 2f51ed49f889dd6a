"""Single steps of small lattices look their source cells up before the step, larger ones recompute
them after it; the batched launches always recompute. All must agree bit for bit, on lattices on both
sides of the line (1140 blocks of 256 cells), with dense, shared and sparse source cells, and on a
lattice of one block."""
import numpy as np
import pytest

from paper_2309_08068_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("model", ["mm", "hv"])
@pytest.mark.parametrize("shape", [(5, 3, 2), (37, 19, 11), (66, 66, 66), (66, 66, 68)])
@pytest.mark.parametrize("storage", ["f32", "f16", "f24"])
def test_step_equals_batched_step(model, shape, storage):
    from paper_2309_08068_gb300.lbm import Batch, lattice_from_workload
    n = int(np.prod(shape))
    w, f = wl.random_state(model, shape, seed=n % 97, media="few", n_sources=4)
    full = np.arange(0, n, 1 if n < 10000 else 3)  # every cell of some blocks, several sources on some cells
    w.sources.append(wl.Source("current", full[: 3000], wl.TimeFunction("sin", 0.3, 11.0, 0.1),
                               w=np.random.default_rng(1).standard_normal((full[:3000].size, 3))))
    w.sources.append(wl.Source("impose", full[-20:], wl.TimeFunction("const", 0.5), E0=(1, 2, 3), B0=(-1, 0, 2)))
    stream = torch.cuda.Stream()
    scale = 0.0 if storage == "f32" else 2.0 ** 8
    pair = []
    for _ in range(2):
        L = lattice_from_workload(w, init=False, stream=stream, storage=storage, storage_scale=scale)
        L.set_step_fusion(0)
        L.set_populations(np.asarray(f, np.float32) * 1e-2, 4)
        pair.append(L)
    pair[0].step(4)
    batch = Batch(pair[1:])
    batch.step(4)
    a, b = pair[0].populations_host(), pair[1].populations_host()
    assert np.all(np.isfinite(a)) and np.array_equal(a, b)
    batch.close()
    for L in pair:
        L.close()
