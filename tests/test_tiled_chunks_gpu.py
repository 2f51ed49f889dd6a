"""The tiled pass on lattices of few waves of blocks, where the chunk of planes per block follows the
lattice: one long wave, a ragged last chunk, a dense source in one block. Populations must be those
of single steps bit for bit."""
import numpy as np
import pytest

from paper_2309_08068_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def stepped(w, f, mode, steps):
    from paper_2309_08068_gb300.lbm import lattice_from_workload
    L = lattice_from_workload(w, init=False)
    L.set_step_fusion(mode)
    L.set_populations(np.asarray(f, np.float32), 5)
    L.step(steps)
    out = L.populations_host(), L.pass_kind
    L.close()
    return out


@pytest.mark.parametrize("model", ["mm", "hv"])
@pytest.mark.parametrize("shape", [(92, 74, 82), (97, 53, 71), (80, 80, 80), (16, 17, 61), (300, 16, 45)])
@pytest.mark.parametrize("source", ["dipole", "columns"])
def test_few_waves_equal_single_steps(model, shape, source):
    w, f = wl.slab_case(model, shape, seed=31, media="few" if source == "columns" else "vacuum", amplitude=1e-2)
    if source == "dipole":
        cells, weights = wl.dipole_cells(shape, tuple(m // 2 for m in shape))
        w.sources = [wl.Source("current", cells, wl.TimeFunction("sin", 1.0, 9.0, 0.3), w=weights)]
    tiled, kind = stepped(w, f, 3, 5)
    assert kind == "tiled"
    single, _ = stepped(w, f, 0, 5)
    q = 48 if model == "mm" else 36
    assert np.all(np.isfinite(single))
    assert np.array_equal(tiled[:q], single[:q])
