"""The forms Lattice.fields takes: letters as a string or a list, one or several, a caller's output
buffer, another current stream; on a whole lattice (source cells within the one launch) and on a
z-slab (source cells in a launch of their own). All give fields_host's values."""
import numpy as np
import pytest

from paper_2309_08068_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("model", ["mm", "hv"])
@pytest.mark.parametrize("z_ghost", [False, True])
def test_fields_forms(model, z_ghost):
    from paper_2309_08068_gb300.lbm import Lattice
    shape = (19, 7, 11)
    w, f = wl.random_state(model, shape, seed=4, media="few", n_sources=0)
    plane = shape[0] * shape[1]
    cells = np.arange(plane, plane * 10, 5)  # inner planes, several blocks of 256 cells
    w.sources = [wl.Source("current", cells, wl.TimeFunction("sin", 1.0, 7.0, 0.4),
                           w=np.random.default_rng(2).standard_normal((cells.size, 3)))]
    L = Lattice(model, shape, w.eps_r, w.mu_r, w.sigma, z_ghost=z_ghost)
    for s in w.sources:
        L.add_source(s)
    L.set_populations(np.asarray(f, np.float32), 3)
    ref = L.fields_host("EBDHJ")
    for names in ("E", "J", "EB", "BE", "EBDHJ", ["D"], ("H", "E")):
        got = L.fields(names)
        assert set(got) == set(names)
        for c in names:
            assert got[c].shape == (3, L.n) and np.array_equal(got[c].cpu().numpy(), ref[c]), (names, c)
    out = torch.empty((2, 3, L.n), device="cuda")
    got = L.fields("HD", out)
    assert np.array_equal(out[0].cpu().numpy(), ref["D"]) and got["H"].data_ptr() == out[1].data_ptr()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        got = L.fields("EJ")
        total = got["E"] + got["J"]
    side.synchronize()
    assert np.array_equal(total.cpu().numpy(), ref["E"] + ref["J"])
    L.close()
