"""Line lattices (nx = ny = 1) run many steps per launch in the default fusion mode; the populations,
fields and time must be those of single steps (mode 0) bit for bit."""
import numpy as np
import pytest

from paper_2309_08068_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

SCALE = {"f32": 0.0, "bf16": 0.0, "f16": 2.0 ** 10, "f24": 2.0 ** 10}


def lattice(w, f, mode, storage="f32", stream=None):
    from paper_2309_08068_gb300.lbm import lattice_from_workload
    L = lattice_from_workload(w, init=False, storage=storage, storage_scale=SCALE[storage], stream=stream)
    L.set_step_fusion(mode)
    L.set_populations(np.asarray(f, np.float32) * 1e-3, 3)
    return L


def state(L):
    return L.populations_host(), L.fields_host("EBDHJ"), L.time


def assert_same(a, b):
    assert np.all(np.isfinite(a[0]))
    assert np.array_equal(a[0], b[0])
    assert all(np.array_equal(a[1][k], b[1][k]) for k in a[1])
    assert a[2] == b[2]


# A block holds 128 cells; a launch takes at most 56 steps (core of 16 cells), fewer for long lines or
# many sources. Lengths around the wrap-around (shorter than the halo), the core and the block.
@pytest.mark.parametrize("model", ["mm", "hv"])
@pytest.mark.parametrize("nz,steps", [(1, 60), (2, 57), (3, 56), (15, 2), (16, 113), (17, 55), (127, 3), (128, 57),
                                      (129, 112), (2433, 60), (9001, 41), (20011, 33)])
def test_line_equals_single_steps(model, nz, steps):
    for media in ("vacuum", "few", "random"):
        w, f = wl.random_state(model, (1, 1, nz), seed=nz, media=media, n_sources=3)
        got = []
        for mode in (1, 0):
            L = lattice(w, f, mode)
            L.step(steps)
            L.step(1)
            L.step(2)
            got.append(state(L))
            L.close()
        assert_same(*got)


@pytest.mark.parametrize("model", ["mm", "hv"])
@pytest.mark.parametrize("storage", ["bf16", "f16", "f24"])
def test_line_rounds_every_step_to_the_storage_format(model, storage):
    w, f = wl.random_state(model, (1, 1, 301), seed=8, media="few")
    got = []
    for mode in (1, 0):
        L = lattice(w, f, mode, storage)
        L.step(61)
        got.append(state(L))
        L.close()
    assert_same(*got)


@pytest.mark.parametrize("model", ["mm", "hv"])
def test_line_with_every_source_slot(model):
    """16 sources that share cells: currents and imposed fields add in slot order; a launch then takes
    at most 32 steps. A table that ends in an infinity reaches its own cells only."""
    w, f = wl.random_state(model, (1, 1, 200), seed=9, media="few", n_sources=16)
    for k, s in enumerate(w.sources):
        s.cells = np.sort((np.asarray(s.cells) % 7) + 60) if k % 3 else np.array([199, 0, 1, 63, 64][: len(s.cells)])
        s.cells = np.unique(s.cells)
        s.w = None if s.w is None else s.w[: s.cells.size]
    got = []
    for mode in (1, 0):
        L = lattice(w, f, mode)
        L.step(70)
        got.append(state(L))
        L.close()
    assert_same(*got)
    w.sources = w.sources[:1]
    w.sources[0].fn = wl.TimeFunction("table", 1.0, table=np.array([0.0] * 9 + [np.inf]))
    finite = []
    for mode in (1, 0):
        L = lattice(w, f, mode)
        L.step(8)
        finite.append(np.isfinite(L.populations_host()))
        L.close()
    assert np.array_equal(*finite) and not finite[0].all() and finite[0].any()


def test_lines_in_a_batch_equal_their_own_steps():
    """Up to six line lattices step on their own inside a batch, more in the batched launches."""
    from paper_2309_08068_gb300.lbm import Batch
    stream = torch.cuda.Stream()
    for count in (2, 9):
        works = [wl.random_state("mm", (1, 1, 40 + 50 * k), seed=k, media="few") for k in range(count)]
        steps = [30 + 7 * k for k in range(count)]
        solo = [lattice(w, f, 1, stream=stream) for w, f in works]
        group = [lattice(w, f, 1, stream=stream) for w, f in works]
        batch = Batch(group)
        for L, n in zip(solo, steps):
            L.step(n)
        batch.step(steps)
        for A, B in zip(solo, group):
            assert_same(state(A), state(B))
        batch.close()
        for L in solo + group:
            L.close()
