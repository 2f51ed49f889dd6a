"""lbm_step captured by the caller into a CUDA graph: the first call of a context, and the first after its
sources changed, may be the captured one (the two-step passes then build their source-cell lists inside the
capture). Replays must give the populations of the same steps launched directly, bit for bit."""
import numpy as np
import pytest

from paper_2309_08068_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


# HV lattices of about a wave of tiles and larger and MM ones of a few waves step as tiled passes, flat ones of
# large planes as ring passes (singly in a capture), the others singly or, lines, many steps per launch; an even number of steps leaves the buffers as a replay finds them
@pytest.mark.parametrize("model,shape,steps", [("hv", (80, 80, 80), 4), ("hv", (97, 53, 71), 4), ("mm", (96, 96, 96), 4),
                                               ("mm", (30, 20, 10), 4), ("hv", (64, 64, 64), 2), ("hv", (80, 80, 80), 2),
                                               ("mm", (96, 96, 96), 6), ("mm", (1, 1, 700), 120), ("hv", (1, 1, 700), 2),
                                               ("mm", (256, 160, 11), 4)])
@pytest.mark.parametrize("before", ["nothing", "steps", "sources"])
def test_captured_steps_equal_direct_ones(model, shape, steps, before):
    from paper_2309_08068_gb300.lbm import lattice_from_workload
    w, f = wl.random_state(model, shape, seed=sum(shape), media="few", n_sources=3)
    for s in w.sources:
        s.fn = wl.TimeFunction("const", 0.5)  # a replay repeats the captured steps' source values
    stream = torch.cuda.Stream()
    out = []
    for captured in (True, False):
        L = lattice_from_workload(w, init=False, stream=stream)
        if before != "nothing":
            L.step(2)
        if before == "sources":
            L.add_source(wl.Source("current", np.arange(7), wl.TimeFunction("const", 0.25), w=np.ones((7, 3))))
        L.set_populations(np.asarray(f, np.float32) * 1e-2, 0)
        L.sync()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                L.step(steps)
            with torch.cuda.stream(stream):
                graph.replay()
                graph.replay()
        else:
            L.step(2 * steps)
        out.append(L.populations_host())
        L.close()
    assert np.all(np.isfinite(out[0])) and np.array_equal(*out)
