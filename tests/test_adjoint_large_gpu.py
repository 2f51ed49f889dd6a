"""The MM backward step of large lattices with a medium per cell (more than 1,200,000 cells) is launched
plainly and reads the adjoint and the records as read-only data. Loss and gradients against the FP64 oracle,
with the tolerances of the other adjoint tests, on the smallest such lattice."""
import numpy as np
import pytest

from helpers import oracle_from_workload, rel_l2
from test_adjoint_gpu import GRAD_TOL, LOSS_TOL, gpu_adjoint, small_case

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("interval", [-1, 2])
def test_large_backward_steps_match_the_oracle(interval):
    w, f0, plane = small_case("mm", seed=97, shape=(108, 108, 103), plane=(0, 5))
    steps = 3
    L, loss, ge, gs = gpu_adjoint(w, f0, steps, plane, interval=interval)
    O = oracle_from_workload(w, init=False, threads=16)
    O.set_populations(f0, 3)
    loss_ref, ge_ref, gs_ref = O.loss_and_gradient(steps, *plane)
    assert abs(loss - loss_ref) <= LOSS_TOL * loss_ref
    assert np.abs(ge_ref).max() > 0 and rel_l2(ge, ge_ref) <= GRAD_TOL
    assert rel_l2(gs, gs_ref) <= GRAD_TOL
    L.close()
