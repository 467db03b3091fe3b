"""FP64 solves in their default form do not fail on a device wait that runs out (a 1 ns limit
makes it run out on the first wait that is not met at once): they go on in two launches per
iteration from the iterate reached, in a step and in the adjoint, as these had no wait before
the on-chip form became their default."""
import numpy as np
import pytest

from paper_1808_04099_gb300 import workloads as W
from _util import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import adjoint, bcm  # noqa: E402

# both sides solve to a relative residual of 1e-12; over these sizes (64 cells along an axis)
# the pressure's error is under N^2 / pi^2 = 415 times that each
TOL = 2 * 415 * 1e-12


def test_steps():
    spec = W.cavity(4, 16)
    state = W.initial_state(spec, 5, 1e-2)
    out = []
    for limit in (1e-9, 2.0):
        g = bcm.Grid(spec, bcm.PREC_F64)
        g.load_state(state)
        g.set_solver(barrier_timeout_s=limit)
        st = g.step(2, rtol=1e-12)
        assert st[0]["converged"] == 1 and st[0]["pcg_form"] == (0 if limit < 1 else 3)
        out.append(np.concatenate([g.numpy(f) for f in (bcm.U, bcm.V, bcm.W)]))
    assert rel_l2(out[0], out[1]) <= TOL


def test_adjoint():
    L = (3.0, 2.0, 2.0)
    spec = W.sphere_channel(6, 4, 4, 16, L, 0.25, (0.75, 1.0, 1.0))
    out = []
    for limit in (1e-9, 2.0):
        run = adjoint.AdjointRun(spec, np.linspace(-0.05, 0.05, 8), (0.75, 1.0, 1.0), 0.25, 2)
        J = run.forward()
        run.g.set_solver(barrier_timeout_s=limit)
        da, dc = run.backward()
        out.append(np.concatenate([[J], da, dc]))
    assert rel_l2(out[0], out[1]) <= 10 * TOL  # two steps and their transposes
