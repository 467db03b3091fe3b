"""QUICK + Crank-Nicolson on an FP64 state with the FP32 pressure solve (with and without
particles) gives the FP64 solver's fields: both pressures are solved to 1e-12, whose error in
the velocities of two steps is below 1e-9 on at most 64 cells an axis (N^2 / pi^2 = 415)."""
import numpy as np
import pytest

from paper_1808_04099_gb300 import workloads as W
from _util import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


@pytest.mark.parametrize("particles", [False, True])
@pytest.mark.parametrize("n,B", [((6, 4, 4), 4), ((4, 2, 3), 8), ((3, 2, 2), 16)])
def test_fields_equal_the_fp64_solver(n, B, particles):
    L = tuple(q * B / 16.0 for q in n)
    spec = W.sphere_channel(*n, B, L, min(L[1:]) / 5, tuple(e / 2 for e in L))
    state = W.initial_state(spec, 3, 1e-2)
    out = []
    for prec in (bcm.PREC_F64, bcm.PREC_F64_REFINE):
        g = bcm.Grid(spec, prec)
        g.load_state(state)
        g.set_momentum_scheme(bcm.SCHEME_QUICK_CN, 1e-13, 500)
        if particles:
            g.set_particles(W.surface_particles(spec))
        st = g.step(2, rtol=1e-12)
        assert st[0]["converged"] == 1 and st[0]["cn_iters"] > 1
        out.append(np.concatenate([g.numpy(f) for f in (bcm.U, bcm.V, bcm.W)]))
    assert rel_l2(out[1], out[0]) <= 1e-9
