"""The FP64 residual of a smooth pressure with a large constant in it (as a closed domain's
may have): the right-hand side is K p itself, so what is reported is rounding alone, and it
does not grow with the constant.  Differences of neighbours are exact there; their sums
round by 2^-53 of the differences' size, up to N / 2 pi = 10 times that of K p on 64 cells,
six additions on each side: under 12 * 10 * 2^-53 = 1.3e-14, plus the right-hand side's two
roundings.  With the pressure's own rounding in the sums it would be above 1e-12."""
import numpy as np
import pytest

from paper_1808_04099_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


@pytest.mark.parametrize("prec", [bcm.PREC_F64, bcm.PREC_F64_REFINE])
@pytest.mark.parametrize("mg", [False, True])
@pytest.mark.parametrize("m,B", [(4, 16), (8, 8), (16, 4)])
def test_residual_of_an_offset_pressure(m, B, mg, prec):
    spec = W.cavity(m, B)
    g = bcm.Grid(spec, prec)
    if mg:
        g.set_preconditioner(bcm.PRECOND_MULTIGRID)
    n, i = m * B, np.arange(B ** 3)
    p = np.empty(spec.n_cells)
    for c, ijk in enumerate(np.asarray(spec.cube_ijk)):
        x = [(ijk[d] + (i // B ** d) % B + 0.5) / n for d in range(3)]
        p[c * B ** 3:(c + 1) * B ** 3] = 0.5 * np.cos(np.pi * x[0]) * np.cos(2 * np.pi * x[1]) \
            * np.cos(np.pi * x[2])
    p = torch.from_numpy(100.0 + p).cuda()
    b = -g.apply_poisson(p) / float(spec.sim_h0[0]) ** 3
    g.field(bcm.RHS).copy_(b)
    g.field(bcm.P).copy_(p)
    st = g.solve_pressure(rtol=1e-3)
    assert st[0]["converged"] == 1 and st[0]["cg_iters"] == 0
    assert st[0]["rel_resid"] <= 1.3e-14 + 3 * 2.0 ** -53
