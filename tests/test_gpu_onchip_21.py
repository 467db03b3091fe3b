"""2:1 ghosts of the on-chip PCG from the items' tables: two-level grids whose launch shape
has whole cubes and slabs of every depth, items of several cubes a block, in the FP32 inner
solve (and FP64, which goes through the cubes' tables), against the two-launch form."""
import pytest

from paper_1808_04099_gb300 import workloads as W
from _util import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402

# B, level-0 cubes, refined box, planes per item on 152 SMs
GRIDS = [(16, (4, 4, 4), (1, 1, 1), (3, 3, 3), 16), (16, (5, 5, 5), (2, 1, 1), (3, 4, 4), 4),
         (16, (7, 5, 5), (2, 1, 1), (5, 4, 4), 0), (8, (5, 5, 5), (2, 1, 1), (3, 4, 4), 4),
         (8, (7, 5, 5), (2, 1, 1), (5, 4, 4), 4), (8, (8, 6, 6), (2, 1, 1), (6, 5, 5), 8),
         (4, (5, 5, 5), (2, 1, 1), (3, 4, 4), 4), (4, (10, 10, 10), (3, 1, 1), (7, 9, 9), 4)]


@pytest.mark.parametrize("prec,tol", [(bcm.PREC_F64, 1e-12), (bcm.PREC_F32_REFINE, 1e-5)])
@pytest.mark.parametrize("B,n,lo,hi,planes", GRIDS)
def test_iterates_equal_the_two_launch_form(B, n, lo, hi, planes, prec, tol):
    spec = W.two_level_channel(*n, B, lo, hi, 1.0 / (4.0 * B))
    if prec != bcm.PREC_F64 and planes and \
            torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert bcm.onchip_shape(B, spec.n_cubes, 1, 1, False)["planes"] == planes
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    rhs = torch.randn(spec.n_cells, generator=gen, device="cuda", dtype=torch.float64)

    def iterate(k, form):
        g = bcm.Grid(spec, prec)
        if form == 0:
            g.set_launch(1, 1, persistent=0)
        g.set_solver(inner_rtol=1e-30, max_cycles=1)
        g.field(bcm.RHS).copy_(rhs)
        g.field(bcm.P).zero_()
        assert g.solve_pressure_iters(k)[0]["pcg_form"] == form
        return g.numpy(bcm.P)

    for k in (1, 2, 7):
        assert rel_l2(iterate(k, 3), iterate(k, 0)) <= tol, k
