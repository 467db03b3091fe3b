"""The on-chip PCG (bcm_stats.pcg_form 3), which runs every Jacobi solve whose vectors fit
the chip unless a launch shape is asked for: after exactly k iterations its iterate is the
two-launch form's up to rounding, in FP64 and in the FP32 inner solve of one
defect-correction cycle, on cubes of 4^3, 8^3 and 16^3, whole and cut into slabs, from one
cube to the largest grid that fits, with every face kind, 2:1 faces and several sims per
block; one cube more than fits takes the streaming form."""
import pytest

from paper_1808_04099_gb300 import workloads as W
from _util import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


def channel(nx, ny, nz, B):
    h = 1.0 / 16
    L = tuple(n * B * h for n in (nx, ny, nz))
    return W.sphere_channel(nx, ny, nz, B, L, L[1] / 8, tuple(e / 2 for e in L))


SPECS = {
    "one_cube_16": lambda: W.periodic_box(1, 16),          # cut into slabs
    "one_cube_4": lambda: W.periodic_box(1, 4),
    "few_16": lambda: channel(3, 2, 1, 16),
    "ragged_8": lambda: channel(7, 3, 5, 8),                # 105 cubes, several blocks each
    "many_8": lambda: channel(11, 9, 8, 8),                 # 792 cubes: whole-cube blocks
    "many_4": lambda: channel(13, 11, 9, 4),
    "whole_16": lambda: channel(9, 7, 7, 16),               # 441 cubes, three per block
    "two_level_16": lambda: W.two_level_channel(5, 4, 4, 16, (1, 1, 1), (4, 3, 3), 1 / 64.),
    "two_level_8": lambda: W.two_level_channel(6, 5, 5, 8, (1, 1, 1), (5, 4, 4), 1 / 32.),
    "two_level_4": lambda: W.two_level_channel(4, 4, 4, 4, (1, 1, 1), (3, 3, 3), 1 / 16.),
    "sims_16": lambda: W.batched_mix(7, 3, 16, 8, 32),
    "sims_8": lambda: W.batched_mix(40, 4, 8, 8, 24),
    "sims_4": lambda: W.concat([W.cavity(2, 4), channel(3, 2, 2, 4), W.periodic_box(1, 4),
                                W.cavity(3, 4)]),
}


def solve(spec, prec, k, rhs, two_launch):
    g = bcm.Grid(spec, prec)
    if two_launch:
        g.set_launch(1, 1, persistent=0)
    g.set_solver(inner_rtol=1e-30, max_cycles=1)  # exactly k inner iterations, one cycle
    g.field(bcm.RHS).copy_(rhs)
    g.field(bcm.P).zero_()
    st = g.solve_pressure_iters(k)
    torch.cuda.synchronize()
    return g.numpy(bcm.P), st


@pytest.mark.parametrize("prec,tol", [(bcm.PREC_F64, 1e-12), (bcm.PREC_F32_REFINE, 1e-5)])
@pytest.mark.parametrize("name", SPECS)
def test_iterates_equal_the_two_launch_form(name, prec, tol):
    spec = SPECS[name]()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)
    rhs = torch.randn(spec.n_cells, generator=gen, device="cuda", dtype=torch.float64)
    for k in (1, 2, 3, 7):
        a, sa = solve(spec, prec, k, rhs, False)
        b, sb = solve(spec, prec, k, rhs, True)
        assert all(s["pcg_form"] == 3 for s in sa) and all(s["pcg_form"] == 0 for s in sb)
        assert [s["cg_iters"] for s in sa] == [s["cg_iters"] for s in sb] == [k] * spec.n_sims
        assert rel_l2(a, b) <= tol, (k, rel_l2(a, b))


def test_largest_grid_and_one_more():
    """FP32: 28,672 cells per SM, i.e. seven cubes of 16^3 on each; one more streams."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n, form in ((7 * sms, 3), (7 * sms + 1, 1)):
        spec = channel(n, 1, 1, 16)
        rhs = torch.sin(torch.arange(spec.n_cells, device="cuda", dtype=torch.float64) / 7)
        a, sa = solve(spec, bcm.PREC_F32_REFINE, 5, rhs, False)
        b, _ = solve(spec, bcm.PREC_F32_REFINE, 5, rhs, True)
        assert sa[0]["pcg_form"] == form
        assert rel_l2(a, b) <= 1e-5
