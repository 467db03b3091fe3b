"""On-chip PCG with several sims per block: sims of one block that converge at different
iterations each return the iterate that their reported residual belongs to (the last
x += alpha p of a sim is not lost to the decisions of the next iteration), with x in
registers and in global memory, whatever the number of sims of a block; and two sims of
4^3 cubes, in numbers of cubes for which half cubes would spread the cells better, give the
two-launch form's iterates (every cell is in its sim's dot products)."""
import numpy as np
import pytest

from paper_1808_04099_gb300 import workloads as W
from _util import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


def channel(nx, ny, nz, B):
    L = tuple(n * B / 16.0 for n in (nx, ny, nz))
    return W.sphere_channel(nx, ny, nz, B, L, L[1] / 8, tuple(e / 2 for e in L))


def mixed_sims(n, B):
    """n sims of 1 to 12 cubes (closed boxes, channels, periodic boxes) in turn."""
    kinds = [W.cavity(1, B), channel(2, 2, 1, B), W.periodic_box(1, B), channel(3, 2, 2, B),
             W.cavity(2, B)]
    return W.concat([kinds[i % len(kinds)] for i in range(n)])


SPECS = {
    "few_8": lambda: mixed_sims(7, 8),
    "many_8": lambda: mixed_sims(96, 8),        # several sims per block, x in registers
    "most_8": lambda: mixed_sims(240, 8),       # ... and in global memory
    "small_16": lambda: mixed_sims(40, 16),     # items of whole cubes of 16^3
}
RTOL = 1e-10


def true_residuals(g, spec, b):
    """||b - A p|| / ||b|| of every sim, formed anew from the pressure (K p = -V (b - mean))."""
    y = g.apply_poisson(g.field(bcm.P)).cpu().numpy()
    b, B3 = b.cpu().numpy(), spec.B ** 3
    out = []
    for s in range(spec.n_sims):
        lo, hi = int(spec.sim_cube_offset[s]) * B3, int(spec.sim_cube_offset[s + 1]) * B3
        q = b[lo:hi]
        if W.OUTFLOW not in list(spec.sim_bc[s]):
            q = q - q.mean()
        rhs = -float(spec.sim_h0[s]) ** 3 * q
        out.append(np.linalg.norm(rhs - y[lo:hi]) / np.linalg.norm(rhs))
    return np.array(out)


@pytest.mark.parametrize("name", SPECS)
def test_reported_residual_is_that_of_the_iterate(name):
    spec = SPECS[name]()
    g = bcm.Grid(spec, bcm.PREC_F64)
    gen = torch.Generator(device="cuda")
    for seed in range(4):
        gen.manual_seed(seed)
        b = torch.randn(spec.n_cells, generator=gen, device="cuda", dtype=torch.float64)
        g.field(bcm.RHS).copy_(b)
        g.field(bcm.P).zero_()
        st = g.solve_pressure(rtol=RTOL)
        assert all(s["pcg_form"] == 3 for s in st)
        rel = true_residuals(g, spec, b)
        # the recurrence's residual ends at or below RTOL; the one formed anew differs from it
        # by rounding, under 2^-53 * 12 |p| h / |rhs| <= 12 * 2^-53 N^2 / pi^2 for N <= 48
        # cells along a sim: 4e-13.  Without its last update an iterate stands above RTOL.
        assert rel.max() <= RTOL * 1.01, (seed, int(rel.argmax()), rel.max())


@pytest.mark.parametrize("prec,tol", [(bcm.PREC_F64, 1e-12), (bcm.PREC_F32_REFINE, 1e-5)])
@pytest.mark.parametrize("sizes", [((1, 1, 1), (1, 1, 1)), ((2, 2, 2), (3, 2, 1)),
                                   ((2, 2, 2), (7, 1, 1)), ((7, 2, 2), (7, 2, 2)),
                                   ((5, 4, 3), (5, 4, 3)), ((10, 5, 5), (10, 5, 5))])
def test_two_sims_of_small_cubes(sizes, prec, tol):
    spec = W.concat([channel(*n, 4) for n in sizes])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    rhs = torch.randn(spec.n_cells, generator=gen, device="cuda", dtype=torch.float64)

    def iterate(k, form):
        g = bcm.Grid(spec, prec)
        if form == 0:
            g.set_launch(1, 1, persistent=0)
        g.set_solver(inner_rtol=1e-30, max_cycles=1)
        g.field(bcm.RHS).copy_(rhs)
        g.field(bcm.P).zero_()
        st = g.solve_pressure_iters(k)
        assert all(s["pcg_form"] == form and s["cg_iters"] == k for s in st)
        return g.numpy(bcm.P)

    for k in (1, 4):
        assert rel_l2(iterate(k, 3), iterate(k, 0)) <= tol, k
