"""The autotuner on FP64 grids times the default shape (the on-chip PCG where the grid fits)
and ends with it on small grids; reset_launch goes back to the default after any shape, also
in captured steps and on a grid that does not fit on chip."""
import pytest

from paper_1808_04099_gb300 import workloads as W
from _util import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import autotune, bcm  # noqa: E402


def grid(nx, ny, nz, B):
    L = tuple(n * B / 16.0 for n in (nx, ny, nz))
    g = bcm.Grid(W.sphere_channel(nx, ny, nz, B, L, L[1] / 8, tuple(e / 2 for e in L)),
                 bcm.PREC_F64)
    g.field(bcm.RHS).copy_(torch.sin(torch.arange(g.spec.n_cells, device="cuda",
                                                  dtype=torch.float64) / 7))
    return g


@pytest.mark.parametrize("size", [(4, 2, 2, 8), (4, 4, 4, 16)])
def test_small_fp64_grids_end_on_chip(size):
    g = grid(*size)
    times = autotune.tune(g, iters=30, use_cache=False)
    # (measured: 9.8 us per iteration against 27.2 in two launches at 8k cells, 16.9 against
    # 48.8 at 262k)
    assert min(times, key=times.get) == "-1,1,1", times
    assert g.solve_pressure(rtol=1e-10)[0]["pcg_form"] == 3
    p = g.numpy(bcm.P)
    h = grid(*size)  # the default
    assert h.solve_pressure(rtol=1e-10)[0]["pcg_form"] == 3
    # both solve to 1e-10; up to 64 cells along an axis (N^2 / pi^2 = 415)
    assert rel_l2(p, h.numpy(bcm.P)) <= 2 * 415 * 1e-10


def test_reset_launch():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for g, form in ((grid(4, 2, 2, 8), 3), (grid(3 * sms + 1, 1, 1, 16), 0)):
        assert g.solve_pressure_iters(3)[0]["pcg_form"] == form
        for shape in ((1, 1, 1), (2, 1, 1), (0, 2, 2)):
            g.set_launch(*shape[1:], persistent=shape[0])
            assert g.solve_pressure_iters(3)[0]["pcg_form"] == shape[0]
            g.reset_launch()
            assert g.solve_pressure_iters(3)[0]["pcg_form"] == form
    g = grid(4, 2, 2, 8)
    g.load_state(W.initial_state(g.spec, 3, 1e-2))
    forms = []
    for change in (None, lambda: g.set_launch(1, 1, persistent=1), g.reset_launch):
        if change:
            change()
        forms.append(g.step_graph(1, rtol=1e-10)[0]["pcg_form"])
    assert forms == [3, 1, 3]
