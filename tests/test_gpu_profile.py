"""The kernel profile counts what ran: an FP64 grid one cube too large for the on-chip PCG
has no launch of class "pcg", one that fits has one per solve."""
import pytest

from paper_1808_04099_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


def test_no_launch_is_counted_for_a_form_that_does_not_fit():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n, form in ((3 * sms, 3), (3 * sms + 1, 0)):  # three 16^3 cubes per SM are the most
        L = (float(n), 1.0, 1.0)
        spec = W.sphere_channel(n, 1, 1, 16, L, 0.1, tuple(e / 2 for e in L))
        g = bcm.Grid(spec, bcm.PREC_F64)
        g.field(bcm.RHS).copy_(torch.sin(torch.arange(spec.n_cells, device="cuda",
                                                      dtype=torch.float64) / 7))
        g.profile_read()
        g.profile(True)
        st = g.solve_pressure_iters(5)
        prof, launches = g.profile_read()
        g.profile(False)
        assert st[0]["pcg_form"] == form
        assert prof["pcg"][1] == (1 if form == 3 else 0)
        assert (prof["cg_a"][1] > 0) == (form == 0)
        assert launches == sum(n for _, n in prof.values())
