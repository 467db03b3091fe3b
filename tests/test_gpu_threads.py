"""Two host threads with grids of different sizes that run the same kernel (the on-chip PCG
with different amounts of shared memory): no launch of one fails because of the other."""
import threading

import pytest

from paper_1808_04099_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


def test_two_sizes_of_one_kernel():
    def grid(n):
        L = tuple(q * 0.5 for q in n)
        g = bcm.Grid(W.sphere_channel(*n, 8, L, L[1] / 8, tuple(e / 2 for e in L)), bcm.PREC_F64)
        t = torch.arange(g.spec.n_cells, device="cuda", dtype=torch.float64)
        g.field(bcm.RHS).copy_(torch.sin(t / 7))
        return g

    grids = [grid((10, 10, 7)), grid((12, 10, 10))]
    errors = []

    def work(g):
        try:
            for _ in range(600):
                st = g.solve_pressure_iters(1)
                assert st[0]["pcg_form"] == 3
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(g,)) for g in grids]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
