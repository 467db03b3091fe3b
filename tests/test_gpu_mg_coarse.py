"""The multigrid's coarse kernel at the edges of its rules: one block and several, against
the oracle's V-cycle to 1e-12; and batches whose aggregate levels have more than 1024 nodes
(the whole cluster works on them), whose 2^3 level has a launch of its own, or which have
more sims than a block has threads, against the V-cycles of their sims alone, which the
same sums give up to the order of additions (1e-13)."""
import numpy as np
import pytest

import oracle as O
from oracle import mg_oracle as MGO
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


SINGLE = {
    "one_cube": lambda: W.cavity(1, 4),
    "two_blocks": lambda: channel(9, 5, 4, 4),              # 180 cubes, tails in every level
    "two_level": lambda: W.two_level_channel(6, 4, 4, 4, (2, 1, 1), (4, 3, 3), 1 / 16., 0),
}
# (the sim, how many of it)
BATCHES = {
    "many_nodes": (lambda: channel(8, 8, 8, 4), 20),        # 10,240 cubes, 1280 nodes above
    "many_sims": (lambda: W.cavity(1, 4), 1100),            # 1100 nodes on the top level too
    "many_8": (lambda: channel(9, 4, 4, 8), 6),
    "two_level": (lambda: W.two_level_channel(8, 6, 6, 4, (2, 1, 1), (6, 5, 5), 1 / 16., 0), 9),
}


@pytest.mark.parametrize("name", SINGLE)
def test_vcycle_matches_oracle(name):
    spec = SINGLE[name]()
    g = bcm.Grid(spec, bcm.PREC_F64)
    r = np.random.default_rng(3).standard_normal(spec.n_cells)
    z = g.apply_preconditioner(r).cpu().numpy()
    assert rel_l2(z, MGO.MG(O.Oracle(spec)).apply(r)) <= 1e-12


@pytest.mark.parametrize("name", BATCHES)
def test_batch_equals_its_sims(name):
    make, n = BATCHES[name]
    one = make()
    g1 = bcm.Grid(one, bcm.PREC_F64)
    gn = bcm.Grid(W.concat([one] * n), bcm.PREC_F64)
    r = np.random.default_rng(4).standard_normal((n, one.n_cells))
    z = gn.apply_preconditioner(r.reshape(-1)).cpu().numpy().reshape(n, -1)
    for s in sorted({0, 1, n // 2, n - 1}):
        assert rel_l2(z[s], g1.apply_preconditioner(r[s]).cpu().numpy()) <= 1e-13, s
