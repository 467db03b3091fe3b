"""The multigrid's coarse kernel with clusters of 1 to 16 blocks, at the sizes where the rule
adds blocks and where it leaves a level to a launch of its own (4096 cells), against the
oracle's V-cycle to 1e-12 (sums of at most 8 terms a level over at most 12 levels in FP64:
rounding under 12 * 8 * 2^-53 times the cycle's condition, far below)."""
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


# 2^3 cells of 4^3 cubes, or 4^3 of 8^3 cubes: 128, 136, 256, 512, 1024, 4096 and 4160 cells
SIZES = [((4, 2, 2), 4), ((17, 1, 1), 4), ((4, 4, 2), 4), ((4, 4, 4), 4), ((8, 4, 4), 4),
         ((8, 8, 8), 4), ((13, 8, 5), 4), ((8, 8, 1), 8), ((13, 5, 1), 8)]


@pytest.mark.parametrize("size,B", SIZES)
def test_vcycle_matches_oracle(size, B):
    spec = channel(*size, B)
    g = bcm.Grid(spec, bcm.PREC_F64)
    r = np.random.default_rng(5).standard_normal(spec.n_cells)
    z = g.apply_preconditioner(r).cpu().numpy()
    assert rel_l2(z, MGO.MG(O.Oracle(spec)).apply(r)) <= 1e-12
