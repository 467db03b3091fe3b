"""Quantization at half-integers (where the product with 1 / step decides nothing and the
quotient is formed), at the largest codes and at steps near the ends of the range: cubes of
one value keep it as their one coefficient, so the streams must equal the oracle's word
for word."""
import numpy as np
import pytest

import oracle as O
from paper_1808_04099_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


@pytest.mark.parametrize("B", [4, 8, 16])
@pytest.mark.parametrize("step", [1e-4, 1.0 / 3.0, 7.3, 2.0 ** -40, 1e-285, 1e285])
def test_ties_and_ends(B, step):
    spec = W.cavity(4, B)  # 64 cubes
    q = np.array([0, 1, 2, 3, 7, 100, 12345, 2 ** 20, 2 ** 28, 2 ** 29 - 1, 2 ** 29, 2 ** 29 + 7,
                  2 ** 30 - 2, -1, -2, -2 ** 29], np.float64)
    v = np.concatenate([(q + 0.5) * step, np.nextafter((q + 0.5) * step, np.inf),
                        np.nextafter((q + 0.5) * step, -np.inf), q * step])
    f = np.repeat(v, B ** 3)
    # a ramp in some cubes: details of every level at multiples of the step
    for c in range(0, 64, 5):
        f[c * B ** 3:(c + 1) * B ** 3] = (np.arange(B ** 3) % 17) * 0.5 * step
    g = bcm.Grid(spec, bcm.PREC_F64)
    g.field(bcm.U).copy_(torch.from_numpy(f).cuda())
    s = g.compress_field(bcm.U, step).cpu().numpy().view(np.uint32)
    ref = O.wavelet_compress(f, B, step)
    assert np.array_equal(s, ref)
    g.decompress_field(bcm.V, torch.from_numpy(s.view(np.int32)))
    assert np.array_equal(g.numpy(bcm.V), O.wavelet_decompress(ref))
