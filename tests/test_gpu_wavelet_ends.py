"""Wavelet streams with steps at the ends of the range of doubles, where halves of subnormal
values round and sums of two equal values overflow: streams and decoded fields are the
oracle's bit for bit, and what the oracle refuses is refused."""
import numpy as np
import pytest

import oracle as O
from paper_1808_04099_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


def grid(B, f):
    g = bcm.Grid(W.cavity(2, B), bcm.PREC_F64)
    g.field(bcm.U).copy_(torch.from_numpy(f).cuda())
    return g


@pytest.mark.parametrize("B", [4, 8, 16])
@pytest.mark.parametrize("k", [1, 3, 1000])
def test_subnormal_values(B, k):
    rng = np.random.default_rng(B + k)
    f = rng.integers(-5000, 5000, 8 * B ** 3) * 5e-324
    step = k * 5e-324
    ref = O.wavelet_compress(f, B, step)
    g = grid(B, f)
    s = g.compress_field(bcm.U, step).cpu().numpy().view(np.uint32)
    assert np.array_equal(s, ref)
    g.decompress_field(bcm.V, torch.from_numpy(ref.view(np.int32)))
    assert np.array_equal(g.numpy(bcm.V), O.wavelet_decompress(ref))


@pytest.mark.parametrize("B", [4, 8, 16])
def test_overflowing_sum_is_refused(B):
    f = np.zeros(8 * B ** 3)
    f[B - 2] = 1e308  # the last even value of a line: its mirrored neighbour doubles it
    with pytest.raises(ValueError):
        O.wavelet_compress(f, B, 1e300)
    g = grid(B, f)
    with pytest.raises(bcm.BCMError) as e:
        g.compress_field(bcm.U, 1e300)
    assert e.value.status == bcm.BCM_E_BOUNDS
    f[B - 2] = 0.7e308  # and one that does not overflow is coded as the oracle codes it
    g = grid(B, f)
    s = g.compress_field(bcm.U, 1e300).cpu().numpy().view(np.uint32)
    ref = O.wavelet_compress(f, B, 1e300)
    assert np.array_equal(s, ref)
    g.decompress_field(bcm.V, torch.from_numpy(ref.view(np.int32)))
    assert np.array_equal(g.numpy(bcm.V), O.wavelet_decompress(ref))
