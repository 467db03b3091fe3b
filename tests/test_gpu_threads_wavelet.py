"""Two host threads that decode wavelet streams with records of different sizes (the decoder
stages a record, over 48 KB of shared memory in both): no launch of one fails because of the
other, and each field is its own."""
import threading

import numpy as np
import pytest

from paper_1808_04099_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


def test_records_of_two_sizes():
    spec = W.cavity(2, 16)
    rng = np.random.default_rng(1)
    work = []
    for bits in (26.0, 26.5):  # of the codes: records of about 14.8 and 15.8 KB
        g = bcm.Grid(spec, bcm.PREC_F64)
        f = rng.uniform(-1.0, 1.0, spec.n_cells) * 2.0 ** bits
        g.field(bcm.U).copy_(torch.from_numpy(f).cuda())
        s = g.compress_field(bcm.U, 1.0)
        assert (s.numel() - 8 - spec.n_cubes) / spec.n_cubes * 4 > 14000
        g.decompress_field(bcm.V, s)
        work.append((g, s, g.field(bcm.V).clone()))
    errors = []

    def decode(g, s, want):
        try:
            for _ in range(600):
                g.decompress_field(bcm.V, s)
            torch.cuda.synchronize()
            assert torch.equal(g.field(bcm.V), want)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=decode, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
