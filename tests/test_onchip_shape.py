"""The on-chip PCG's launch rule on the CPU: with several sims its sums run over units of 64
cells of a block, so no unit may reach into another item (a z-slab of one cube, hence of
one sim), whatever the number of cubes, sims and SMs."""
import pytest

from paper_1808_04099_gb300 import bcm


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("B", [4, 8, 16])
def test_units_stay_inside_items(B, fp64):
    fits = 0
    for sms in (152, 132, 40):
        for n in [*range(2, 700), 1000, 1291, 1292, 2000, 3600]:
            for sims in (2, n):
                s = bcm.onchip_shape(B, n, sims, 0, fp64, sms)
                if s is None:
                    continue
                fits += 1
                assert s["planes"] * B * B >= 64, (n, sims, sms, s)
                # every cell of the fullest block lies in a thread's quads
                assert s["items"] * s["planes"] * B * B <= 4 * s["threads"] * s["quads"]
                assert s["items"] * s["blocks"] * s["planes"] >= n * B
    assert fits > 500
    # one sim: half cubes of 4^3 are taken where they spread the cells better
    if B == 4 and fp64:
        assert bcm.onchip_shape(4, 230, 1, 0, True)["planes"] == 2
