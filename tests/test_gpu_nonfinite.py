"""A right-hand side whose <r, z> is finite and whose first <p, Kp> overflows: the FP64 solve
ends with BCM_E_NONFINITE at once and leaves the pressure as it was, on chip as in two
launches, with one sim and with several."""
import numpy as np
import pytest

from paper_1808_04099_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1808_04099_gb300 import bcm  # noqa: E402


def channel(nx, ny, nz, B):
    L = tuple(n * B / 16.0 for n in (nx, ny, nz))
    return W.sphere_channel(nx, ny, nz, B, L, L[1] / 8, tuple(e / 2 for e in L))


@pytest.mark.parametrize("form", [0, 3])
@pytest.mark.parametrize("sims", [1, 3])
def test_overflowing_direction(sims, form):
    spec = W.concat([channel(3, 2, 2, 8)] * sims) if sims > 1 else channel(3, 2, 2, 8)
    g = bcm.Grid(spec, bcm.PREC_F64)
    if form == 0:
        g.set_launch(1, 1, persistent=0)
    B, h = spec.B, float(spec.sim_h0[0])
    i = np.arange(B ** 3)
    sign = 1.0 - 2.0 * ((i % B + i // B % B + i // (B * B)) % 2)  # a checkerboard, cube by cube
    r1 = np.tile(sign, spec.n_cubes)
    # diag(K) / h: six faces, none for a closed domain face, two for an outflow face
    diag = np.full(spec.n_cells, 6.0)
    ends = np.array(spec.sim_extent[0])
    for c, ijk in enumerate(np.asarray(spec.cube_ijk)):
        cell = diag[c * B ** 3:(c + 1) * B ** 3]
        for f in range(6):
            x = ijk[f // 2] + (i // B ** (f // 2)) % B
            at = x == (ends[f // 2] - 1 if f % 2 else 0)
            cell[at] += 1.0 if spec.sim_bc[0][f] == W.OUTFLOW else -1.0
    z1 = r1 / (diag * h)
    n = spec.n_cells // sims
    rz = float(r1[:n] @ z1[:n])
    pq = float(z1[:n] @ g.apply_poisson(torch.from_numpy(z1)).cpu().numpy()[:n])
    assert pq > 1.5 * rz
    amp = np.sqrt(0.9 * np.finfo(float).max / rz)
    b = -(amp * r1) / h ** 3
    g.field(bcm.RHS).copy_(torch.from_numpy(b).cuda())
    p0 = torch.zeros(spec.n_cells, dtype=torch.float64, device="cuda")
    g.field(bcm.P).copy_(p0)
    with pytest.raises(bcm.BCMError) as e:
        g.solve_pressure(rtol=1e-12, max_iter=50)
    assert e.value.status == bcm.BCM_E_NONFINITE
    assert torch.equal(g.field(bcm.P), p0)
    # the grid works on
    g.field(bcm.RHS).copy_(torch.from_numpy(r1).cuda())
    st = g.solve_pressure(rtol=1e-10)
    assert all(s["converged"] == 1 and s["pcg_form"] == form for s in st)
