"""Workspace of grids with an FP64 state and the FP32 pressure solve on the CPU: the six
vectors that the Crank-Nicolson iteration shares with the solver hold FP64 values."""
import ctypes as C

import numpy as np
import pytest

from paper_1808_04099_gb300 import bcm
from paper_1808_04099_gb300 import workloads as W


@pytest.mark.parametrize("B", [4, 8, 16])
def test_crank_nicolson_vectors_fit(B):
    sp = W.sphere_channel(4, 2, 2, B)
    arrs = [np.ascontiguousarray(a, t) for a, t in (
        (sp.sim_cube_offset, np.int32), (sp.cube_ijk, np.int32), (sp.cube_level, np.int8),
        (sp.sim_extent, np.int32), (sp.sim_origin, np.float64), (sp.sim_h0, np.float64),
        (sp.sim_bc, np.int32), (sp.sim_bc_vel, np.float64), (sp.sim_nu, np.float64),
        (sp.sim_dt, np.float64), (sp.sim_uconv, np.float64))]
    d = bcm.GridDesc()
    d.n_sims, d.n_cubes, d.cells_per_edge, d.max_level = sp.n_sims, sp.n_cubes, sp.B, 0
    (d.sim_cube_offset, d.cube_ijk, d.cube_level, d.sim_extent, d.sim_origin, d.sim_h0, d.sim_bc,
     d.sim_bc_vel, d.sim_nu, d.sim_dt, d.sim_uconv) = [a.ctypes.data for a in arrs]
    size = {}
    for prec in (bcm.PREC_F64, bcm.PREC_F32_REFINE, bcm.PREC_F64_REFINE):
        d.precision = prec
        size[prec] = bcm.lib().bcm_workspace_bytes(C.byref(d))
    n = sp.n_cells
    # against the FP32 state: ten state fields and six shared vectors of 4 bytes more (the
    # face velocities a little more still)
    assert size[bcm.PREC_F64_REFINE] - size[bcm.PREC_F32_REFINE] >= 16 * 4 * n
