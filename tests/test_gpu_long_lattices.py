"""Lattices so long that a coarse level has more planes than a grid's z axis
holds (65535), on the path that launches the V-cycle's kernels one by one."""
import numpy as np
import pytest

from paper_1907_04732_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_restriction_beyond_the_grid_limit(lbe, precision):
    """4 x 2 x 264000 (level 2: 66000 planes) between plates, a pair of solid
    planes every 40 so that the potential of each cell is a short solve.
    Cells are copies of each other: their charges and potentials agree, also
    those beyond plane 65535 of level 2, within the solve's tolerance times
    the bound L^2/2 of the inverse across a gap of L nodes."""
    nx, ny, nz, cell = 4, 2, 264000, 40
    ids = np.zeros((nz, ny, nx), np.uint8)
    ids[::cell] = 1
    ids[cell - 1::cell] = 2
    w = wl.Workload("cells", ids, 2, (1, 1, 0), (-0.05, 0.15), 1.44, 4.0, flow=False)
    tol = 1e-11
    prec = lbe.LBE_FP64 if precision == "fp64" else lbe.LBE_FP32
    g = lbe.Lattice.from_workload(w, precision=prec, tol=tol)
    g.init()
    g.step(1)
    phi = g.phi().reshape(nz // cell, cell, ny, nx)
    g.close()
    mid = phi[:, cell // 2 - 1:cell // 2 + 1].mean()
    assert abs(mid - 0.05) < 0.01  # the middle of the two potentials
    assert np.abs(phi - phi[:1]).max() <= tol * cell ** 2
