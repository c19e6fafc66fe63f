"""Density, velocity and populations of the FP32 form's state (summed in
floats with error terms, widened to FP64) against their definitions, on both
step kinds of the in-place streaming.

Tolerance of the density: each of the 19 populations handed out is rounded
once, and numpy's sum of them 18 times more, to 2^-53 of values that add up
to one: 37 * 2^-53 = 4.1e-15."""
import numpy as np
import pytest

from paper_1907_04732_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [0, 1, 2, 7])
@pytest.mark.parametrize("shape", [(5, 3, 12), (17, 15, 14)])
def test_density_is_the_sum_of_the_populations(lbe, shape, steps):
    ids = wl.random_blobs(*shape, 2, 0.2, seed=3)
    w = wl.Workload("blob", ids, 2, (1, 1, 1), (0.0, 0.25), 1.1, 2.5, e_app=(2e-3, -1e-3, 5e-4))
    g = lbe.Lattice.from_workload(w, precision=lbe.LBE_FP32, tol=1e-12)
    g.init()
    g.step(steps)
    f, rho, u = g.populations(), g.rho(), g.u()
    fluid = ids == 0
    assert np.abs(rho - f.sum(axis=0))[fluid].max() <= 37 * 2.0 ** -53
    assert not rho[~fluid].any() and not f[:, ~fluid].any() and not u[:, ~fluid].any()


def test_rest_state_is_exact(lbe):
    """Zero deviations widen to zero: the weights, density one, no velocity."""
    w = wl.plate_capacitor(4, 3, 12, psi=(0.0, 0.0))
    g = lbe.Lattice.from_workload(w, precision=lbe.LBE_FP32, tol=1e-12)
    g.init()
    fluid = w.ids == 0
    wt = np.array([1 / 3 if not any(c) else (1 / 18 if sum(map(abs, c)) == 1 else 1 / 36) for c in lbe.VELOCITIES])
    np.testing.assert_array_equal(g.populations()[:, fluid], np.repeat(wt[:, None], fluid.sum(), axis=1))
    np.testing.assert_array_equal(g.rho()[fluid], 1.0)
    np.testing.assert_array_equal(g.u(), 0.0)
