"""Periodic boxes without electrodes: the potential of a neutral charge
distribution is defined up to a constant, and every solve converges, in few
iterations, at sizes whose coarsest operator has one node, two, or hundreds,
with chains, single planes and odd sides, alone and in a batch.

The residual is evaluated here with numpy from the fields read back.  Bounds: the
library's own max |res|/diag <= tol, plus what the read-back rounds (the charge,
18 potentials of magnitude |phi| and their sum, in units of 2^-53)."""
import itertools

import numpy as np
import pytest

from paper_1907_04732_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(2, 1, 1), (3, 1, 1), (5, 4, 3), (16, 16, 16), (17, 16, 15), (32, 32, 1), (24, 24, 24), (1, 1, 300),
          (128, 128, 1), (64, 32, 16), (160, 128, 80)]
TOL = {"fp32": 1e-12, "fp64": 1e-13}
ITERATIONS = 60  # of one solve (Jacobi-preconditioned: 110 to 220 on the longer ones)


def box(shape):
    return wl.Workload("box", np.zeros(shape[::-1], np.uint8), 0, (1, 1, 1), (), 1.44, 4.0, flow=False)


def amounts(w, seed):
    """Neutral: noise, or one wave per axis, opposite for the two species."""
    rng = np.random.default_rng(seed)
    nz, ny, nx = w.ids.shape
    if seed == 0:
        d = rng.uniform(-1.0, 1.0, (nz, ny, nx))
    else:
        wave = lambda k: np.cos(2 * np.pi * np.arange(k) / k + rng.uniform(0, 6.28))
        d = wave(nz)[:, None, None] + wave(ny)[:, None] * wave(nx)
    d = 0.1 * w.rho_bulk[0] * (d - d.mean())
    return np.stack([w.rho_bulk[0] + d, w.rho_bulk[0] - d])


def check(w, n, phi, tol):
    assert np.isfinite(phi).all()
    lap = np.zeros_like(phi)
    diag = 0.0
    for c in itertools.product((-1, 0, 1), repeat=3):
        k = sum(map(abs, c))
        if k not in (1, 2):
            continue
        if all(a == 0 or s == 1 for a, s in zip(c, phi.shape)):
            continue  # a link of a node to itself
        wt = 1.0 / 3.0 if k == 1 else 1.0 / 6.0
        diag += wt
        lap += wt * (np.roll(phi, tuple(-a for a in c), (0, 1, 2)) - phi)
    res = 4 * np.pi * w.bjerrum * (n[0] - n[1]) + lap
    rounding = 2.0 ** -53 * (40 * np.abs(phi).max() + 4 * 4 * np.pi * w.bjerrum * np.abs(n).max())
    assert np.abs(res).max() / diag <= tol + rounding


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shape", SHAPES)
def test_closed_box(lbe, shape, precision):
    w = box(shape)
    prec = lbe.LBE_FP64 if precision == "fp64" else lbe.LBE_FP32
    for seed in range(2):
        g = lbe.Lattice.from_workload(w, precision=prec, tol=TOL[precision])
        g.init()
        g.set_state(n=amounts(w, seed))
        g.step(3)
        assert g.stats().poisson_max_iters <= ITERATIONS
        check(w, g.n(), g.phi(), TOL[precision])
        g.close()
