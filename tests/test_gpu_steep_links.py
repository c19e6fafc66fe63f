"""FP64 link fluxes (Eq. LF2) across potential steps from a fraction of kT/e to
twenty, near equilibrium, against 50-digit arithmetic.

Fluid nodes of even and odd z hold opposite potentials, so every link between
planes has the same exactly representable step, and the amounts are the Boltzmann
factors of that potential times 1 + 1e-3 xi.  One step without flow returns
n* = n + (d/2) sum_i J_i/|c_i|,  J = n' (1 + e^dmu) - n (1 + e^-dmu), with d = 1.

Tolerance: a flux formed from expm1 (1 ulp), rounded products and a few additions
is within 8 u of |n'| (2 + |expm1(dmu)|) + |n| (2 + |expm1(-dmu)|), u = 2^-53;
18 of them are added (17 more roundings of the partial sums, bounded by the
same terms: 8 + 17 u), and the last addition and d/2 round n* (4 u)."""
from decimal import Decimal, getcontext
import itertools
import math

import numpy as np
import pytest

from paper_1907_04732_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

LINKS = [c for c in itertools.product((-1, 0, 1), repeat=3) if 0 < sum(map(abs, c)) < 3]


@pytest.mark.parametrize("z", [(1.0, -1.0), (4.0, -2.0)])
@pytest.mark.parametrize("dmu", [0.125, 0.25, 1.0, 5.0, 8.0, 20.0])
def test_steep_links(lbe, z, dmu):
    getcontext().prec = 50
    a0 = 1.0 + 2.0 * math.sqrt(2.0)
    w = wl.plate_capacitor(4, 4, 10, debye=4.0, psi=(0.0, 0.0))
    p = lbe.params_for(w, precision=lbe.LBE_FP64, tol=1e-9)
    step = dmu / max(abs(v) for v in z)  # a power of two times 1 or 5: exact
    top = math.exp(dmu / 2)
    p.flow = 0
    p.bjerrum = 1e-3 / top  # the solve that follows meets charges of order 1e-3
    for k in range(2):
        p.z[k] = z[k]
        p.D[k] = a0
        p.rho_bulk[k] = 1.0
    g = lbe.Lattice(p)
    g.set_geometry(w.ids, w.n_elec)
    g.set_voltage(w.psi)
    g.init()
    ids = w.ids
    nz, ny, nx = ids.shape
    rng = np.random.default_rng(int(dmu * 1000) + int(z[0]))
    phi = np.zeros(ids.shape)
    phi[::2] = 0.5 * step
    phi[1::2] = -0.5 * step
    phi[ids > 0] = 0.0
    n = np.zeros((2,) + ids.shape)
    for k in range(2):
        n[k] = np.exp(-z[k] * phi) * (1.0 + 1e-3 * rng.standard_normal(ids.shape))
        n[k][ids > 0] = 0.0
    g.set_state(n=n, phi=phi)
    g.step(1)
    got = g.n()
    g.close()
    em1 = {s: Decimal(s).exp() - 1 for s in {float(z[k] * s) for k in range(2) for s in (0.0, step, -step)}}
    u = Decimal(2) ** -53
    for k in range(2):
        d = Decimal(a0 / a0)
        for Z, Y, X in np.argwhere(ids == 0):
            n0 = Decimal(float(n[k, Z, Y, X]))
            total, size = Decimal(0), Decimal(0)
            for cx, cy, cz in LINKS:
                q = (Z + cz) % nz, (Y + cy) % ny, (X + cx) % nx
                if ids[q]:
                    continue
                x = float(z[k] * (phi[q] - phi[Z, Y, X]))
                n1 = Decimal(float(n[k][q]))
                inv = Decimal(1) / Decimal(abs(cx) + abs(cy) + abs(cz)).sqrt()
                total += inv * (n1 * (2 + em1[x]) - n0 * (2 + em1[-x]))
                size += inv * (n1 * (2 + abs(em1[x])) + n0 * (2 + abs(em1[-x])))
            want = n0 + d / 2 * total
            err = abs(Decimal(float(got[k, Z, Y, X])) - want)
            assert err <= u * (25 * d / 2 * size + 4 * abs(want)), (z[k], int(Z), float(err / (u * size)))
