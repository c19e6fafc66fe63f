"""The Poisson solve's kernels at the sizes where they can go wrong: chains,
single planes, two-node axes, ragged planes around the 256-column blocks, node
counts that are no multiple of the vector width, electrodes that touch the
column chunks' ends, lattices on both sides of the single-kernel solve's size.

Tolerances.  Every path stops at max |res|/diag <= tol.  Across a gap of L
nodes the inverse of the Jacobi-scaled operator is bounded by L^2/2 in the
maximum norm (the parabola that solves -u'' = 4 between grounded plates; a
chain has half of that, solid inclusions only lower it), so a potential is
within tol L^2/2 of the solution and two of them within tol L^2; a factor two
is left for the few steps' feedback through the ions."""
import numpy as np
import pytest

from paper_1907_04732_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 24), (1, 1, 203), (2, 1, 40), (1, 7, 33), (2, 2, 18), (3, 5, 61), (17, 15, 12), (31, 9, 10),
          (16, 16, 32), (257, 3, 8), (33, 8, 21)]


def lattice(nx, ny, nz, **kw):
    """Plates; where the cross-section has room, a bump on one plate that
    ends in the middle of a column chunk and of an aggregate."""
    w = wl.plate_capacitor(nx, ny, nz, debye=4.0, psi=(-0.05, 0.15), D=(0.05, 0.08))
    ids = w.ids.copy()
    if nx >= 8:
        ids[: nz // 2 + 1, : max(1, ny // 3), 1:4] = 1
    return w.with_(ids=ids, **kw)


@pytest.mark.parametrize("shape", SHAPES)
def test_fp64_solve_against_oracle(lbe, shape):
    from oracle import Oracle
    w = lattice(*shape)
    o = Oracle(w.shape, w.periodic, tau=w.tau, bjerrum=w.bjerrum, z=w.z, D=w.D, rho_bulk=w.rho_bulk,
               e_app=w.e_app, flow=w.flow, tol=1e-14)
    o.set_geometry(w.ids, w.n_elec)
    o.set_voltage(w.psi)
    o.init()
    g = lbe.Lattice.from_workload(w, tol=1e-14, flow=w.flow)
    g.init()
    o.step(3)
    g.step(3)
    bound = 2 * 1e-14 * shape[2] ** 2
    assert np.abs(g.phi() - o.phi()).max() <= bound
    # electrode charge: 18 links a node of eps * 2/3 times two potentials
    assert np.abs(g.charge() - o.charge()).max() <= 24 * bound * max((w.ids == e).sum() for e in (1, 2))


@pytest.mark.parametrize("salt", ["1:1", "three species"])
@pytest.mark.parametrize("shape", SHAPES + [(128, 96, 127), (128, 128, 97)])
def test_fp32_solve_paths_agree(lbe, monkeypatch, shape, salt):
    """The single-kernel solve (the first lattice, up to 3 2^19 nodes; the last
    shape is beyond) and the kernels launched one by one from the host."""
    w = lattice(*shape)
    if salt != "1:1":
        w = w.with_(z=(1.0, 2.0, -1.0), D=(0.05, 0.03, 0.06))
    phi, q = [], []
    for graph in ("1", "0"):
        monkeypatch.setenv("LBE_POISSON_GRAPH", graph)
        p = lbe.params_for(w, precision=lbe.LBE_FP32, tol=1e-12)
        if salt != "1:1":
            for k, r in enumerate((0.002, 0.001, 0.004)):
                p.rho_bulk[k] = r
        g = lbe.Lattice(p)
        g.set_geometry(w.ids, w.n_elec)
        g.set_voltage(w.psi)
        g.init()
        g.step(2)
        phi.append(g.phi())
        q.append(g.charge())
    bound = 2 * 1e-12 * shape[2] ** 2
    assert np.abs(phi[0] - phi[1]).max() <= bound
    assert np.abs(q[0] - q[1]).max() <= 24 * bound * max((w.ids == e).sum() for e in (1, 2))


def test_single_kernel_solve_reports_failures(lbe):
    """An iteration cap that cannot suffice, as the other paths report it."""
    w = lattice(16, 16, 32)
    p = lbe.params_for(w, precision=lbe.LBE_FP32, tol=1e-12, maxit=1)
    g = lbe.Lattice(p)
    g.set_geometry(w.ids, w.n_elec)
    g.set_voltage(w.psi)
    with pytest.raises(lbe.LBEError) as e:
        g.init()
    assert e.value.code == lbe.LBE_ERR_NOCONVERGE


@pytest.mark.parametrize("nz", [64, 203])
def test_chain_takes_few_iterations(lbe, nz):
    """A 1 x 1 column is a chain, whose Jacobi weight differs (weight 1 does not
    damp its alternating mode: 110 iterations a solve)."""
    for prec in (lbe.LBE_FP32, lbe.LBE_FP64):
        w = lattice(1, 1, nz)
        g = lbe.Lattice.from_workload(w, precision=prec, tol=1e-12)
        g.init()
        g.step(2)
        assert g.stats().poisson_max_iters <= 30


def test_single_kernel_solves_of_two_threads(lbe):
    """Two lattices, each on its own stream and host thread, both solving with
    as many blocks as the GPU holds: each grid is resident as a whole before
    it starts, and the results are bitwise those of one after the other."""
    import threading
    ws = [lattice(64, 64, 64), lattice(96, 48, 60)]

    def run(w, out, k):
        g = lbe.Lattice.from_workload(w, precision=lbe.LBE_FP32, tol=1e-12)
        g.init()
        g.step(40)
        out[k] = (g.phi(), g.charge())

    alone, together = [None, None], [None, None]
    for k, w in enumerate(ws):
        run(w, alone, k)
    th = [threading.Thread(target=run, args=(w, together, k)) for k, w in enumerate(ws)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    for a, b in zip(alone, together):
        np.testing.assert_array_equal(a[0], b[0])
        np.testing.assert_array_equal(a[1], b[1])
