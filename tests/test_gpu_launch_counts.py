"""kernel_launches of a profile counts the kernels of the path that each solve
took: one for a single-kernel solve; for a solve as a graph (here a lattice
small enough for the single kernel, with its coarsest level left to Jacobi
sweeps) the reset, two per residual test and, per iteration, the V-cycle's
kernels (three at least: restriction, coarsest solve, post-smoothing), stencil
and update."""
import pytest

from paper_1907_04732_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("graph", [False, True])
def test_launches_follow_the_path(lbe, monkeypatch, precision, graph):
    if graph:
        monkeypatch.setenv("LBE_MG_DIRECT", "0")
    w = wl.plate_capacitor(16, 12, 20, debye=4.0, flow=False)
    prec = lbe.LBE_FP64 if precision == "fp64" else lbe.LBE_FP32
    g = lbe.Lattice.from_workload(w, precision=prec, tol=1e-11)
    g.init()
    steps = 3
    lbe.lbe_profile_begin(g.h)
    g.step(steps)
    p = lbe.lbe_profile_end(g.h)
    g.close()
    assert p.poisson_iters >= 1
    if graph:  # sweep, warm start and the solve's kernels
        assert p.kernel_launches >= steps * (1 + 1 + 1 + 2) + 5 * p.poisson_iters
    else:
        assert p.kernel_launches == 3 * steps
