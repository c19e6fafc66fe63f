"""The single-kernel solve's waits between its blocks are bounded: one that
runs out ends the kernel with an error status, whichever block met it, and the
context stays usable."""
import numpy as np
import pytest

from paper_1907_04732_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_wait_that_runs_out_is_reported(lbe, monkeypatch, precision):
    """A limit of no polls: the first block to arrive at a barrier gives up.
    Every time, also where block 0 had left the barrier before that."""
    w = wl.plate_capacitor(24, 20, 30, debye=4.0, psi=(-0.05, 0.15))
    prec = lbe.LBE_FP64 if precision == "fp64" else lbe.LBE_FP32
    monkeypatch.setenv("LBE_SOLVE_SPINS", "0")
    g = lbe.Lattice.from_workload(w, precision=prec, tol=1e-12)
    for _ in range(20):
        with pytest.raises(lbe.LBEError) as e:
            g.init()
        assert e.value.code == lbe.LBE_ERR_CUDA, e.value
        assert "wait" in str(e.value)
    g.close()
    monkeypatch.delenv("LBE_SOLVE_SPINS")
    g = lbe.Lattice.from_workload(w, precision=prec, tol=1e-12)
    g.init()
    g.step(1)
    assert np.isfinite(g.phi()).all()
    g.close()
