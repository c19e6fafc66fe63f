"""A periodic lattice of one fluid node has no Poisson equation: every link joins
the node to itself and the diagonal is zero.  It is refused, as a non-finite
residual, alone and in a batch; one solid node is a lattice like any other."""
import numpy as np
import pytest

from paper_1907_04732_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def node(solid):
    ids = np.full((1, 1, 1), 1 if solid else 0, np.uint8)
    return wl.Workload("node", ids, int(solid), (1, 1, 1), (0.1,) if solid else (), 1.44, 4.0)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_lone_fluid_node_is_refused(lbe, precision):
    prec = lbe.LBE_FP64 if precision == "fp64" else lbe.LBE_FP32
    g = lbe.Lattice.from_workload(node(False), precision=prec, tol=1e-12)
    with pytest.raises(lbe.LBEError) as e:
        g.init()
    assert e.value.code == lbe.LBE_ERR_NONFINITE
    g.close()
    g = lbe.Lattice.from_workload(node(True), precision=prec, tol=1e-12)
    g.init()
    g.step(1)
    assert g.phi().item() == pytest.approx(0.1, abs=1e-14)
    g.close()


def test_lone_fluid_node_in_a_batch_is_refused(lbe):
    b = lbe.Batch([node(False), wl.plate_capacitor(4, 4, 16, debye=4.0)], tol=1e-12)
    with pytest.raises(lbe.LBEError) as e:
        b.init()
    assert e.value.code == lbe.LBE_ERR_NONFINITE
    b.close()
