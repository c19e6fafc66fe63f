"""A hierarchy that cannot be built (out of memory) leaves freed arrays behind the
solve graphs of the geometry before it.  Read as text, since no test may exhaust
the memory of a GPU: the graphs are dropped and the handle refuses to step
before the old hierarchy is freed, and after the arguments have been checked."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1907_04732_gb300", "csrc")


@pytest.mark.parametrize("file,name,checked,drop,state", [
    ("lbe_api.cu", "lbe_set_geometry", "fluid node on a non-periodic face", "poisson_drop_graphs(h)",
     r"have_geometry = h->initialised = false"),
    ("batch.cu", "lbe_batch_init", "an instance has no geometry", "drop_graphs(b)", r"b->initialised = false"),
])
def test_graphs_go_before_the_hierarchy(file, name, checked, drop, state):
    with open(os.path.join(CSRC, file)) as f:
        text = f.read()
    body = text[re.search(r"^int %s\(" % name, text, re.M).start():]
    body = body[:body.index("\n}\n")]
    build = re.search(r"\bmg_setup\(", body).start()
    assert body.index(checked) < body.index(drop) < build
    assert body.index(checked) < re.search(state, body).start() < build
