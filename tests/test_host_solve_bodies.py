"""The bodies that the single-kernel Poisson solve runs as phases between grid
barriers, read as text: only arrays that no phase writes (the operators A, their
weights W, the link masks, the node codes) may be declared __restrict__ there.
A pointer so qualified may be loaded through the read-only cache, which a
barrier does not refresh, and would show values from before another block's
write."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1907_04732_gb300", "csrc")
CONSTANT = {"A", "AF", "W", "WC", "M", "Ainv", "mask", "code"}
BODIES = [("mg_device.cuh", f) for f in ("presmoothed_res_z", "post_value_w", "post_value_z")] + [
    ("fp32_device.cuh", f) for f in ("lap6_ff_", "lap6_fx_")] + [
    ("solve_device.cuh", f) for f in ("lap_at", "res_column", "cg_b_column")] + [
    ("vcycle.cuh", f) for f in ("restrict0_block", "restrict_block", "post0_column", "inverse_row", "dense_row")] + [
    ("march.cuh", f) for f in ("plane_sums", "begin", "step")] + [
    ("poisson.cu", f) for f in ("cg_a_nodes", "correct_fx_nodes", "correct_nodes", "grid_sums", "grid_max", "one_vcycle",
                                "one_solve")]


def definition(text, name):
    """A function's text, from its parameter list to the end of its body."""
    m = re.search(r"__forceinline__[^;{}()]*\b%s\(" % re.escape(name), text)
    assert m, name
    start, depth = text.index("{", m.end()), 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[m.start():i + 1]
    raise AssertionError(name)


@pytest.mark.parametrize("file,name", BODIES)
def test_no_restrict_on_what_a_phase_writes(file, name):
    with open(os.path.join(CSRC, file)) as f:
        body = definition(f.read(), name)
    assert set(re.findall(r"__restrict__\s+(\w+)", body)) <= CONSTANT
