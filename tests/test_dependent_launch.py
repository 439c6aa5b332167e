"""Kernels that may start before their predecessor in the stream has ended (programmatic
dependent launch) wait before they touch what an earlier launch writes: only the wait makes
those writes visible.  Read from the CUDA sources, since a missing wait is a race that a run
need not show."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_00682_gb300", "csrc")


def _function(source, name):
    """Body of the function `name`, without comments."""
    text = open(os.path.join(CSRC, source)).read()
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    m = re.search(r"\bvoid\s+(?:__launch_bounds__\s*\([^\n]*?\)\s+)?%s\(" % name, text)
    start = text.index("{", m.end())
    return text[start:_close(text, start)]


def _close(text, at):
    """Index behind the brace that closes the one at text[at]."""
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return i + 1
    raise ValueError("unbalanced braces")


def _without_lambdas(body):
    while True:
        m = re.search(r"auto \w+ = \[&\]\([^)]*\) \{", body)
        if not m:
            return body
        body = body[:m.start()] + body[_close(body, m.end() - 1):]


def test_local_solve_loads_its_state_after_the_wait():
    body = _without_lambdas(_function("fused_tile.cuh", "tile_solve"))
    assert re.findall(r"^.*pdl_wait\(\).*$", body, flags=re.M) == ["    pdl_wait();"], "one wait, on every path"
    before, after = body.split("pdl_wait();")
    assert "data(" in before and "state(" not in before and "step(" not in before
    # no element of the state, the multipliers or the strips (only addresses are formed)
    assert not re.search(r"\bA\.(u0?|P1|P2|P10|P20|lam\w*|x_in\.\w+)\s*\[", before)
    assert not re.search(r"\bg[u12]\s*\[", before)
    assert "state(" in after


@pytest.mark.parametrize("source,kernel", [
    ("kernels_interface.cu", "k_interface_v4"), ("kernels_interface.cu", "k_interface_v1"),
    ("kernels_interface.cu", "k_interface_batch"), ("kernels_adjoint.cu", "k_adj_interface")])
def test_updates_wait_first(source, kernel):
    assert _function(source, kernel)[1:].lstrip().startswith("pdl_wait();")


def test_full_dimension_blocks_wait_before_every_array():
    body = _function("kernels_full.cu", "k_full")
    assert body.count("pdl_wait();") == 1
    assert not re.search(r"\bA\.(f|mask|coef|in|out)\b", body.split("pdl_wait();")[0])
