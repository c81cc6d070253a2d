"""Launches that may begin before the one ahead of them is complete
(programmatic dependent launch): what a kernel reads was written by that
launch or an earlier one, and is guaranteed to be visible only after the
kernel's own wait.  Checked on the source of the surrogate's kernels: no load
helper stands before the wait; and of the step kernels: the step counter,
which they read before it, comes from L2."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1401_6047_gb300", "csrc",
                   "bte_sur_kernels.cu")
LOADS = re.compile(r"\b(load_xh|load_rows|load_stage_mn|ld8|over_samples|reduced|adam_one|weight_tile)\s*\(|\bP\[|"
                   r"\ba\.(params|partial|Yh|Zin|g|p|x|y)\[")
TEXT = re.sub(r"/\*.*?\*/", "", open(SRC).read(), flags=re.S)


def _body(name):
    at = re.search(rf"\bvoid\b[^;{{}}]*\b{name}\s*\([^;{{}}]*\)\s*{{", TEXT).end()
    depth, i = 1, at
    while depth:
        depth += {"{": 1, "}": -1}.get(TEXT[i], 0)
        i += 1
    return TEXT[at:i]


def _launched():
    return sorted(set(re.findall(r"launch_pdl\(\s*(\w+)\s*[<,]", TEXT)))


@pytest.mark.parametrize("kernel", _launched())
def test_no_load_before_the_wait(kernel):
    body = _body(kernel)
    parts = [body]
    if "pdl_wait" not in body:  # a kernel that only picks between device functions
        parts = [_body(f) for f in ("weight_gradients", "reduce_partial") if f + "(" in body]
        assert len(parts) == 2
    for part in parts:
        before, wait, _ = part.partition("pdl_wait();")
        assert wait, f"{kernel} never waits"
        assert not LOADS.search(before), LOADS.search(before).group(0)


def test_every_dependent_launch_is_covered():
    assert {"gemm_tc_kernel", "grad_kernel", "l1_kernel", "head_kernel", "adam_kernel"} == set(_launched())


@pytest.mark.parametrize("name", ["bte_step.cu", "bte_pair.cu"])
def test_step_counter_read_before_the_wait_comes_from_l2(name):
    text = re.sub(r"/\*.*?\*/", "", open(os.path.join(os.path.dirname(SRC), name)).read(), flags=re.S)
    assert not re.search(r"\*\s*\(?\s*(BATCH \? )?(A|Bt)\.base", text)
    assert re.search(r"__ldcg\((A\.)?base\)", text)
