"""Ordering between the grids of a step, read from the source.  A grid that is launched under the tail of the one before it
is promised to see what earlier grids wrote only behind its own ``griddepcontrol.wait``: that the grid before it has
waited promises nothing to this one.  So no kernel may touch memory that a grid or the caller writes ahead of its wait;
the plan's tables, which are uploaded before any launch that reads them, are the exception."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_17686_b200", "csrc")
PLAN_TABLES = {"desc", "work", "pieces", "cta_first"}
# Launched without a wait only when the caller states that its inputs are complete (FICOCO_BACK_TO_BACK).
OPT_IN = {"k_filter_fused": "if (dep_wait_first) grid_dep_wait();"}


def kernels():
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", text):
            end = text.index(")", m.end())                    # (no parameter list of these holds a parenthesis)
            depth, at = 1, text.index("{", end) + 1
            start = at
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            yield m.group(1), text[m.end():end], text[start:at - 1]


KERNELS = list(kernels())
DEPENDENT = [k for k in KERNELS if "grid_dep_wait" in k[2]]


def test_the_dependent_kernels_are_found():
    names = {k[0] for k in DEPENDENT}
    assert {"k_filter_fused", "k_colsum_wide", "k_head_mean", "k_score_wide", "k_select", "k_correlate_umma",
            "k_correlate_umma_f32", "k_correlate_rel", "k_merge_rows", "k_equivalent_token"} <= names


@pytest.mark.parametrize("name,params,body", DEPENDENT, ids=[k[0] for k in DEPENDENT])
def test_nothing_is_touched_ahead_of_the_wait(name, params, body):
    wait = OPT_IN.get(name, "grid_dep_wait();")
    ahead = body[:body.index(wait)]
    if name not in OPT_IN:
        assert not re.search(r"(if|while)\s*\([^;{}]*\)\s*$|(else|\?)\s*$", ahead), "the wait hangs on a condition"
    pointers = {re.search(r"(\w+)\s*$", p).group(1) for p in params.split(",") if "*" in p}
    touched = {p for p in pointers - PLAN_TABLES if re.search(rf"\b{p}\b", ahead)}
    assert not touched, f"{name} names {sorted(touched)} ahead of its wait"


def without_lambdas(body):
    while m := re.search(r"\[&\]\s*(\([^()]*\))?\s*\{", body):
        depth, at = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(body[at], 0)
            at += 1
        body = body[:m.start()] + body[at:]
    return body


@pytest.mark.parametrize("name,params,body", DEPENDENT, ids=[k[0] for k in DEPENDENT])
def test_no_way_out_ahead_of_the_wait(name, params, body):
    """A grid that gave up has waited all the same: the one behind it waits for it alone."""
    ahead = without_lambdas(body[:body.rindex("grid_dep_wait();")])
    if name not in OPT_IN:
        ahead = ahead[:ahead.index("grid_dep_wait();")] if "grid_dep_wait();" in ahead else ahead
    assert not re.search(r"\breturn\b", ahead), f"{name} can end without having waited"
