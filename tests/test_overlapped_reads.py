"""Kernels that overlap the launch of their predecessor (programmatic dependent
launch) are resident while it still writes, so what such kernels write must not
be read through the read-only path: no __restrict__ on it, no __ldg, and no
__ldcg, which the wait does not order.  Checked on the sources, for every
kernel that calls pdl_wait() and the device functions it calls."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1206_6409_gb300", "csrc")

# what no overlapped kernel writes: X and its copies in the plans, y, the fold
# of each row, tables, the columns' curvature, partitions, colours, and the
# slots' parameters (copied between steps)
CONSTANT = {
    "col_ptr", "row_idx", "val", "row", "y", "fold", "tab", "bjs", "ib", "ibs", "bj32", "ib32", "part_lo", "color_ptr",
    "cols_by_color", "s_row", "s_val", "pmask", "pair_col", "tile_pair", "lrow", "lval", "lmask", "tile_lc",
    "light_cols", "light_row", "tstart", "tile_cc", "nzcols", "bnd", "smask", "sset", "group", "scale",
}
# base expressions of __ldg: the above, and pointers formed from them
LDG = CONSTANT | {"bjv", "ibv"}


def _matching(text, at, opening, closing):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == opening) - (text[i] == closing)
        if depth == 0:
            return i
    raise AssertionError("unbalanced source")


def _functions():
    """name -> (parameters, body, is a kernel) of the device code"""
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(CSRC, f)) as fh:
            text = re.sub(r"//[^\n]*", "", fh.read())
        for m in re.finditer(r"__(global|device)__", text):
            at, name = m.end(), None
            while True:
                head = re.compile(r"[;{(]").search(text, at)
                if head is None or head.group() != "(":
                    break
                word = re.search(r"(\w+)\s*$", text[at:head.start()])
                close = _matching(text, head.start(), "(", ")")
                if word and word.group(1) != "__launch_bounds__":
                    name = word.group(1)
                    break
                at = close + 1
            if not name:
                continue
            after = re.compile(r"\s*(const)?\s*\{").match(text, close + 1)
            if not after:
                continue  # a declaration
            body = text[after.end() - 1:_matching(text, after.end() - 1, "{", "}") + 1]
            old = out.get(name)
            params = text[head.start() + 1:close]
            if old:  # overloads and specialisations are checked together
                params, body = old[0] + "," + params, old[1] + body
            out[name] = (params, body, m.group(1) == "global" or bool(old and old[2]))
    return out


FUNCTIONS = _functions()
# loads of constant data by their parameter's own name (the callers' arguments are checked as theirs)
LOADERS = {"load_idx", "load_val", "load_vals", "load_rows8", "load", "load_lane", "lane_mask", "logistic_poly"}


def _reaches(name, seen):
    if name in seen or name not in FUNCTIONS:
        return
    seen.add(name)
    for callee in set(re.findall(r"\b(\w+)\s*(?:<[^;(){}]*>)?\s*\(", FUNCTIONS[name][1])):
        _reaches(callee, seen)


def _overlapped():
    found = []
    for name, (_, _, kernel) in FUNCTIONS.items():
        if kernel:
            seen = set()
            _reaches(name, seen)
            if "pdl_wait" in seen:
                found.append((name, sorted(seen)))
    return found


OVERLAPPED = _overlapped()


def test_the_overlapped_kernels_are_found():
    names = {n for n, _ in OVERLAPPED}
    assert {"k_accept_partitions", "k_propose_slabs", "k_propose_fused", "k_propose_light_runs", "k_update_flat",
            "k_refresh_flat", "k_update_refresh", "k_shotgun_step", "k_coloring_iter", "k_b_prep", "k_b_spmm",
            "k_b_spmm_runs8", "k_b_accept", "k_b_merge", "k_b_update", "k_b_update_grouped", "k_b_refresh",
            "k_b_refresh_all"} <= names


@pytest.mark.parametrize("kernel", [n for n, _ in OVERLAPPED])
def test_overlapped_kernels_read_changing_memory_coherently(kernel):
    for name in dict(OVERLAPPED)[kernel]:
        params, body, _ = FUNCTIONS[name]
        if name not in LOADERS:
            restrict = set(re.findall(r"__restrict__\s+(\w+)", params + ";" + body))
            assert restrict <= CONSTANT, (kernel, name, restrict - CONSTANT)
            ldg = set(re.findall(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?(\w+)", body))
            assert ldg <= LDG, (kernel, name, ldg - LDG)
        assert "__ldcg" not in body, (kernel, name)


def test_a_problems_launches_follow_its_overlap():
    # large problems of a serving slot launch plainly: every overlapped launch
    # for a problem takes the stream together with the problem's choice
    for f in ("kernels_propose.cu", "kernels_update.cu", "propose_plan.cu"):
        with open(os.path.join(CSRC, f)) as fh:
            text = fh.read()
        calls = [text[m.start():_matching(text, m.end() - 1, "(", ")")]
                 for m in re.finditer(r"\blaunch_(?:cluster_)?overlapped\(", text)]
        assert calls and all("launch_on(p)" in c and "p->stream" not in c for c in calls), f
