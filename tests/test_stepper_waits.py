"""The serving loop's stepper advances every running solve from one thread, so a
solve's step must not wait for its stream: checked on the sources, for
solve_advance and what it calls."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1206_6409_gb300", "csrc")

# waits that come with the first use of a variant or the growth of a buffer, not
# with a step: power iteration and colouring, scratch that grows, profiling's
# event pool
FIRST_USE = {"compute_pstar", "compute_block_pstar", "run_coloring", "ensure_slots", "ensure_part_bounds",
             "ensure_sort_tmp", "prof_begin"}


def _host_functions():
    out = {}
    for f in ("api.cu", "kernels_propose.cu", "kernels_update.cu", "kernels_setup.cu", "propose_plan.cu"):
        with open(os.path.join(CSRC, f)) as fh:
            text = re.sub(r"//[^\n]*", "", fh.read())
        for m in re.finditer(r"^(?:static )?(?:int|void) (\w+)\([^;{]*\)\s*\{\n.*?^\}", text, re.M | re.S):
            out[m.group(1)] = out.get(m.group(1), "") + m.group(0)
    return out


def test_a_solves_step_does_not_wait():
    functions = _host_functions()
    seen, todo = set(), ["solve_advance"]
    while todo:
        name = todo.pop()
        if name in seen or name in FIRST_USE or name not in functions:
            continue
        seen.add(name)
        body = functions[name]
        assert "Synchronize" not in body and not re.search(r"\bcudaMemcpy\(", body), name
        todo += re.findall(r"\b(\w+)\(", body.split("{", 1)[1])
    assert {"solve_evaluate", "enqueue_iteration", "launch_state_from_w", "build_csr", "launch_update_refresh"} <= seen
