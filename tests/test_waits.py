"""What a kernel reads before it waits for its predecessor.  A kernel launched
behind another one starts while that one drains; what earlier kernels of the
cycle wrote is only guaranteed to be visible after griddepcontrol.wait
(pdl_enter).  In the sources, a kernel's text before the wait may therefore name
parameters that are constants of the solve, and no others."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_05279_gb300", "csrc")

# written by the setup, or uploaded before the first launch of a solve
CONSTANTS = {
    "down_body": {"v", "grid", "ci", "nu1"},
    "up_body": {"v", "grid", "ci", "nu2"},
    "k_tail": {"d"},
    "k_p_coarse_solve": {"g", "L"},
}


def waiting_functions():
    """(name, parameters, text before the wait) of every function that calls pdl_enter."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"pdl_enter\(\);", src):
            start = max(src.rfind(k, 0, m.start()) for k in ("__global__", "__device__ __forceinline__ void"))
            head = re.compile(r"\b(\w+)\(((?:[^()]|\([^()]*\))*)\)\s*\{").search(src, start)
            name, params = head.group(1), re.findall(r"(\w+)\s*(?:,|$)", re.sub(r"<[^<>]*>", "", head.group(2)))
            out.append((name, params, src[head.end():m.start()]))
    return out


FUNCTIONS = waiting_functions()


def test_every_wait_is_found():
    names = [f[0] for f in FUNCTIONS]
    assert len(names) >= 40 and CONSTANTS.keys() <= set(names)
    assert all(f[1] for f in FUNCTIONS if f[0] != "k_wait_selftest")


@pytest.mark.parametrize("name,params,before", FUNCTIONS, ids=[f[0] for f in FUNCTIONS])
def test_only_constants_before_the_wait(name, params, before):
    used = {p for p in params if re.search(rf"(?<!\.)\b{p}\b", before)}
    assert used <= CONSTANTS.get(name, set()), (name, used)
