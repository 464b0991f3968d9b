"""Kernels that may start before the kernel ahead of them ends (programmatic dependent
launch) read memory that it is still writing, behind griddepcontrol.wait.  A const
__restrict__ pointer or __ldg tells the compiler that nobody writes that memory while the
kernel runs, so neither may stand in such a kernel.  Read from the source."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1405_2232_gb300", "csrc")
WAITS = re.compile(r"\b(grid_wait|grid_begin|grid_dependency_wait)\(\)")
# written by the host only, between synchronised steps
HOST_TABLES = ("BatchDomain* __restrict__ doms", "BatchStepTile* __restrict__ tiles", "int* __restrict__ n_tiles")


def closing(s, i, pair):
    depth = 0
    for j in range(i, len(s)):
        depth += (s[j] == pair[0]) - (s[j] == pair[1])
        if depth == 0:
            return j
    raise AssertionError("unbalanced")


def kernels():
    """(name, parameters, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        s = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__ void\s+(?:__launch_bounds__)?", s):
            i = m.end()
            if s[:i].endswith("__launch_bounds__"):
                i = closing(s, i, "()") + 1
            p = s.index("(", i)
            q = closing(s, p, "()")
            b = s.index("{", q)
            yield s[i:p].strip(), s[p:q], s[b:closing(s, b, "{}")]


PROGRAMMATIC = [k for k in kernels() if WAITS.search(k[2])]


def test_the_kernels_are_found():
    names = {n for n, _, _ in PROGRAMMATIC}
    assert {"k_step_tile", "k_batch_tile", "k_fd_front", "k_fd_rk2", "k_conv3_tc", "k_conv3_tcs", "k_wgrad_tc",
            "k_pool", "k_up_bwd", "k_skip_bwd", "k_head_fwd", "k_head_bwd", "k_sum_doubles"} <= names


@pytest.mark.parametrize("name,params,body", PROGRAMMATIC, ids=[k[0] for k in PROGRAMMATIC])
def test_no_read_only_promise_on_what_the_kernel_ahead_writes(name, params, body):
    for table in HOST_TABLES:
        params = params.replace(table, "")
    assert not re.search(r"const [^,*]*\*\s*(const\s*)?__restrict__", params), params
    assert "__ldg" not in body and ".nc" not in body


def test_no_launch_of_the_network_drops_its_error():
    """Every launch, convolution and weight gradient of a pass is used in an expression (a
    return, an assignment or UTRY), not called as a statement."""
    s = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "unet.cu")).read())
    names = r"(?:launch|launch_after|conv|wgrad|queue_sums)\("
    statements = [t.strip() for t in re.split(r"[;{}]", s)]
    assert sum(bool(re.search(r"\b" + names, t)) for t in statements) > 30
    dropped = [t for t in statements
               if re.match(r"(?:(?:if|for) \(.*\)\s*|else\s+|case \w+:\s*|default:\s*)*" + names, t, flags=re.S)]
    assert not dropped, dropped
