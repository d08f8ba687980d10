"""Kernels that may be scheduled while their predecessor still runs (launch_after / after_previous): what the
source must keep to for their loads to stay behind the wait."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_10158_gb300", "csrc")


def kernels():
    """(file, name, parameters, body) of every __global__ function."""
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
            close = depth = 0
            for i in range(m.end() - 1, len(text)):
                depth += {"(": 1, ")": -1, "{": 1, "}": -1}.get(text[i], 0)
                if depth == 0 and text[i] == ")" and not close:
                    close = i
                if depth == 0 and text[i] == "}":
                    yield name, m.group(1), text[m.end():close], text[close:i]
                    break


def dependent():
    return [k for k in kernels() if "after_previous()" in k[3]]


def test_kernels_are_found():
    names = {k[1] for k in dependent()}
    assert {"rs_hist", "rs_pass", "det_begin", "fold_validate", "fold_tiles", "det_finish", "oe_validate", "oe_fold",
            "oe_in_order", "oe_commit", "rank_mark", "rank_scan", "rank_assign"} <= names


def test_no_restricted_pointers():
    """The compiler may take `const T* __restrict__` for data that nobody writes during the kernel; these
    kernels' predecessors do."""
    bad = [(f, n) for f, n, params, _ in dependent() if "__restrict__" in params]
    assert not bad, bad


def test_every_launch_after_names_a_kernel_that_waits():
    waits = {k[1] for k in dependent()}
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
            for m in re.finditer(r"launch_after\(\s*(\w+)", text):
                if m.group(1) not in ("void",):
                    kernel = m.group(1)
                    if kernel == "validate":           # the three widths of fold_validate
                        kernel = "fold_validate"
                    assert kernel in waits, (name, kernel)


def test_only_shared_memory_is_touched_before_the_wait():
    """Before after_previous() a kernel clears its own shared memory and nothing else."""
    for f, n, params, body in dependent():
        before = body[:body.index("after_previous()")]
        for p in re.findall(r"\*\s*(?:const\s+)?(\w+)\s*(?:,|$)", params):
            assert not re.search(rf"\b{p}\b\s*(\[|\+|->)|\*\s*{p}\b", before), (f, n, p)
        assert not re.search(r"\ba\.\w+\[", before), (f, n)
