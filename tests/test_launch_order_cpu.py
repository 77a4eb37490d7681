"""Kernels that start early touch no data before they have waited.

A kernel launched with launch_after() becomes resident while the kernel before it still writes.
after_previous_grid() is a memory barrier to the compiler, but not for a __restrict__ pointer that
does not go through it: nothing else may write its data, so its loads may move above the barrier.
Read from the sources: every kernel that is launched early waits, before its first access to
anything but its arguments and indices, and passes every __restrict__ pointer it has.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1703_02652_gb300", "csrc")


def _kernels():
    """Name, parameter list and body of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as fh:
            src = re.sub(r"//[^\n]*", "", fh.read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(([^{]*?)\)\s*\{", src):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            yield m.group(1), m.group(2), src[m.end():end - 1]


def _sources():
    return "".join(open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))))


def test_every_early_kernel_waits_and_passes_its_restrict_pointers():
    waits = {}
    for name, params, body in _kernels():
        calls = list(re.finditer(r"after_previous_grid\(([^)]*)\)", body))
        if not calls:
            continue
        waits[name] = True
        restrict = set(re.findall(r"__restrict__\s+(\w+)", params))
        for c in calls:
            passed = set(re.findall(r"\w+", c.group(1)))
            assert restrict <= passed, (name, restrict - passed)
        before = body[:calls[0].start()]
        for p in re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)\s*(?:,|$)", params):
            assert not re.search(rf"\b{p}\b\s*\[|\*\s*{p}\b", before), (name, p)
    src = _sources()
    early = set(re.findall(r"launch_after\(\s*(?:a\.flow \? )?(k_\w+)", src))
    early |= {"k_steps_cluster"}  # its own launch, with the cluster attribute
    assert {"k_step", "k_step_pull_x2", "k_step_aa_x2", "k_macro", "k_finalize", "k_check",
            "k_adj_reverse", "k_adj_reverse_x2"} <= early
    assert early <= set(waits), early - set(waits)
