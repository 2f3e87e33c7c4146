"""Kernels that are there while the kernel before them still writes read by ordinary loads.

A load through the read-only path promises memory that does not change during the kernel's life, and the compiler may move
it ahead of the wait for the kernel before.  No run shows that reliably, so the sources are looked at.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_16579_b200", "csrc")


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def _kernels(code):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__", code):
        params_at = re.compile(r"(\w+)\s*\(((?:[^()]|\([^()]*\))*)\)\s*\{").search(code, m.end())
        depth, i = 1, params_at.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            i += 1
        yield params_at.group(1), params_at.group(2), code[params_at.end():i]


def test_no_read_only_loads_in_overlapped_kernels():
    seen, bad = 0, []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        code = _code(path)
        overlapped = [k for k in _kernels(code) if "grid_dependency_" in k[2]]
        seen += len(overlapped)
        if overlapped and "__ldg" in code:     # (in a kernel or in a function that one of them calls)
            bad.append(f"{os.path.basename(path)}: __ldg")
        for name, params, _ in overlapped:
            if re.search(r"const\s[^,]*\*\s*__restrict__", params):
                bad.append(f"{os.path.basename(path)}: {name}: a const pointer with __restrict__")
    assert seen >= 12
    assert not bad, bad
