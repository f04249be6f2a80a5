"""Kernels launched as programmatic dependents (dg_launch_after): what they may
declare read-only, and that they wait before they touch memory."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_01492_gb300", "csrc")

# coefficient data: written by dg_set_coefficient, which waits for the device
FIXED = {"lineop", "gam", "expM", "expG"}


def sources():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        yield re.sub(r"//[^\n]*", "", open(f).read())


def dependents():
    """(name, parameters, body) of every kernel launched with dg_launch_after."""
    texts = list(sources())
    names = {n for t in texts for n in re.findall(r"dg_launch_after\(\s*(k_\w+)", t)}
    out = []
    for t in texts:
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(([^{]*)\)\s*\{", t):
            if m.group(1) in names:
                out.append((m.group(1), m.group(2), t[m.end():m.end() + 4000]))
    assert {n for n, _, _ in out} == names and names
    return out


def test_data_of_earlier_kernels_is_not_declared_read_only():
    for name, params, _ in dependents():
        const = re.findall(r"const\s+[\w ]+\*\s*__restrict__\s+(\w+)", params)
        assert set(const) <= FIXED, (name, const)


def test_dependents_wait_before_they_touch_memory():
    for name, _, body in dependents():
        stmts = [s.strip() for s in body.split(";")]
        at = next(i for i, s in enumerate(stmts) if s.endswith("dg_wait_before()"))
        for s in stmts[:at]:
            assert s.startswith("constexpr") or s == "dg_release_next()", (name, s)
