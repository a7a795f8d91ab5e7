"""Kernels launched as programmatic dependents may be resident while the kernel
before them still writes.  What they load through global pointers must
therefore not take the non-coherent path (ld.global.nc, __ldg), which is for
data that nothing writes for the kernel's whole life, and no pointer parameter
may be const __restrict__, which lets the compiler take that path by itself.
Checked in the sources: every kernel that launch_after starts begins with
griddepcontrol.wait, its parameters carry no const __restrict__, and neither
its body nor the step object it runs loads non-coherently."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1705_10045_gb300", "csrc")


def _sources():
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(f) as fh:
            out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", fh.read())
    return out


SOURCES = _sources()


def _block(text, at):
    """The brace block of `text` that opens at or after `at`."""
    start = text.index("{", at)
    depth, i = 0, start
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
        if depth == 0:
            return text[start:i]


def _dependent_kernels():
    names = set()
    for text in SOURCES.values():
        for m in re.finditer(r"launch_after\(\s*(\w+)", text):
            names.add(m.group(1))
    found = set()
    for name in names:
        if name.endswith("_kernel"):
            found.add(name)
        else:   # a variable that picks an instance
            for text in SOURCES.values():
                for m in re.finditer(r"auto\s+%s\s*=([^;]*);" % name, text):
                    if "launch_after(" + name in text[m.end():m.end() + 400]:
                        found.update(re.findall(r"(\w+_kernel)<", m.group(1)))
    return sorted(found)


def _kernel(name):
    for f, text in SOURCES.items():
        m = re.search(r"__global__[^;{]*?\b%s\(([^{]*)\)\s*\{" % name, text)
        if m:
            return f, m.group(1), _block(text, m.end() - 1)
    raise AssertionError(f"{name} not found")


def test_the_dependent_launches_are_found():
    assert _dependent_kernels() == ["phase_collide_kernel", "phase_force_kernel", "phase_moments_kernel",
                                    "row_march_kernel", "strip_step_kernel"]


@pytest.mark.parametrize("name", _dependent_kernels())
def test_dependent_kernel_loads_are_coherent(name):
    f, params, body = _kernel(name)
    assert not re.search(r"const\s+\w+(<\w+>)?\s*\*\s*__restrict__", params), params
    text = body
    # the object the kernel hands its work to, in the same file
    for cls in ("RowMarch", "Strip"):
        if re.search(r"\b%s<" % cls, body):
            text += _block(SOURCES[f], re.search(r"struct %s\s*\{" % cls, SOURCES[f]).start())
    wait = body.index("griddepcontrol.wait")
    before = body[:wait]
    for bad in ("load_pop", "__ldg", "ld.global", "load2", "cp.async"):
        assert bad not in before, (name, bad)
    for bad in ("load_pop<false", "__ldg", "ld.global.nc", "load2(", "load2_keep(", "load2_last("):
        assert bad not in text, (name, bad)
    assert not re.search(r"const\s+\w+(<\w+>)?\s*\*\s*__restrict__", text), name
