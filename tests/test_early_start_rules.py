"""The rules that a kernel which may start before the one ahead of it ends has
to keep, checked in the sources: it waits before it touches global memory, and
the pointers whose loads the compiler may take for read-only (`const
__restrict__`, __ldg) are hidden from it until then by settled()."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1802_07210_gb300", "csrc")
SOURCES = {os.path.basename(f): re.sub(r"//[^\n]*", "", open(f).read())
           for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}
# of a kernel that is only launched in order: the dense argmin's cells
IN_ORDER = {("dense.cu", "ref"), ("dense.cu", "oth"), ("dense.cu", "glist")}
# read-only parameters that every caller passes a settled pointer for
SETTLED_BY_CALLERS = {"load_win", "warp_best_disparity"}


def _early_kernels():
    names = set()
    for text in SOURCES.values():
        for call in re.findall(r"launch_after\(([^;]*);", text):
            names |= set(re.findall(r"\b(\w+_kernel)\b", call))
    return sorted(names)


def test_early_kernels_are_found():
    assert {"redundancy_grid_kernel", "dt_pass_block_kernel", "median3_kernel", "speckle_border_kernel"} <= \
        set(_early_kernels())
    assert len(_early_kernels()) >= 24


@pytest.mark.parametrize("name", _early_kernels())
def test_waits_first(name):
    bodies = [text[m.end():] for text in SOURCES.values()
              for m in re.finditer(r"\b%s\([^;{}]*\)\s*\{" % name, text)]
    assert bodies
    for body in bodies:
        for statement in body.split(";"):
            statement = statement.strip()
            if not re.match(r"(extern\s+)?__shared__|constexpr", statement):
                assert statement == "after_previous()"
                break


def test_read_only_locals_are_settled():
    for file, text in SOURCES.items():
        found = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)\s*=\s*([^;]*);", text)
        assert file != "support.cu" or found
        for name, value in found:
            assert value.startswith("settled(") or (file, name) in IN_ORDER, "%s: %s = %s" % (file, name, value)


def test_read_only_parameters_are_settled():
    """Of device functions (kernels' own are covered above: a kernel that waits settles them)."""
    seen = 0
    for file, text in SOURCES.items():
        for m in re.finditer(r"__device__ __forceinline__ [\w ]+?(\w+)\(([^;{}]*)\)\s*\{", text):
            for p in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", m.group(2)):
                seen += 1
                start = text[m.end():m.end() + 400]
                assert m.group(1) in SETTLED_BY_CALLERS or "%s = settled(%s);" % (p, p) in start, (file, m.group(1), p)
    assert seen >= 5
    d = SOURCES["post.cu"]
    assert "d = settled(d);" in d[d.index("median3_kernel(const"):][:600]
