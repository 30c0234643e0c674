"""Kernels launched as dependents of the one before them (csrc/launch.cuh) are resident while
that one still writes.  What it may write they read by ordinary loads: no __restrict__ on the
parameter, which lets the compiler take the array as constant for the whole kernel, and no __ldg.
Read from the sources: which load the compiler picks shows in no output."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1407_1309_gb300", "csrc")
CONSTANT = {"G", "R", "r", "b"}  # no kernel of a call writes these


def closing(text, start, pair):
    depth = 0
    for i in range(start, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0 and text[i] == pair[1]:
            return i
    raise AssertionError("unbalanced source")


def chained_kernels():
    """(file, kernel, parameter list, body) of every kernel that calls grid_wait()."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^;{]*?\)\s+)?(\w+)\(", text):
            end = closing(text, m.end() - 1, "()")
            stop = closing(text, text.index("{", end), "{}")
            body = text[end:stop]
            if "grid_wait()" in body:
                yield os.path.basename(path), m.group(1), text[m.end():end], body


KERNELS = {k: (f, params, body) for f, k, params, body in chained_kernels()}


def test_the_families_are_found():
    assert {"k_donor", "k_antidiff", "k_antidiff3v", "k_corr3v", "ka_fct_a", "ka_donor_flux", "k_vip_cells",
            "k_trapez_post", "k_tile2d", "k_band2d", "k_fused2d", "k_fused2d_batched"} <= set(KERNELS)


@pytest.mark.parametrize("kernel", sorted(KERNELS))
def test_no_read_only_parameter_that_an_earlier_kernel_writes(kernel):
    file, params, _ = KERNELS[kernel]
    names = set(re.findall(r"__restrict__\s+(\w+)", params))
    # the reverse sweep starts as a dependent of whatever the caller launched: not even G
    assert names <= (set() if file == "adjoint.cu" else CONSTANT), names


@pytest.mark.parametrize("file", sorted({f for f, _, _ in KERNELS.values()}))
def test_read_only_loads_are_of_constant_arrays(file):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, file)).read())
    for arg in re.findall(r"__ldg\(([^;]*)", text):
        assert re.match(r"\(?(G|R|r|b)\b", arg), arg
