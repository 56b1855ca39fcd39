"""Kernels that may begin while the launch before them still runs (no GPU needed).

Such a kernel waits (grid_dep_wait) before it touches what that launch writes.
A __restrict__ pointer among its parameters would tell the compiler that
nothing else writes that memory while the kernel runs, so that a load could
move above the wait or go through the read-only path, which need not see the
other launch's writes.  So these kernels take none."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_10965_gb300", "csrc")


def _kernels():
    """(name, parameters, body) of every kernel in the sources"""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\b[^;{]*?\b(k_\w+)\s*\(", text):
            body = text.index(") {", m.end() - 1)
            yield m.group(1), text[m.end():body], text[body:text.index("\n}\n", body)]


OVERLAPPED = {name: params for name, params, body in _kernels() if "grid_dep_wait()" in body}


def test_every_overlapping_launch_waits():
    """launch_pdl starts only kernels that wait"""
    text = "".join(open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cu*")))
    started = set()
    for m in re.finditer(r"launch_pdl\((.*?);", re.sub(r"\\\n", " ", text), flags=re.S):
        started |= set(re.findall(r"\b(k_\w+)", m.group(1)))
    started |= set(re.findall(r"k_s2_panel_rot\b", text))  # by a pointer
    assert started and started <= set(OVERLAPPED)


@pytest.mark.parametrize("name", sorted(OVERLAPPED))
def test_no_restrict_on_what_the_launch_before_writes(name):
    assert "__restrict__" not in OVERLAPPED[name]
