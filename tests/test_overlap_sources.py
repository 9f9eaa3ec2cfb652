"""Kernels that may start while the stream's previous kernel drains (they call grid_wait) read what that kernel
writes with plain loads or cp.async: a load through the non-coherent path (__ldg, or a pointer that is const and
__restrict__) is valid only for data that nothing writes in the kernel's whole lifetime, and grid_wait() does not
order it.  Checked on the sources: such a fault need not show in a run.
"""

import glob
import os
import re

from paper_1603_06442_gb300 import build

# tables that are complete before the first launch that reads them
TABLES = {"omega", "tw_line", "tw_hi", "tw_lo"}


def _kernels(text):
    """(name, parameters, body) of each __global__ function with a body."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__", text):
        head = re.compile(r"(\w+)\s*\(").finditer(text, m.end())
        for h in head:
            end = _close(text, h.end() - 1, "()")
            if h.group(1) in ("__launch_bounds__", "sizeof"):
                continue
            brace = re.compile(r"\s*\{").match(text, end)
            if brace:
                yield h.group(1), text[h.end():end - 1], text[brace.end():_close(text, brace.end() - 1, "{}")]
            break


def _close(text, at, pair):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i + 1
    raise AssertionError("unbalanced %s" % pair)


def test_overlapped_kernels_read_their_field_coherently():
    seen = set()
    for path in glob.glob(os.path.join(build.CSRC, "*.cu")) + glob.glob(os.path.join(build.CSRC, "*.cuh")):
        with open(path) as f:
            text = f.read()
        for name, params, body in _kernels(text):
            if "grid_wait" not in body and "grid_await" not in body:
                continue
            seen.add(name)
            assert "__ldg" not in body, name
            ro = re.findall(r"const\s[^,]*__restrict__\s+(\w+)", params)
            assert set(ro) <= TABLES, (name, ro)
    assert {"march1d_kernel", "march2d_kernel", "march3d_kernel", "fft2f_kernel", "evolve_kernel"} <= seen
