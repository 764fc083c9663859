"""Kernels that follow one another programmatically (csrc/lbmhd_pdl.cuh): such a
grid starts while the one before it still writes what it will read, so its
loads must be ordinary ones behind the wait.  A `__restrict__` on a kernel's
pointer, or __ldg, lets the compiler take them for loads of data that no one
writes while the grid exists (the non-coherent path), which may also move above
the wait.
"""
import glob
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1607_08675_gb300", "csrc")


def kernels():
    """(file, name, parameters, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__", text):
            # the parameter list: the last parenthesis before the body
            start = text.index("{", m.end())
            head = text[m.end():start]
            name = re.findall(r"(\w+)\s*\(", head)[-1]
            params = head[head.rindex(name):]
            depth, end = 0, start
            while True:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
                if depth == 0:
                    break
            yield os.path.basename(path), name, params, text[start:end]


def test_programmatic_kernels_load_what_the_grid_before_them_wrote():
    found = {k[1]: k for k in kernels() if "after_previous()" in k[3]}
    assert {"step_kernel", "step_kernel_h8", "pipe_kernel", "kin_pipe_kernel", "batch_pipe_kernel",
            "adj_step_kernel"} <= set(found)
    for file, name, params, body in found.values():
        assert "__restrict__" not in params, (file, name)
        assert "__ldg" not in body, (file, name)
        # nothing but types, constants and shared memory before the wait
        before = [x.strip() for x in body[1:body.index("after_previous()")].split(";")]
        assert all(re.match(r"using |constexpr |__shared__ |$", x) for x in before), (file, name, before)


def test_only_kernels_that_wait_are_launched_programmatically():
    waits = {k[1] for k in kernels() if "after_previous()" in k[3]}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(path).read()
        for m in re.finditer(r"launch_after\(\s*(\w+)", text):
            name = m.group(1)
            if name == "even":  # a choice between two instances
                name = "batch_pipe_kernel"
            if name not in waits:  # a local: every kernel it may hold
                held = re.findall(r"auto %s = ([^;]*);|\b%s = ([^;]*);" % (name, name), text)
                names = {w for h in held for w in re.findall(r"(\w+_kernel(?:_\w+)?)\b", " ".join(h))}
                assert names and names <= waits, (path, name, names)
