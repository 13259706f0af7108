"""Order of the programmatic-launch instructions in the kernels, read from their sources (no GPU).

A kernel that runs ahead of its own griddepcontrol.wait (the window kernel copies its prepared image there)
relies on every launch but its direct predecessor having ended.  That holds when no kernel launched with
programmatic serialization releases its successor before its own wait.  And its inputs may still be written
while it lives, which the read-only loads (__ldg) do not allow."""
import glob
import os
import re

import pytest

from paper_1908_11263_gb300 import build as qbuild

WAIT = re.compile(r"pdl_wait\(\)|griddepcontrol\.wait")
TRIGGER = re.compile(r"pdl_trigger\(\)|griddepcontrol\.launch_dependents")
# launched in full stream order (<<<>>>): everything before it has ended when it starts
PLAIN = {"conv_tc_prep_kernel"}


def kernels():
    """(name, body) of every __global__ function of the library, comments removed."""
    found = {}
    for path in sorted(glob.glob(os.path.join(qbuild.CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
            start = text.index("{", m.end())
            depth, end = 0, start
            for end in range(start, len(text)):
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                if depth == 0:
                    break
            found[m.group(1)] = (text, text[start:end + 1])
    return found


KERNELS = kernels()


def test_kernels_are_found():
    assert {"conv_win_kernel", "conv_gather_kernel", "conv_tc_prep_kernel", "pack_kernel", "unpack_kernel",
            "maxpool_vec_kernel", "linear_smem_kernel"} <= set(KERNELS)
    # the exemption holds only while that kernel is launched plainly
    text = KERNELS["conv_tc_prep_kernel"][0]
    start = text.index("cudaError_t launch_conv_tc_prep(")
    launch = text[start:text.index("\n}\n", start)]
    assert "<<<" in launch and "cudaLaunchKernelEx" not in launch and "launch_pdl" not in launch


@pytest.mark.parametrize("name", sorted(k for k, (_, body) in KERNELS.items() if TRIGGER.search(body)))
def test_successors_are_released_after_the_own_wait(name):
    if name in PLAIN:
        return
    body = KERNELS[name][1]
    wait = WAIT.search(body)
    assert wait is not None
    assert all(m.start() > wait.end() for m in TRIGGER.finditer(body))


def overlapped_sources():
    """(file, text without the kernels launched in full stream order) of the files with overlapped kernels."""
    for path in sorted(glob.glob(os.path.join(qbuild.CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        if os.path.basename(path) == "device.cuh" or not WAIT.search(text):
            continue
        for name, (_, body) in KERNELS.items():
            if name in PLAIN or not WAIT.search(body):
                text = text.replace(body, "")
        yield os.path.basename(path), text


def test_no_read_only_loads_where_the_predecessor_may_still_write():
    texts = dict(overlapped_sources())
    assert {"pack.cu", "pool.cu", "linear.cu", "conv_win.cuh", "conv_gather.cuh"} <= set(texts)
    assert [name for name, text in texts.items() if re.search(r"__ldg|ld\.global\.nc|__restrict__", text)] == []
