"""Kernels launched with programmatic serialization are resident while the kernel before them still writes
their inputs: they may not read those through the non-coherent path.  A check of the sources (CPU only):
no kernel that waits for the one before it uses __ldg, ld.global.nc or __restrict__ pointers, but for plan
memory (plan_load), which no kernel writes after the plan is made."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1812_00904_gb300", "csrc")
READ_ONLY = re.compile(r"__ldg\s*\(|ld\.global\.nc|__restrict__")
PLAN_ARRAYS = {"p.rank", "p.seglist"}  # filled while the plan is made


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def kernels(text):
    """(name, text from __global__ to the closing brace) of every kernel."""
    for m in re.finditer(r"__global__", text):
        head = text[m.start():text.index("{", m.start())]
        depth, i = 0, m.start() + len(head)
        while True:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
            if depth == 0:
                break
        name = re.findall(r"(\w+)\s*\(", head)[-1] if "launch_bounds" not in head else \
            re.findall(r"\)\s*(\w+)\s*\(", head)[-1]
        yield name, text[m.start():i]


def overlapped_kernels():
    files = [f for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))]
    launched = set()
    for f in files:
        for call in re.findall(r"launch_overlapped\(\s*(\w+)", source(f)):
            launched.add(call)
    for f in files:
        for name, body in kernels(source(f)):
            if "grid_wait()" in body or "StepFeed" in body or name in launched:
                yield f, name, body


def test_every_overlapped_kernel_is_seen():
    names = {n for _, n, _ in overlapped_kernels()}
    assert {"pass_kernel", "mvdot_kernel", "mvscatter_kernel", "dvalues_kernel", "finish_kernel", "interleave_kernel",
            "dot_kernel", "xr_update_kernel", "p_update_kernel"} <= names


@pytest.mark.parametrize("f,name,body", list(overlapped_kernels()), ids=lambda v: v if len(v) < 40 else "")
def test_overlapped_kernel_reads_its_inputs_by_plain_loads(f, name, body):
    assert not READ_ONLY.findall(body), f"{f}: {name}"
    assert set(re.findall(r"plan_load\(([\w.]+)", body)) <= PLAN_ARRAYS, f"{f}: {name}"


def test_helpers_of_the_passes_read_by_plain_loads():
    for f in ("pass_kernel.cuh", "zones.cuh"):
        assert not READ_ONLY.findall(source(f)), f
