"""Kernels launched while the previous one finishes: every thread waits for it before the kernel
lets the next one start (a trigger of one thread counts for its whole block, so one that came
before the wait would let a third kernel take SMs while the first still runs)."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_19959_gb300", "csrc")


def kernels():
    """(file, name, body without comments) of every kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as fh:
            src = re.sub(r"//[^\n]*", "", fh.read())
        for m in re.finditer(r"\b__global__\b", src):
            at = src.index("{", m.start())
            depth, end = 1, at + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            name = re.findall(r"\b(k_\w+)\s*\(", src[m.start():at])[-1]
            yield os.path.basename(path), name, src[at + 1:end - 1]


def at_top_level(body, call):
    """Places where `call` is a statement of its own outside every branch and loop."""
    out = []
    for m in re.finditer(re.escape(call), body):
        before = body[:m.start()].rstrip()
        if before.count("{") == before.count("}") and before[-1:] in (";", "}", ""):
            out.append(m.start())
    return out


def test_the_kernels_are_found():
    assert {name for _, name, _ in kernels()} >= {"k_front", "k_front_tc", "k_enc_tc", "k_conv_tc", "k_dec1_tc", "k_tail",
                                                  "k_conv5_f32", "k_convT_f32"}


@pytest.mark.parametrize("file,name,body", [pytest.param(*k, id=k[1]) for k in kernels()])
def test_all_threads_wait_before_the_next_kernel_may_start(file, name, body):
    waits = at_top_level(body, "grid_dep_wait();")
    assert waits, f"{name} ({file}) has threads that do not wait for the previous kernel"
    for m in re.finditer(re.escape("grid_dep_launch();"), body):
        assert waits[0] < m.start(), f"{name} ({file}) triggers the next kernel before its wait"
