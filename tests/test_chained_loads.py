"""Kernels launched chained do not read their input through the read-only path (source check, no GPU).

A chained kernel's blocks are resident while the kernel in front still writes their input, and CUDA asks that data
read with __ldg (or through a const __restrict__ pointer read directly) stay unchanged for the kernel's lifetime.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_00477_gb300", "csrc")
CHAINED = ["cu_kernels.cuh", "k_band.cu", "k_wide.cu"]


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_every_chained_kernel_is_looked_at():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")) and ("chain_wait()" in code(name) or "griddepcontrol.wait" in code(name)):
            assert name in CHAINED, name


def test_no_read_only_loads():
    for name in CHAINED:
        text = code(name)
        assert "__ldg(" not in text, name
        # in[...] read directly: only through cp.async, __ldcg or ld_chained
        assert not re.search(r"(?<!\w)in\[", text), name
