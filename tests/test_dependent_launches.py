"""Kernels of a dependent launch read nothing before their wait that the kernels before them may have written.

A kernel may start before its predecessors' writes have been made visible; wait_previous() is where they are.  Only
the tensor and tile tables may be read ahead of it, and only a handle's, which no kernel writes: the kernels that the
allocation-free global step launches, whose tables are written by a kernel of the same call, wait for those first
(Problem::fresh_tables).  A missing wait shows in the source; on a GPU it would show as rare wrong statistics, if at all.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_17866_gb300", "csrc")
FRESH_WAIT = "if (p.fresh_tables) wait_previous();"
# the kernels of dsm_global_step_noalloc after its table kernel: K4 and K5
OF_THE_ALLOCATION_FREE_CALL = {"k_global", "k_global_many", "k_stats"}


def _kernels():
    """name -> body, for every __global__ function."""
    out = {}
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", src):
            start = src.index("{", m.end())
            depth, i = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            out[m.group(1)] = src[start:i]
    return out


KERNELS = _kernels()


def _before_the_wait(body):
    """The statements ahead of the kernel's unconditional wait."""
    m = re.search(r"(?m)^\s*wait_previous\(\);", body)
    assert m, "no unconditional wait_previous()"
    return body[:m.start()]


def test_every_kernel_is_found():
    assert OF_THE_ALLOCATION_FREE_CALL | {"k_init", "k_grad_fill", "k_local_adamw", "k_local_sgdm", "k_noalloc_tables",
                                          "k_fused_last_global"} == set(KERNELS)


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_only_the_tables_are_read_before_the_wait(name):
    head = _before_the_wait(KERNELS[name])
    head = re.sub(r"auto (\w+) = \[&\][\s\S]*?\n    \};", "", head)      # lambdas run where they are called
    assert set(re.findall(r"\bp\.(x|m|gv|X|opt_m|opt_v|grad|partials|stats)\b(?=\s*[\[+])", head)) == set()


@pytest.mark.parametrize("name", sorted(OF_THE_ALLOCATION_FREE_CALL))
def test_tables_of_the_same_call_are_waited_for(name):
    head = _before_the_wait(KERNELS[name])
    reads = [m.start() for m in re.finditer(r"\bp\.(tensors|tiles)\b", head)]
    assert not reads or FRESH_WAIT in head[:reads[0]], f"{name} reads the tables before it waits for their writer"
