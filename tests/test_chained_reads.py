"""Kernels of a step that start while the one before drains (launch_chained) read what that one
writes with ordinary loads only. The read-only path (__ldg, const __restrict__) requires memory
that is unchanged for the kernel's whole lifetime, which begins before its wait for the kernel
before; that holds only for the tables that host copies write. Read from the sources, without a GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_19277_gb300", "csrc")
TABLES = {"bd", "wl", "solve_of", "seg"}     # written by copies between launches, never by a kernel


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _kernels(text):
    """name -> text of each kernel, parameters and body."""
    out = {}
    for m in re.finditer(r"__global__[^;{]*?(\w+_kernel)\(", text):
        i = text.index("{", m.end())
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        out[m.group(1)] = text[m.start():j]
    return out


def test_chained_kernels_read_kernel_written_memory_with_ordinary_loads():
    names = [f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))]
    texts = {f: _source(f) for f in names}
    plain = {k for t in texts.values() for k in re.findall(r"(\w+_kernel)(?:<[^<>]*>)?<<<", t)}
    seen = set()
    for f, t in texts.items():
        for k, body in _kernels(t).items():
            if "chain_wait()" not in body or k in plain:
                continue
            seen.add(k)
            assert "__ldg" not in body, (f, k)
            assert set(re.findall(r"__restrict__\s+(\w+)", body)) <= TABLES, (f, k)
    assert seen == {"stage_kernel", "prim_pass_kernel", "speeds_kernel", "set_dt_kernel", "glm_decay_kernel",
                    "cooling_kernel"}
    # the halo view's helpers, inlined into the stage kernel
    assert set(re.findall(r"__restrict__\s+(\w+)", texts["kernels.cuh"])) <= TABLES


def test_a_failed_chained_launch_leaves_no_error_behind():
    """A launch by <<< >>> is followed by cudaGetLastError, which reports its error and clears it; the
    extended launch returns its error and has to clear it as well, or the next launch would report it."""
    body = _source("launch.h").split("launch_chained(", 1)[1].split("\n}", 1)[0]
    call = re.search(r"cudaLaunchKernelEx\([^;]*;(.*)", body, re.S)
    assert call and "cudaGetLastError()" in call.group(1)
