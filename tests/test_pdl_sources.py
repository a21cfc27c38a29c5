"""Kernels that are launched as programmatic dependents begin before the kernels
in front of them have written what they read.  Every such kernel waits before
its first access to memory, and nothing lets the compiler or the read-only data
path take a load before that wait: no __ldg and no __restrict__ kernel
parameter in the library's sources."""
import os
import re

import pytest

from paper_1512_03662_gb300 import build

CSRC = build.CSRC


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        s = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))


def _closing(s, i):
    depth = 0
    while True:
        depth += {"(": 1, ")": -1}.get(s[i], 0)
        if depth == 0:
            return i
        i += 1


def _kernels(s):
    """(name, parameters, start of the body) of every __global__ function defined in s."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(k_\w+)\s*\(", s):
        end = _closing(s, m.end() - 1)
        yield m.group(1), s[m.end():end], s[end + 1:end + 200]


@pytest.mark.parametrize("name", build.SOURCES)
def test_kernels_wait_first_and_their_parameters_promise_nothing(name):
    s = _code(name)
    found = list(_kernels(s))
    assert len(found) == s.count("__global__")
    for kernel, params, body in found:
        assert "__restrict__" not in params, kernel
        assert re.match(r"\s*\{\s*pdl_wait\(\);", body), kernel


@pytest.mark.parametrize("name", build.SOURCES + ["common.cuh", "kernels.h", "emu64.cuh"])
def test_no_load_takes_the_read_only_path(name):
    s = _code(name)
    assert "__ldg" not in s and "ld.global.nc" not in s
    assert "<<<" not in s                                   # every launch goes through launch_k or its attribute


@pytest.mark.parametrize("name", build.SOURCES + ["common.cuh", "kernels.h"])
def test_no_kernel_lets_its_dependent_in_before_it_ends(name):
    """Kernels that trigger at their start pile up on the SMs when calls are queued
    one after another, each waiting for the one before, and a later one's blocks
    go to whichever SMs are left: mid-size residuals took up to 2.5 times as long."""
    s = _code(name)
    assert "launch_dependents" not in s and "cudaTriggerProgrammaticLaunchCompletion" not in s
