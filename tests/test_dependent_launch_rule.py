"""A kernel launched dependently on the one before (launch.cuh) starts while that one still writes: it has to wait
before it reads, and its loads must not claim that the data is read-only for the kernel's whole life."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2608_18469_b200", "csrc")


def _sources():
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            text = open(os.path.join(CSRC, f)).read()
            out[f] = re.sub(r"//[^\n]*", "", text)
    return out


def _kernels():
    """name -> (parameters, body) of every __global__ function."""
    out = {}
    for text in _sources().values():
        for m in re.finditer(r"__global__\s+void\s+(?:__\w+__\s*\([^)]*\)\s*)*(\w+)\s*\(", text):
            at, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(text[at], 0)
                at += 1
            params, beg = text[m.end():at - 1], text.index("{", at)
            end, depth = beg + 1, 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            out[m.group(1)] = (params, text[beg:end])
    return out


def _dependent():
    """Names of the kernels that go through pdl_launch / pdl_launch_cluster: all but the ones launched with <<< >>>."""
    plain = set()
    for text in _sources().values():
        plain |= set(re.findall(r"(\w+)(?:<[^<>;]*>)?\s*<<<", text))
    return sorted(set(_kernels()) - plain)


def test_every_dependent_kernel_waits():
    names = _dependent()
    assert len(names) > 40
    kernels = _kernels()
    assert [n for n in names if "pdl_wait();" not in kernels[n][1]] == []


@pytest.mark.parametrize("name", _dependent())
def test_inputs_are_not_declared_read_only(name):
    params, body = _kernels()[name]
    assert not re.search(r"const\s+[\w:]+\s*\*\s*__restrict__", params), params
    assert "__ldg(" not in body


def test_no_read_only_loads_in_shared_helpers():
    for name, text in _sources().items():
        assert "__ldg(" not in text and "ld.global.nc" not in text, name
