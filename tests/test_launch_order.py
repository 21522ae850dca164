"""Kernels that may be set up while the one before them still runs (programmatic
dependent launch) wait before their first access, and take no __restrict__
pointer, which would let the compiler move a load above that wait."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1907_02289_gb300", "csrc")


def kernels():
    """(name, parameters, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(", src):
            brace = src.index("{", m.end())
            if ";" in src[m.end():brace]:
                continue  # a declaration
            depth, end = 0, brace
            while True:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
                if depth == 0:
                    break
            yield pytest.param(src[m.end():brace], src[brace + 1:end - 1], id=m.group(1))


def test_every_kernel_is_seen():
    names = [k.id for k in kernels()]
    launched = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        launched |= set(re.findall(r"(?<![\w>.])(k_[a-z]\w*)\b", re.sub(r"//[^\n]*", "", open(path).read())))
    assert launched == set(names)


@pytest.mark.parametrize("params,body", list(kernels()))
def test_waits_before_its_first_access(params, body):
    if "launch_wait();" not in body:
        assert "launch_" not in body  # (launched the plain way: see below)
        return
    assert re.match(r"\s*launch_wait\(\);", body), "not the first statement"
    assert "__restrict__" not in params


def test_plain_kernels_are_launched_the_plain_way():
    plain = {k.id for k in kernels() if "launch_wait();" not in k.values[1]}
    early = re.compile(r"\b(?:launch|launch_on|launch_levels)\((?:[^;]*?)\b(k_\w+)\b")
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        assert not plain & set(early.findall(src))
