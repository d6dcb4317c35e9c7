"""Every copy and clear of device memory names its stream (CPU, by reading the sources).

A context's stream is a non-blocking one: it does not wait for the default stream, and a copy
from pageable memory on the default stream may return before its data is on the device.  A kernel
launched next on the context's stream could then read what is not there yet, so nothing in the
library may use the default stream's forms."""
import os
import re

import pytest

from .conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2312_05890_gb300", "csrc")
DEFAULT_STREAM = re.compile(r"\b(cudaMemcpy(2D|3D|ToSymbol|FromSymbol|ToArray|FromArray|Peer)?|cudaMemset(2D|3D)?)\s*\(")


def _code(path):
    src = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h"))))
def test_no_copy_on_the_default_stream(name):
    assert [m.group(0) for m in DEFAULT_STREAM.finditer(_code(os.path.join(CSRC, name)))] == []


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_every_launch_names_a_stream(name):
    for m in re.finditer(r"<<<(.*?)>>>", _code(os.path.join(CSRC, name)), flags=re.S):
        depth, commas = 0, 0
        for ch in m.group(1):
            depth += (ch in "([{") - (ch in ")]}")
            commas += ch == "," and depth == 0
        assert commas == 3, m.group(0)
