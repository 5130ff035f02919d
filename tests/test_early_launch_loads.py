"""Kernels that may be on the device before their predecessor has ended
(launch_after in csrc/wcns_internal.h) read what that predecessor writes with
ordinary loads.  A non-coherent load (__ldg, or a const __restrict__ pointer)
promises an array that is read-only for the whole life of the kernel, which
there begins before the wait.  Read from the sources, without a GPU; only the
Dirichlet face arrays, which no kernel writes, may be read that way."""
import os
import re

import pytest

from tests.conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2102_05287_gb300", "csrc")
SWEEPS = ("wcns_sweep.cuh", "wcns_mixed_body.cuh")  # the sweep kernels and their bodies


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/|//[^\n]*", "", text, flags=re.S)


@pytest.mark.parametrize("name", SWEEPS)
def test_noncoherent_loads_read_dirichlet_faces_only(name):
    text = source(name)
    assert "after_predecessor()" in text
    loads = re.findall(r"(?:__ldg|ld\.global\.nc|__ldcs|__ldlu)\b[^;]*;", text)
    assert all(re.match(r"__ldg\(face \+", x) for x in loads), loads
    assert "__restrict__" not in text


def test_early_arguments_are_not_restrict():
    """SweepArgs carries the sweeps' pointers, StepCtl those of step_begin."""
    assert "__restrict__" not in source("wcns_internal.h")
    early = re.findall(r"__global__[^{]*\{\s*(?:extern[^;]*;\s*)?after_predecessor\(\);", source("wcns_api.cu"))
    assert len(early) == 1 and all("__restrict__" not in k for k in early), early
