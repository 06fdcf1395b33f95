"""Kernels that call overlap_wait() are resident while the kernel before them still writes the
buffers they read, so they must not read them through the non-coherent path: __ldg is left to
tables and weights that no kernel writes. Checked in the sources, since a stale read shows on a
GPU by chance only.
"""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_08229_gb300", "csrc")

# what the loads of these files may read non-coherently: the symmetry table, the network's
# parameters, the phase tables
TABLES = re.compile(r"__ldg\(reinterpret_cast<const (int4\*>\(d\.sym|uint4\*>\(src\)|float4\*>\(tab)")


def _code(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def _with_headers(name, seen=None):
    seen = set() if seen is None else seen
    if name not in seen:
        seen.add(name)
        for inc in re.findall(r'#include "([^"/]+)"', _code(name)):
            _with_headers(inc, seen)
    return seen


OVERLAPPED = sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu"))
                    if "overlap_wait()" in _code(os.path.basename(p)))


def test_overlapped_kernels_are_known():
    assert OVERLAPPED == ["kernels_adjoint.cu", "kernels_force.cu", "kernels_nco_f32.cu", "kernels_step.cu"]


@pytest.mark.parametrize("name", OVERLAPPED)
def test_overlapped_kernels_read_by_plain_loads(name):
    for part in _with_headers(name):
        for line in _code(part).splitlines():
            if "__ldg(" in line:
                assert TABLES.search(line), (part, line.strip())
