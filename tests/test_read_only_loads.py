"""Which loads take the read-only path (__ldg, const __restrict__ parameters).

That path is for data nobody writes while the grid exists.  The kernels of a step's chain are
scheduled while the one before them still runs (sph_launch.cuh), and the ensemble's one launch
writes its lists and records anew in every step, so a read-only load of what the kernel before, or
the same launch, writes is a race that no run has to show; the sources are checked instead."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2005_02656_gb300", "csrc")

# file -> the arrays that may be read through the read-only path there
ALLOWED = {
    "sph_find.cuh": set(),
    "sph_neighbors.cu": set(),
    "sph_staged.cu": set(),
    "sph_pairs_fp64.cu": set(),
    "sph_lanes64.cuh": set(),
    "sph_sort.cu": {"org"},       # cell origins: written by k_zero_table, six kernels before
    "sph_pairs32.cuh": set(),     # the ensemble's pair phases
    "sph_ensemble.cu": {"A.hfac"},  # factor table: filled when the ensemble is made
    "sph_update.cu": {"hfac"},    # factor table: its kernel and k_update are ordered plainly
}


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        s = f.read()
    s = re.sub(r"/\*.*?\*/", " ", s, flags=re.S)
    return re.sub(r"//[^\n]*", " ", s)


@pytest.mark.parametrize("name", sorted(ALLOWED))
def test_chain_kernels_read_predecessors_by_ordinary_loads(name):
    s = _code(name)
    assert "__restrict__" not in s
    assert "ld.global.nc" not in s
    bases = set(re.findall(r"__ldg\(\s*&?\s*([A-Za-z_][\w.]*)", s))
    assert len(re.findall(r"__ldg\s*\(", s)) == len(re.findall(r"__ldg\(\s*&?\s*[A-Za-z_]", s))
    assert bases <= ALLOWED[name], bases - ALLOWED[name]


def test_every_dependent_launch_file_is_listed():
    files = {f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))
             and re.search(r"\blaunch_dep(_if)?\(", _code(f)) and f != "sph_launch.cuh"}
    assert files <= set(ALLOWED), files - set(ALLOWED)
