"""Loads of the chained kernels (no GPU: reads the sources).

A kernel launched with programmatic stream serialization is resident while its
predecessor still writes the data it will read.  The non-coherent path
(ld.global.nc, __ldg) is defined only for memory that nothing writes during the
kernel, so it is allowed for weights, DFT matrices, tile lists and what earlier
passes left, and for nothing else.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1804_02418_gb300", "csrc")

# what a __ldg may read: (file, a part of its argument)
CONSTANT = {
    "kernels.cuh": ["b.tile_start"],
    "massive.cu": [],
    "fno_fused.cuh": ["(p + (long long)r * N + kg * 8)",      # load_modes: DFT matrices
                      "(p) + i",                              # load_sites: DFT matrices
                      "p.A1", "p.A2",                         # DFT matrices
                      "w + i * kC + lane",                    # mixing matrices
                      "(Q1) + i", "(p.Q1) + i", "(p.W) + tid",   # weights
                      "(p.z + "],                             # kept by the forward pass
}


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", ["site.cuh", "kernels.cuh", "prec_impl.cuh", "massive.cu", "fno_fused.cuh"])
def test_no_non_coherent_assembly(name):
    assert "ld.global.nc" not in _code(name)


@pytest.mark.parametrize("name", sorted(CONSTANT))
def test_read_only_loads_touch_constant_data_only(name):
    for line in _code(name).splitlines():
        for arg in re.findall(r"__ldg\((.*)", line):
            assert any(c in arg for c in CONSTANT[name]), line.strip()
