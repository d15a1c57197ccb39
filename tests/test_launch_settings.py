"""The process-wide launch setting of the 3-D codec kernels, which answers without
a GPU."""
import pytest

from paper_2609_24294_gb300 import build, zfpx as z


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


# 0 is the library's choice by the launch's size, which no single value stands for: what
# the call returns can be set again without changing anything
@pytest.mark.parametrize("encode", [True, False])
@pytest.mark.parametrize("rate", [8, 16])
def test_units_per_warp_reads_back_what_was_set(encode, rate):
    for other in (True, False):
        for r in (8, 16):
            assert z.zfpx_get_units_per_warp(other, r) == 0
    try:
        for upw in (1, 4096, 2, 0):
            z.zfpx_set_units_per_warp(encode, rate, upw)
            assert z.zfpx_get_units_per_warp(encode, rate) == upw
            assert z.zfpx_get_units_per_warp(not encode, rate) == 0
            assert z.zfpx_get_units_per_warp(encode, 24 - rate) == 0
    finally:
        z.zfpx_set_units_per_warp(encode, rate, 0)
    assert z.zfpx_get_units_per_warp(encode, 12) == -1
