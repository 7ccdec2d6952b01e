"""Sizing of the created-electron scratch: the largest slices only in contexts
that stage their cells at the large-cell pass's size."""
import ctypes as C

import pytest

import paper_1704_01202_gb300 as pkg
import pic_inputs as P
from paper_1704_01202_gb300 import _grid, _species

NEW_E = 20                         # bytes of a created electron's record (FP32 build)


@pytest.fixture(scope="module")
def build():
    pkg.build()


def _bytes(nx):
    cfg = P.SlabConfig(nx=nx, ppc_e=8, ppc_i=2)
    return pkg.lib().pic_required_bytes(C.byref(_grid(cfg)), C.byref(_species(cfg, 4096, 4096)), 4096, 4096)


def test_whole_staging_scratch_ends_where_the_staging_does(build):
    """Two cells an SM, 304 on 152 SMs: up to there 1536 entries for each cell
    (and 64 more), from there 768."""
    at = 2 * 152
    drop = _bytes(at) - _bytes(at + 1)
    want = NEW_E * ((at + 64) * 1536 - (at + 1 + 64) * 768)
    assert abs(drop - want) < 8192          # the other arrays' cell, alignment of 256
    for nx in (at + 1, 340, 384, 400):
        assert 0 < _bytes(nx + 1) - _bytes(nx) < 2 * 768 * NEW_E, nx
