"""The lattice argument of a call (built once per lattice and kept) holds the
extents the caller passed, whatever kind of integers they are."""
import numpy as np
import pytest
import torch


@pytest.fixture(scope="module")
def H():
    from paper_1805_03560_gb300 import build, hmc
    build.build()
    return hmc


def _sites(H, L):
    return H.lib().hmc_spinor_bytes(H._lat_ref(L), H.F64, 1) // 192


@pytest.mark.parametrize("make", [tuple, list, np.array, torch.tensor,
                                  lambda v: [np.array(e) for e in v],
                                  lambda v: [np.int32(e) for e in v],
                                  lambda v: [torch.tensor(e) for e in v]])
def test_kinds_of_extents(H, make):
    assert _sites(H, make([8, 4, 6, 10])) == 8 * 4 * 6 * 10 // 2


def test_extents_changed_in_place(H):
    L = [torch.tensor(v) for v in (8, 4, 6, 10)]
    assert _sites(H, L) == 960
    L[0].fill_(16)
    assert _sites(H, L) == 1920


def test_other_numbers_and_counts(H):
    """Whole floats convert and missing extents are zero (an invalid lattice), as lattice() has it."""
    assert _sites(H, (8.0, 4.0, 6, 10)) == 960
    assert _sites(H, (8, 4, 6)) == 0
    with pytest.raises(IndexError):
        _sites(H, (8, 4, 6, 10, 2))
