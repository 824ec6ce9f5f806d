"""The rules that choose a kernel's form by sizes, types and fields (wos_rules.h), asked through the
host check library."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def hc():
    from paper_2201_13240_gb300 import build as B
    return C.CDLL(B.build_hostcheck())


@pytest.mark.parametrize("lanes", [4, 6, 8])
def test_only_gathered_ends_change_the_sums(hc, lanes):
    """Window and mesh walks end one by one: their sums and items are the same in every kernel, also
    in those compiled for problems whose plain walks gather six or eight ends."""
    assert not hc.wos_hc_sums_in_fp64(0, 0, lanes)
    assert not hc.wos_hc_finds_item_again(0, lanes)
    assert bool(hc.wos_hc_sums_in_fp64(0, 1, lanes)) == (lanes >= 6)
    assert bool(hc.wos_hc_finds_item_again(1, lanes)) == (lanes == 8)
    assert hc.wos_hc_sums_in_fp64(1, 0, lanes) and hc.wos_hc_sums_in_fp64(1, 1, lanes)
