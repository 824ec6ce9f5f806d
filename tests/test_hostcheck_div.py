"""The division by a known integer of the next-flight series (w_div_known) against the division."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def hc():
    from paper_2201_13240_gb300 import build as B
    lib = C.CDLL(B.build_hostcheck())
    lib.wos_hc_div_known.restype = C.c_int64
    return lib


@pytest.mark.parametrize("d", range(3, 14))
def test_every_mantissa_divides_exactly(hc, d):
    """Every 24-bit mantissa, at the smallest exponent that is claimed (|t| >= 2^-100) and at |t| < 1 / 2."""
    assert hc.wos_hc_div_known(d, -123) == 0
    assert hc.wos_hc_div_known(d, -25) == 0
