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


def test_register_variants_by_the_walks_of_a_launch(hc):
    """Per-point counts are launched twice, at most 2^20 walks in the small form: that launch takes the
    variant of small solves, whatever the total on the device, the other one that of large ones."""
    for f in (hc.wos_hc_walks_of_launch,):
        f.argtypes, f.restype = [C.c_uint64, C.c_int], C.c_uint64
    hc.wos_hc_value_variant.argtypes = [C.c_int, C.c_int, C.c_uint64]
    limit, unknown = 1 << 20, (1 << 64) - 1

    def variant(dim, bspline, total, small):
        return hc.wos_hc_value_variant(dim, bspline, hc.wos_hc_walks_of_launch(total, small))
    for dim in (2, 3):
        assert variant(dim, 0, unknown, 1) == 0 and variant(dim, 0, unknown, 0) == 1
        for total in (1, limit):
            assert variant(dim, 0, total, 1) == variant(dim, 0, total, 0) == 0
        assert variant(dim, 0, limit + 1, 0) == 1
        for total in (1, limit, limit + 1, unknown):
            for small in (0, 1):
                assert variant(dim, 1, total, small) == (2 if dim == 3 else 0)


def test_next_flight_register_caps(hc):
    """More than four blocks per SM only where they are the faster ones: never for few walks (more of them
    count as few on meshes and with B-spline fields), and never for the printed approximations with 3D
    B-spline fields, whose taps would spill."""
    hc.wos_hc_nf_blocks.argtypes = [C.c_int] * 4 + [C.c_uint64]
    for series in (0, 1):
        for bspline in (0, 1):
            for walks in (1, 1 << 18, 3 << 18):
                assert hc.wos_hc_nf_blocks(3, 1, series, bspline, walks) == 4
            assert hc.wos_hc_nf_blocks(3, 1, series, bspline, (3 << 18) + 1) == 5
        for dim in (2, 3):
            assert hc.wos_hc_nf_blocks(dim, 0, series, 0, 1 << 18) == 4
            assert hc.wos_hc_nf_blocks(dim, 0, series, 1, 1 << 20) == 4
            assert hc.wos_hc_nf_blocks(dim, 0, series, 0, (1 << 18) + 1) == (5 if series else 6)
    assert hc.wos_hc_nf_blocks(3, 0, 0, 1, 1 << 30) == 4
    assert hc.wos_hc_nf_blocks(2, 0, 0, 1, 1 << 30) == 6
    assert hc.wos_hc_nf_blocks(3, 0, 1, 1, 1 << 30) == 5


def test_gradient_forms(hc):
    """Compiled kernels of closed-form fields name their own rounding; generic kernels and those with B-spline
    fields name the same one."""
    assert hc.wos_hc_gradient_form(1, 0) == 2
    assert hc.wos_hc_gradient_form(0, 0) == hc.wos_hc_gradient_form(0, 1) == hc.wos_hc_gradient_form(1, 1) == 1


@pytest.mark.parametrize("real", [4, 8])
@pytest.mark.parametrize("res", [(4, 4, 4), (8, 8, 8), (16, 16, 16), (16, 16, 32), (5, 5, 327), (4, 4, 512), (20, 20, 20),
                                 (17, 16, 32), (64, 128, 1), (65, 126, 1), (4, 2048, 1), (8192, 1, 1), (1, 1, 8192), (65, 127, 1)])
def test_adjoint_copies_fit_and_cost_no_block(hc, res, real):
    """The padded copy of an alpha grid holds every node at its own address, and costs no resident block
    against rows and planes that are one apart; grids above 8192 nodes have none."""
    dim, other = (2 if res[2] == 1 else 3), 5312 + 4 * 33 * 4 * 4 * (2 if res[2] == 1 else 3) * real
    r, out = (C.c_int64 * 3)(*res), (C.c_int * 4)()
    hc.wos_hc_adjoint_copy.argtypes = [C.c_int, C.POINTER(C.c_int64), C.c_int64, C.c_int, C.POINTER(C.c_int)]
    hc.wos_hc_adjoint_copy(dim, r, other, real, out)
    s1, s2, nodes, blocks = out
    close = ((res[0] + 1) * res[1] + 1) * res[2] * real + other
    want = 0 if close > 200 * 1024 else min(4, 228 * 1024 // (close + 1024))
    if res[0] * res[1] * res[2] > 8192:
        assert nodes == 0
    elif nodes:
        assert s1 >= res[0] and (dim == 2 or s2 >= s1 * (res[1] - 1) + res[0])
        assert (res[0] - 1) + s1 * (res[1] - 1) + s2 * (res[2] - 1) < nodes
        assert blocks >= want and other + nodes * real <= 200 * 1024
    else:
        assert want == 0
