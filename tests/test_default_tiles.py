"""The library's tile choice in modes with limits of their own: a grid split over ranks needs a tile a
rank, a warp tile is 32, 64, 128 or 256 points wide and divides the grid, a cluster holds at most 16
tiles of one width.  What the rule without the least width accepts stays accepted.  Host only."""
import ctypes

import pytest

from paper_1612_02495_gb300 import swept as S

SMS = 152  # of the plan without a device
CASES = [(S.HEAT, S.F32, 1), (S.HEAT, S.F64, 1), (S.KS, S.F32, 2), (S.KS, S.F64, 2), (S.EULER, S.F64, 2)]
SIZES = [36, 60, 64, 100, 128, 256, 508, 512, 600, 1000, 1009, 1024, 1500, 2048, 3000, 4096, 9760, 19520, 30000, 65536]


def plan(scheme, dtype, n, **kw):
    """(tile width, tiles) of a plan without a tile, or None where swept_init refuses it"""
    cfg = S.make_config(scheme, dtype, n, 0.1, 0.001, 1.4, **kw)
    h = ctypes.c_void_p()
    if S.swept_init(ctypes.byref(cfg), ctypes.byref(h)) != S.SWEPT_OK:
        return None
    info = S.swept_plan_info()
    assert S.swept_get_plan(h.value, ctypes.byref(info)) == S.SWEPT_OK
    S.swept_free(h.value)
    return info.tile_w


def plain_width(n, R):
    """the widest tile up to 1024 with two blocks a SM, else with one, else the narrowest; dividing n if any does"""
    for divides in (True, False):
        legal = [w for w in range(4 * R, 4097, 4 * R) if n // w >= 2 and (n % w == 0 or not divides)]
        for least in (2 * SMS, SMS):
            fit = [w for w in legal if w <= 1024 and n // w >= least]
            if fit:
                return max(fit)
        if legal:
            return min(legal)
    return 0


@pytest.mark.parametrize("scheme,dtype,R", CASES)
def test_warp_tiles(scheme, dtype, R):
    for n in SIZES:
        got = plan(scheme, dtype, n, warp_tiles=1)
        w = plain_width(n, R)
        if scheme != S.EULER and w in (32, 64, 128, 256) and n % w == 0:
            assert got, n
        assert got is None or (got in (32, 64, 128, 256) and n % got == 0)


@pytest.mark.parametrize("scheme,dtype,R", CASES)
def test_cluster(scheme, dtype, R):
    for n in SIZES:
        got = plan(scheme, dtype, n, cluster=1)
        w = plain_width(n, R)
        if w and n % w == 0 and n // w <= 16:
            assert got, n
        assert got is None or (n % got == 0 and n // got <= 16)


@pytest.mark.parametrize("scheme,dtype,R", CASES)
@pytest.mark.parametrize("nranks", [2, 3, 8, 16])
def test_slabs(scheme, dtype, R, nranks):
    for n in SIZES[:16]:
        w = plain_width(n, R)
        if w and n // w >= nranks:
            S.slab_check(scheme, dtype, n, 0.1, 0.001, 1.4, nranks, 5)


def test_calls_of_before():
    """heat warp tiles at 9,760 and 19,520 points, clusters at 36 and 60, eight ranks on 512 and 1,024"""
    for dtype in (S.F32, S.F64):
        assert plan(S.HEAT, dtype, 9760, warp_tiles=1) == 32
    assert plan(S.HEAT, S.F64, 19520, warp_tiles=1) == 64
    for n in (36, 60):
        assert plan(S.HEAT, S.F32, n, cluster=1) and plan(S.HEAT, S.F64, n, cluster=1)
    for scheme in (S.HEAT, S.KS):
        for n, dtype in ((1024, S.F32), (512, S.F32), (512, S.F64)):
            S.slab_check(scheme, dtype, n, 0.1, 0.001, 1.0, 8, 7)


@pytest.mark.parametrize("scheme,dtype", [(S.HEAT, S.F64), (S.EULER, S.F32), (S.KS, S.F32), (S.KS, S.F64)])
def test_last_tile(scheme, dtype):
    """Where no width divides the grid the last tile takes the rest, and every pass waits for it: the widened
    tile leaves less than a quarter of itself (33,003 points in tiles of 256 left 235)"""
    for n in (20011, 33003, 48017, 65003):
        cfg = S.make_config(scheme, dtype, n, 0.1, 0.001, 1.4)
        h = ctypes.c_void_p()
        assert S.swept_init(ctypes.byref(cfg), ctypes.byref(h)) == S.SWEPT_OK
        info = S.swept_plan_info()
        S.swept_get_plan(h.value, ctypes.byref(info))
        S.swept_free(h.value)
        if info.tile_w != plain_width(n, 1 if scheme == S.HEAT else 2):
            assert 4 * info.last_tile_extra <= info.tile_w, (n, info.tile_w, info.last_tile_extra)
