"""The runtime-length forms' radix schedules and index arithmetic (csrc/any_sched.h, built here
with g++ through a test shim): for every length a plan can have, the in-place stages touch
each slot once, stay inside the tile, and leave the DFT in the slots the kernels read it
from.  No GPU needed."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1612_01799_gb300", "csrc")


def counts():
    for n in range(4, 1025, 2):
        m = n
        for f in (2, 3, 5):
            while m % f == 0:
                m //= f
        if m == 1:
            yield n


SMS = 152
TILE = ("lg", "threads", "few", "ctas", "smem", "rounds", "few_rounds")


def tile(shim, L, df, f32, rows, groups=10 ** 6, planes=1):
    out = (ctypes.c_int * 7)()
    assert shim.shim_any_tile(L, df, f32, rows, ctypes.c_longlong(groups), planes, SMS, out) == 0, L
    return dict(zip(TILE, out))


def plane(shim, nx, ny, df, f32, planes=1):
    out = (ctypes.c_int * 3)()
    shim.shim_plane_tile(nx, ny, df, f32, SMS, planes, out)
    return tuple(out)


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("shim") / "any_sched.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC,
                    os.path.join(HERE, "native", "any_sched_shim.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    P = ctypes.POINTER(ctypes.c_double)
    lib.shim_any_transform.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_int, P, P]
    return lib


@pytest.mark.parametrize("max_radix", [10, 12])
@pytest.mark.parametrize("rows", [0, 1])
@pytest.mark.parametrize("pad", [0, 1])
def test_every_length_is_a_dft(shim, max_radix, rows, pad):
    """rows: the x passes' lengths n (last radix at most 8), else the column passes' 2 n."""
    P = ctypes.POINTER(ctypes.c_double)
    for n in counts():
        L = n if rows else 2 * n
        rng = np.random.default_rng(L)
        x = rng.standard_normal(2 * L)
        X = np.zeros(2 * L)
        rc = shim.shim_any_transform(L, max_radix, 8 if rows else max_radix, pad, x.ctypes.data_as(P),
                                     X.ctypes.data_as(P))
        assert rc == 0, (L, rc)
        ref = np.fft.fft(x.view(complex))
        assert np.abs(X.view(complex) - ref).max() <= 1e-12 * np.abs(ref).max() * np.log2(L), L


@pytest.mark.parametrize("max_radix", [10, 12])
@pytest.mark.parametrize("rows", [0, 1])
def test_kernel_covers_the_radices(shim, max_radix, rows):
    """Radix 12 only where it saves a stage, and never in a kernel compiled up to 10."""
    for n in counts():
        L = n if rows else 2 * n
        for pad in (0, 1):
            assert shim.shim_any_radix_rule(L, max_radix, 8 if rows else max_radix, pad) == 0, L


@pytest.mark.parametrize("df,f32", [(0, 1), (0, 0), (1, 0)])
@pytest.mark.parametrize("rows", [0, 1])
def test_tiles_fit_and_few_threads_save_rounds(shim, df, f32, rows):
    """Every tile fits a block's shared memory and the kernels' threads; the threads of a launch
    of few tiles are those of a full chip or take fewer rounds."""
    for n in counts():
        t = tile(shim, n if rows else 2 * n, df, f32, rows)
        assert t["smem"] <= 232448 - 1024 and t["lg"] in (1, 2, 3), (n, t)
        assert 64 <= t["threads"] <= 256 and t["threads"] % 32 == 0, (n, t)
        assert 64 <= t["few"] <= 256 and t["few"] % 32 == 0 and t["ctas"] >= 1, (n, t)
        assert t["few"] == t["threads"] or t["few_rounds"] < t["rounds"], (n, t)


def test_few_tiles(shim):
    """Double-float N = 30: the z pass's 80 butterflies of radix 6 take one round instead of two.  A
    launch is of few tiles up to the CTAs that fit the SMs and three warps to a scheduler."""
    t = tile(shim, 60, 1, 0, 0)
    assert t["threads"] == 64 and t["few"] == 96 and (t["rounds"], t["few_rounds"]) == (22, 16)
    assert shim.shim_any_is_few(64, 5, SMS, 5 * SMS) and not shim.shim_any_is_few(64, 5, SMS, 5 * SMS + 1)
    assert shim.shim_any_is_few(128, 8, SMS, 3 * SMS) and not shim.shim_any_is_few(128, 8, SMS, 3 * SMS + 1)


@pytest.mark.parametrize("nx,ny,df,f32,on", [(6, 4, 0, 1, 1), (60, 60, 0, 1, 1), (72, 54, 0, 1, 1), (72, 64, 0, 1, 0),
                                             (6, 4, 1, 0, 1), (18, 18, 1, 0, 1), (20, 20, 1, 0, 0), (30, 24, 1, 0, 0)])
def test_plane_kernels_up_to(shim, nx, ny, df, f32, on):
    """Both sides of the largest plane that takes its x and y passes in one kernel."""
    got = plane(shim, nx, ny, df, f32)
    assert got[0] == on and 128 <= got[1] <= 384
    assert not on or got[2] <= 232448 - 1024


@pytest.mark.parametrize("L,rows,groups,planes,lg", [(400, 1, 144, 1, 2), (400, 1, 608, 1, 2), (400, 1, 616, 1, 3),
                                                     (40, 1, 60, 1, 3), (400, 0, 13, 12, 2), (400, 0, 16, 39, 3)])
def test_tiles_of_four_on_idle_sms(shim, L, rows, groups, planes, lg):
    """Double-float: eight groups to a tile, four where the eights leave half of 152 SMs idle and
    a stage of them takes several rounds (not at L = 40)."""
    assert tile(shim, L, 1, 0, rows, groups, planes)["lg"] == lg


@pytest.mark.parametrize("n,f32,lg", [(810, 0, 2), (900, 0, 1), (1000, 0, 1), (1000, 1, 2)])
def test_tiles_of_two_for_long_wide_columns(shim, n, f32, lg):
    """Columns of 2 n points in the wider arithmetics: two groups where four fill an SM."""
    assert tile(shim, 2 * n, 0, f32, 0)["lg"] == lg
    assert f32 or tile(shim, 2 * n, 1, f32, 0)["lg"] == lg


@pytest.mark.parametrize("n,df,planes,on", [(18, 0, 1, 1), (30, 0, 152, 1), (30, 0, 160, 0), (30, 0, 304, 1),
                                                (36, 0, 304, 0), (20, 1, 304, 1), (20, 1, 320, 0), (24, 1, 304, 0)])
def test_plane_kernels_of_many_planes(shim, n, df, planes, on):
    """Wider arithmetics: planes up to 48 KB (FP64) and 20 KB (double-float) where their CTAs fill the
    SMs."""
    assert plane(shim, n, n, df, 0, planes)[0] == on
