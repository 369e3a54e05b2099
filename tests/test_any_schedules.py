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
