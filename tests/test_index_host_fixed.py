"""Shared-memory layouts of the block fixed-point rows, of float rows with an odd part and of the twiddle tables,
compiled for the host: every slot is in range and used once at every length the planner can choose, and the offsets that
the Stockham passes take in place of the layout function are the function's.  No GPU is used."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
POW2 = [1 << k for k in range(13)]
ODD = [80, 96, 160, 192, 200, 320, 384, 400, 640, 768, 800]


@pytest.fixture(scope="module")
def lib():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    so = os.path.join(tempfile.mkdtemp(), "idxfx.so")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC",
                    "-gencode", "arch=compute_103a,code=sm_103a",
                    os.path.join(HERE, "index_host_fixed_harness.cu"), "-o", so], check=True)
    return ctypes.CDLL(so)


def passes(L):
    """(radix, product of the radices before it) of a row's passes."""
    pow2 = L & -L
    log, odd = pow2.bit_length() - 1, L // pow2
    radices = ([2] if log % 3 == 1 else [4] if log % 3 == 2 else []) + [8] * (log // 3)
    radices += {1: [], 3: [3], 5: [5], 25: [5, 5]}[odd]
    out, ns = [], 1
    for r in radices:
        out.append((r, ns))
        ns *= r
    assert ns == L
    return out


@pytest.mark.parametrize("L", POW2 + ODD)
def test_fixed_point_rows(lib, L):
    pos = [lib.h_spos_fx(i) for i in range(L)]
    assert len(set(pos)) == L and min(pos) >= 0 and max(pos) < lib.h_row_stride_fx(L)
    if L < 8:
        return
    for R, Ns in passes(L):
        LR = L // R
        for b in range(LR):
            k = b % Ns if R in (2, 4, 8) else (b if Ns == LR else b & (Ns - 1))
            i0 = (b - k) * R + k
            for r in range(R):
                assert b + r * LR < L and i0 + r * Ns < L
                if LR % 64 == 0:
                    assert pos[b] + r * LR == pos[b + r * LR]
                if Ns % 64 == 0:
                    assert pos[i0] + r * Ns == pos[i0 + r * Ns]


@pytest.mark.parametrize("L", ODD)
def test_float_rows_with_an_odd_part(lib, L):
    pos = [lib.h_pidx(i) for i in range(L)]
    assert [lib.h_rpos_float(L, i) for i in range(L)] == pos
    assert len(set(pos)) == L and max(pos) < lib.h_row_stride(L, 8)
    for R, Ns in passes(L):
        LR = L // R
        for b in range(LR):
            k = b & (Ns - 1) if Ns & (Ns - 1) == 0 else b    # a power of two, or the last pass of 25
            assert Ns & (Ns - 1) == 0 or Ns == LR
            i0 = (b - k) * R + k
            for r in range(R):
                if LR % 8 == 0:
                    assert pos[b] + r * (LR + LR // 8) == pos[b + r * LR]
                if Ns % 8 == 0:
                    assert pos[i0] + r * (Ns + Ns // 8) == pos[i0 + r * Ns]


@pytest.mark.parametrize("which", ["fx", "float"])
@pytest.mark.parametrize("L", POW2 + ODD)
def test_twiddle_tables(lib, L, which):
    f = getattr(lib, "h_tpos_" + which)
    # a row's own table (y and z), and the x kernels' table of twice the row's length
    for n in (L, 2 * L):
        pos = [f(t, L) for t in range(n)]
        assert len(set(pos)) == n and min(pos) >= 0 and max(pos) < lib.h_tw_slots(n)
        if n & (n - 1) == 0 or n >= 16 and n % 16 == 0:
            assert max(pos) < n       # the x and film kernels hold n slots


def test_every_odd_length_is_compiled_where_it_is_used(lib):
    for P in (512, 1024):
        for num in (5, 6):
            L = P // 8 * num
            assert lib.h_compiled(L // 2, 0) == L // 2 and lib.h_compiled(L, 1) == L
    for P in (128, 256, 512, 1024):
        for num, den in ((5, 8), (3, 4), (25, 32)):
            L = P // den * num
            if L % 8 == 0:
                assert lib.h_compiled(L, 2) == L
