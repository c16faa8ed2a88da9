"""Columns of the strip-and-band sweep, for every width and thread (the library's own functions, compiled for the
host): X-pass rows pass from lane to lane of a warp without a barrier, so a thread may only read a column of its
own warp, and the threads whose values reach an output (three columns on either side of the strip's) have to
find the image column that they stand for."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def columns(tmp_path_factory):
    d = tmp_path_factory.mktemp("columns")
    src = d / "columns.cpp"
    src.write_text(f'#include "{ROOT}/paper_1907_05993_gb300/csrc/demons_wide_columns.cuh"\n'
                   'extern "C" int strip(int x0, int x1, int w, int nt, int *col)\n'
                   '{ int xl = strip_origin(x0, x1, w); for (int t = 0; t < nt; ++t) col[t] = edge_column(xl, t, w); return xl; }\n')
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-x", "c++", str(src), "-o", str(d / "columns.so")], check=True)
    return C.CDLL(str(d / "columns.so")).strip


@pytest.mark.parametrize("nt", [128, 256])
def test_columns_of_every_strip(columns, nt):
    col = np.empty(nt, np.int32)
    t = np.arange(nt)
    for w in range(8, 1400):
        strips = -(-w // (nt - 15))
        sw = -(-w // strips)
        if w - (strips - 1) * sw < 6:   # not taken by the plan
            continue
        for s in range(strips):
            x0, x1 = s * sw, min(w, (s + 1) * sw)
            xl = columns(x0, x1, w, nt, col.ctypes.data_as(C.POINTER(C.c_int)))
            assert (col // 32 == t // 32).all(), (w, s)
            assert xl <= x0 - 6 and xl + nt >= x1 + 6
            x = xl + t
            need = (x >= x0 - 3) & (x < x1 + 3)   # du there enters an output's y pass of G_u's x-passed rows
            assert (xl + col[need] == np.clip(x[need], 0, w - 1)).all(), (w, s)
