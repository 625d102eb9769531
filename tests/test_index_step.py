"""One step of a cell index (csrc/gbees_keys.cuh, step_index), built for the host: every
neighbour that has a key is found, and in one dimension, where an index takes all 32
bits, the last index has no neighbour beyond it (a wrapped one would have a key)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2508_13986_gb300", "csrc")
SRC = r"""
#include "gbees_keys.cuh"
template <int N>
static int step(int* I, int j, int up, int b) {
    unsigned long long k;
    return gbees::step_index<N>(I, j, up) && gbees::pack_key_bits<N>(b, I, k);
}
extern "C" int step1(int* I, int j, int up) { return step<1>(I, j, up, 32); }
extern "C" int step2(int* I, int j, int up) { return step<2>(I, j, up, 31); }
extern "C" int step6(int* I, int j, int up) { return step<6>(I, j, up, 10); }
"""


@pytest.mark.parametrize("n,bits", [(1, 32), (2, 31), (6, 10)])
def test_a_step_beyond_the_last_key_has_none(tmp_path, n, bits):
    src, so = tmp_path / "s.cpp", tmp_path / "s.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fwrapv", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)],
                   check=True)
    f = getattr(ctypes.CDLL(str(so)), f"step{n}")
    top, low = 2 ** (bits - 1) - 1, -2 ** (bits - 1)
    for j in range(n):
        for start, up, want in ((top, 1, False), (top - 1, 1, True), (low, 0, False), (low + 1, 0, True),
                                (top, 0, True), (low, 1, True), (0, 1, True), (0, 0, True)):
            I = np.zeros(n, dtype=np.int32)
            I[j] = start
            assert bool(f(I.ctypes.data_as(ctypes.POINTER(ctypes.c_int)), j, up)) == want, (j, start, up)
            if want:
                assert I[j] == start + (1 if up else -1)
