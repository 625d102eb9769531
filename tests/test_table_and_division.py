"""The hashtable's probe sequence and the division by a cell width (csrc/gbees_keys.cuh),
built for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2508_13986_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2508_13986_gb300", "csrc")
SRC = r"""
#include "gbees_keys.cuh"
#include <cstdint>
using namespace gbees;
extern "C" {
uint64_t home(uint64_t k, uint64_t m) { return table_home(k, m); }
uint64_t slot_at(uint64_t h, uint64_t p, uint64_t m) { return table_slot(h, p, m); }
uint64_t next(uint64_t s, uint64_t p, uint64_t m) { return table_next(s, p, m); }
// insert n keys into table (size mask + 1, all-ones = free), then the mean
// probes of a hit and of a miss
void lengths(const uint64_t* in, long n, const uint64_t* out, long nm, uint64_t* table, uint64_t mask, double* r) {
    for (uint64_t i = 0; i <= mask; ++i) table[i] = ~0ull;
    for (long i = 0; i < n; ++i) {
        uint64_t h = table_home(in[i], mask);
        for (uint64_t p = 0; table[h] != ~0ull; ++p) h = table_next(h, p, mask);
        table[h] = in[i];
    }
    double hit = 0, miss = 0;
    for (long i = 0; i < n; ++i) {
        uint64_t h = table_home(in[i], mask), p = 0;
        for (; table[h] != in[i]; ++p) h = table_next(h, p, mask);
        hit += p + 1;
    }
    for (long i = 0; i < nm; ++i) {
        uint64_t h = table_home(out[i], mask), p = 0;
        for (; table[h] != ~0ull; ++p) h = table_next(h, p, mask);
        miss += p + 1;
    }
    r[0] = hit / n;
    r[1] = miss / nm;
}
}
"""
U = ctypes.c_uint64


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("table")
    src, so = d / "t.cpp", d / "t.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    for f in ("home", "slot_at", "next"):
        getattr(L, f).restype = U
        getattr(L, f).argtypes = [U] * (2 if f == "home" else 3)
    P = ctypes.POINTER(U)
    L.lengths.argtypes = [P, ctypes.c_long, P, ctypes.c_long, P, U, ctypes.POINTER(ctypes.c_double)]
    return L


@pytest.mark.parametrize("slots", [64, 128, 4096])
def test_sequence_visits_every_slot_once(lib, slots):
    mask = slots - 1
    for key in (0, 1, 15, 16, 2 ** 62 + 7, 2 ** 63 - 1):
        h = home = lib.home(key, mask)
        seen = []
        for p in range(slots):
            assert h == lib.slot_at(home, p, mask)
            seen.append(h)
            h = lib.next(h, p, mask)
        assert sorted(seen) == list(range(slots))


def test_neighbours_along_the_last_dimension_share_a_group(lib):
    mask = (1 << 20) - 1
    for key in (0, 16 * 12345, 2 ** 62):
        homes = [lib.home(key + i, mask) for i in range(16)]
        assert len({h >> 4 for h in homes}) == 1 and len(set(homes)) == 16


def _keys(idx):
    n, b = idx.shape[1], 63 // idx.shape[1]
    k = np.zeros(idx.shape[0], dtype=np.uint64)
    for j in range(n):
        k = (k << np.uint64(b)) | (idx[:, j].astype(np.int64) + (1 << (b - 1))).astype(np.uint64)
    return k


def _ball(n, r):
    g = np.stack([a.reshape(-1) for a in np.meshgrid(*[np.arange(-r, r + 1)] * n, indexing="ij")], axis=1)
    return g[(g ** 2).sum(1) <= r * r]


def _lattice(n, count):
    # isolated cells with period 16 along the last dimension, with their face neighbours
    idx, _ = W.random_cells(n, count, 300, seed=3)
    idx = np.unique(np.concatenate([idx[:, :-1] * 4, idx[:, -1:] * 16], axis=1), axis=0)
    out = [idx]
    for j in range(n):
        for s in (-1, 1):
            v = idx.copy()
            v[:, j] += s
            out.append(v)
    return np.unique(np.concatenate(out), axis=0)


@pytest.mark.parametrize("name", ["ball3", "ball6", "lattice3"])
def test_probe_lengths_at_half_load(lib, name):
    """The mean probes of hits and misses at load 1/2 are those of linear probing
    with a random hash (Knuth: 1.5 and 2.5). The occupied share of the cells'
    groups varies, and with it the load of a subtable's neighbourhood: the mean of
    10^4 to 10^5 keys lies within 10 % (hits) and 20 % (misses)."""
    idx = {"ball3": lambda: _ball(3, 24), "ball6": lambda: _ball(6, 4), "lattice3": lambda: _lattice(3, 6000)}[name]()
    keys = np.random.Generator(np.random.PCG64(1)).permutation(_keys(idx))
    mask = (1 << int(np.floor(np.log2(2 * keys.size)))) - 1
    n = (mask + 1) // 2
    assert n <= keys.size
    present = np.ascontiguousarray(keys[:n])
    absent = np.ascontiguousarray(_keys(idx + 1000))
    table = np.empty(mask + 1, dtype=np.uint64)
    r = (ctypes.c_double * 2)()
    P = ctypes.POINTER(U)
    lib.lengths(present.ctypes.data_as(P), present.size, absent.ctypes.data_as(P), absent.size,
                table.ctypes.data_as(P), mask, r)
    assert 1.35 <= r[0] <= 1.65 and 2.0 <= r[1] <= 3.0


def test_division_by_a_width_is_the_ieee_division(tmp_path):
    """div_round (a product with the reciprocal and two corrections) against the
    division, for widths and velocities over the range in which it is used, random
    mantissas and those at the ends of the binade."""
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(r"""
#include "gbees_keys.cuh"
#include <cstdint>
#include <cstdio>
#include <cstring>
static uint64_t s = 88172645463325252ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static double make(int e_lo, int e_hi) {
    uint64_t man = rnd() >> 12;
    switch (rnd() % 8) {
        case 0: man = rnd() % 8; break;
        case 1: man = (1ull << 52) - 1 - rnd() % 8; break;
        case 2: man &= ~0ull << (rnd() % 52); break;
    }
    const uint64_t b = (uint64_t)(1023 + e_lo + (int)(rnd() % (uint64_t)(e_hi - e_lo + 1))) << 52 | man;
    double d;
    memcpy(&d, &b, 8);
    return d;
}
int main() {
    for (long i = 0; i < 6000000; ++i) {
        const double x = i % 3 ? make(-20, 20) : make(-760, 760), h = i % 3 ? make(-10, 4) : make(-127, 127);
        volatile double want = x / h;
        if (gbees::div_round(x, h, 1.0 / h) != want) { printf("%a %a\n", x, h); return 1; }
    }
    return 0;
}
""")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True)
