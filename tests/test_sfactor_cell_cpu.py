"""The grid cell and weights of the structure factor's deposit, compiled for the host: every
value of a coordinate (positions that were refused stay stored) lands on the grid, and the
cell is the remainder by G of the coordinate's floor."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1808_06381_gb300", "csrc")
UNIT = 2.0 ** 50

SOURCE = """
#include "sfactor_cell.cuh"
extern "C" void cell(double v, int G, int* i, unsigned long long* f)
{
    const ss::GridCell c = ss::grid_cell(v, G);
    i[0] = c.i0, i[1] = c.i1, f[0] = c.f, f[1] = c.g;
}
extern "C" unsigned long long weight(unsigned long long a, unsigned long long b) { return ss::cell_weight(a, b); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cell")
    (d / "cell.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "cell.cpp"), "-o", str(d / "cell.so")],
                   check=True)
    so = ctypes.CDLL(str(d / "cell.so"))
    so.cell.argtypes = [ctypes.c_double, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    so.weight.argtypes = [ctypes.c_uint64, ctypes.c_uint64]
    so.weight.restype = ctypes.c_uint64
    return so


def _cell(lib, u, G):
    i, f = (ctypes.c_int * 2)(), (ctypes.c_uint64 * 2)()
    lib.cell(u * UNIT, G, i, f)
    return i[0], i[1], f[0], f[1]


@pytest.mark.parametrize("G", [8, 9, 256, 1500, 8192])
def test_every_value_lands_on_the_grid(lib, G):
    rng = np.random.Generator(np.random.PCG64(G))
    values = [0.0, -0.0, 0.5, G - 0.25, np.nextafter(G, 0.0), float(G), G + 0.75, 2.0 * G, -0.25, -G, -G - 0.5, -1e-300,
              -3.5 * G, 17.25 * G, 8191.5, 8192.0, -8192.0, -8192.5, 1e6 + 0.5, -1e6 - 0.5, 1e15, -1e15, 1e18, 1e290, -1e290]
    values += list(rng.uniform(-G, G, 200)) + list(rng.uniform(-50.0 * G, 50.0 * G, 50))
    for u in values:
        i0, i1, f, g = _cell(lib, u, G)
        assert 0 <= i0 < G and i1 == (i0 + 1) % G and f + g == 1 << 63, u
        if abs(u) < 8192:
            want = math.floor(Fraction(u))
            assert i0 == want % G, u
            assert 0 <= Fraction(u) - want - Fraction(f, 1 << 63) < Fraction(1, 1 << 50), u
        else:
            assert i0 == math.floor(u) % G, u
    for u in (math.inf, -math.inf, math.nan):
        assert _cell(lib, u, G) == (0, 1, 0, 1 << 63)


def test_weights_are_the_rounded_products(lib):
    rng = np.random.Generator(np.random.PCG64(1))
    for _ in range(200):
        a, b = (int(x) << 13 for x in rng.integers(0, (1 << 50) + 1, 2))
        assert abs(Fraction(lib.weight(a, b)) - Fraction(a * b, 1 << 94)) <= Fraction(1, 2) + Fraction(1, 1 << 30)
    one = 1 << 63
    assert lib.weight(one, one) == 1 << 32 and lib.weight(one, 0) == 0
