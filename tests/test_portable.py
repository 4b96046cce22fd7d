"""Arithmetic of the kernels at the ends of its range (csrc/portable.cuh), compiled
for the host: indices near 2^31, of sizes that the entry points accept and that
are too large to run in a test, and scalars near the ends of the FP64 range."""
import ctypes
import glob
import math
import os
import re
import subprocess
from fractions import Fraction

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_01395_gb300", "csrc")
SOURCE = r"""
#include "portable.cuh"
using namespace pbcg;
extern "C" double gain(double alpha_rho, double inv_omega) { return beta_gain(alpha_rho, inv_omega); }
extern "C" int has_reached(unsigned counter, unsigned target) { return reached(counter, target); }
extern "C" int groups(int n, int g) { return groups_of(n, g); }
struct Dim { unsigned x; };
static Dim blockIdx, blockDim, threadIdx, gridDim;
// The first four elements of a thread of a grid of grid x block threads.
extern "C" int elements(unsigned grid, unsigned block, unsigned b, unsigned t, unsigned count, int *out) {
    gridDim.x = grid; blockDim.x = block; blockIdx.x = b; threadIdx.x = t;
    int c = 0;
    PBCG_ELEMENTS(i, count) {
        out[c++] = i;
        if (c == 4) break;
    }
    return c;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("portable")
    src, so = d / "portable.cpp", d / "portable.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(so), str(src)])
    lib = ctypes.CDLL(str(so))
    lib.gain.argtypes, lib.gain.restype = [ctypes.c_double] * 2, ctypes.c_double
    return lib


@pytest.mark.parametrize("count", [0, 1, 1000, 46340 * 46340, 2 ** 31 - 1, 2 ** 31])
@pytest.mark.parametrize("grid,block", [(608, 256), (2432, 128), (1, 32)])
def test_last_elements_of_a_thread(lib, grid, block, count):
    """A block index beyond the grid stands for a later step of a block of it."""
    out = (ctypes.c_int * 4)()
    step = grid * block
    for start in {0, 5, max(0, count - 1), max(0, count - step), max(0, count - step - 1), max(0, count - 2 * step)}:
        c = lib.elements(grid, block, start // block, start % block, ctypes.c_uint(count), out)
        expect = [i for i in range(start, start + 4 * step, step) if i < count]
        assert list(out[:c]) == expect


@pytest.mark.parametrize("g", [1, 2, 4])
@pytest.mark.parametrize("n", [0, 1, 2, 3, 4, 5, 2 ** 31 - 4, 2 ** 31 - 3, 2 ** 31 - 2, 2 ** 31 - 1])
def test_groups_of_rows(lib, n, g):
    """Groups of a system or of an x-line; their first rows stay below 2^31."""
    assert lib.groups(n, g) == -(-n // g)
    assert (lib.groups(n, g) - 1) * g < 2 ** 31


@pytest.mark.parametrize("target", [1, 152, 2 ** 31, 2 ** 32 - 1, 2 ** 32, 2 ** 32 + 151, 5 * 2 ** 32 + 7])
def test_counter_of_arrivals_past_2_32(lib, target):
    """Within the blocks of an exchange of its target, on both sides, at any lap."""
    for d in (-2040, -1, 0, 1, 2040):
        if target + d >= 0:
            assert lib.has_reached(ctypes.c_uint((target + d) % 2 ** 32), ctypes.c_uint(target % 2 ** 32)) == (d >= 0)


@pytest.mark.parametrize("rho,alpha,omega", [(3.7, 0.21, 0.7), (1.7e300, 0.3, 0.9), (1.3 * 2.0 ** 1021, 0.3, 0.01),
                                             (1.7e300, 1.3e-12, 1e-6), (1.1e-300, 7e9, 1.7e-290),
                                             (1.3e-5, 1.7 * 2.0 ** 40, 1.3 * 2.0 ** 1023), (1.0, 1e-200, 1e200)])
def test_beta_by_one_product_is_as_exact_as_its_factors(lib, rho, alpha, omega):
    """alpha, rho and omega stand for values known exactly. Four roundings of 2^-53 (two
    quotients, two products) where the short form is used; 0 asks for the long one."""
    g = lib.gain(alpha / rho, 1.0 / omega)
    rho_next = 0.77 * rho
    exact = Fraction(alpha) / Fraction(rho) / Fraction(omega) * Fraction(rho_next)
    if g != 0.0:
        assert abs(Fraction(g * rho_next) - exact) <= 4.5 * exact / 2 ** 53
    else:
        assert any(not 2.0 ** -1022 <= v < math.inf for v in (alpha / rho, 1.0 / omega, alpha / rho * (1.0 / omega)))


def test_kernels_step_through_elements_by_this_loop():
    """No kernel adds the threads of the grid to a signed 32-bit index of its own."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        if not path.endswith("portable.cuh"):
            assert not re.search(r"\+=\s*(gridDim\.x|stride)\b", text), path
