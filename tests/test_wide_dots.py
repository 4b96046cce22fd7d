"""The fixed-point dot products of the FP64 sweeps (csrc/dots.cuh), compiled for
the host and compared with exact rational sums.

A term is formed with an error of at most 3 units and truncated by less than
one unit of 2^-(60 - 6) = 2^-54 of the largest product met; a move of the
reference drops less than one unit, at most once a term; the result is rounded
to 53 bits. So the error of a sum of n terms is at most
5 n 2^-54 max|a b| + 2^-53 |sum|. The sums of a warp's lanes, which share their
first reference, are held to what their code keeps (test of a warp).
"""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_01395_gb300", "csrc")
SOURCE = r"""
#include <algorithm>
#include <vector>
#include "dots.cuh"
using namespace pbcg;
template <class P> static void run(int n, const double *v, double *out) {
    WideSlot slots[P::np];
    WideDots<P> d(slots, 1, n > 0);
    for (int i = 0; i < n; ++i) {
        double r[P::nv];
        for (int j = 0; j < P::nv; ++j) r[j] = v[i * P::nv + j];
        d.add(r);
    }
    double o[P::np];
    d.values(n > 0, o);
    for (int k = 0; k < P::np; ++k) out[k] = o[k];
}
// One warp: lane l has the rows l, l + 32, ...; the first references are common, as in a kernel.
extern "C" void warp_one(int rows, const double *v, double *out) {
    using D = WideDots<PairsOne>;
    std::vector<WideSlot> slots(32);
    std::vector<D> lanes;
    int top = 0;
    for (int l = 0; l < 32; ++l) {
        lanes.emplace_back(&slots[l], 1, 1);
        double r[2] = {v[2 * l], v[2 * l + 1]};
        WideParts p[2] = {wide_parts(r[0]), wide_parts(r[1])};
        D probe(nullptr, 1, 1);
        probe.unusual(r, p, p[0].e > p[1].e ? p[0].e : p[1].e);
        top = std::max(top, D::product_exponent(p, 0));
    }
    for (int l = 0; l < 32; ++l) {
        lanes[l].begin(0, top);
        lanes[l].lanes = 0u;
    }
    for (int i = 0; i < rows * 32; ++i) lanes[i % 32].add({v[2 * i], v[2 * i + 1]});
    for (int l = 0; l < 32; ++l) {
        double o[1];
        lanes[l].values(true, o);
        out[l] = o[0];
    }
}
extern "C" void pipe_a(int n, const double *v, double *o) { run<PairsPipeA>(n, v, o); }
extern "C" void pipe_b(int n, const double *v, double *o) { run<PairsPipeB>(n, v, o); }
extern "C" void one(int n, const double *v, double *o) { run<PairsOne>(n, v, o); }
extern "C" void omega(int n, const double *v, double *o) { run<PairsOmega>(n, v, o); }
extern "C" void rho(int n, const double *v, double *o) { run<PairsRho>(n, v, o); }
"""
PAIRS = {"pipe_a": (5, [(0, 1), (1, 1), (0, 0), (2, 3), (2, 4)]), "pipe_b": (3, [(0, 1), (0, 2), (1, 1)]),
         "one": (2, [(0, 1)]), "omega": (2, [(0, 1), (1, 1), (0, 0)]), "rho": (2, [(0, 1), (1, 1)])}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("wide")
    src, so = d / "wide.cpp", d / "wide.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-shared", "-fPIC", "-I", CSRC,
                           "-o", str(so), str(src)])
    return ctypes.CDLL(str(so))


def sums(lib, name, v):
    v = np.ascontiguousarray(v, dtype=np.float64)
    out = np.empty(len(PAIRS[name][1]))
    getattr(lib, name)(len(v), v.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p))
    return out


def rows(kind, n, nv):
    g = np.random.default_rng(n * 7 + len(kind))
    v = g.standard_normal((n, nv))
    if kind == "lognormal":      # products over more than 64 binades
        v *= np.exp(6.0 * g.standard_normal((n, nv)))
    if kind == "sparse":         # zeros and signed zeros among the values
        v *= g.random((n, nv)) < 0.5
    if kind == "rising":         # every row above the reference of the rows before it
        v *= 2.0 ** (9.0 * np.arange(n)[:, None] % 450)
    if kind == "tiny":           # products at the bottom of the normal range
        v *= 1e-153
    if kind == "huge":           # products near the top of the range
        v *= 1e150
    return v


@pytest.mark.parametrize("name", list(PAIRS))
@pytest.mark.parametrize("kind", ["normal", "lognormal", "sparse", "rising", "tiny", "huge"])
@pytest.mark.parametrize("n", [1, 2, 3, 64, 500])
def test_error_bound_against_rational_sums(lib, name, kind, n):
    nv, pairs = PAIRS[name]
    v = rows(kind, n, nv)
    got = sums(lib, name, v)
    for k, (a, b) in enumerate(pairs):
        p = [Fraction(float(x)) * Fraction(float(y)) for x, y in zip(v[:, a], v[:, b])]
        exact = sum(p)
        bound = 5 * n * Fraction(1, 2 ** 54) * max(map(abs, p)) + Fraction(1, 2 ** 53) * abs(exact)
        bound += Fraction(1, 2 ** 1074)   # a result below the normal range
        assert abs(Fraction(float(got[k])) - exact) <= bound, (name, kind, n, k)


def test_exact_cancellation_and_small_integers(lib):
    v = np.array([[3.0, 5.0], [-3.0, 5.0], [2.0, 1.0], [-1.0, 2.0]])
    assert sums(lib, "one", v)[0] == 0.0
    g = np.random.default_rng(1)
    v = g.integers(-1000, 1000, (200, 2)).astype(float)
    assert sums(lib, "one", v)[0] == float(np.dot(v[:, 0].astype(np.int64), v[:, 1].astype(np.int64)))


def test_no_rows_zero_rows_and_non_finite_values(lib):
    assert not sums(lib, "pipe_a", np.empty((0, 5))).any()
    assert not sums(lib, "pipe_a", np.zeros((7, 5))).any()
    inf, nan = math.inf, math.nan
    one = lambda *r: sums(lib, "one", np.array(r))[0]   # noqa: E731
    assert one([1.0, 2.0], [inf, 3.0], [1.0, 1.0]) == inf
    assert one([inf, -3.0], [1.0, 1.0]) == -inf
    assert math.isnan(one([inf, 3.0], [-inf, 3.0]))
    assert math.isnan(one([inf, 0.0], [1.0, 1.0]))
    assert math.isnan(one([1.0, nan], [1.0, 1.0]))
    assert one([1e200, 1e200], [1.0, 1.0]) == inf   # a sum above the range
    b = sums(lib, "pipe_b", np.array([[1.0, 2.0, 3.0], [1.0, 4.0, nan]]))   # r0, r, w: only (r0, w) meets the NaN
    assert b[0] == 6.0 and math.isnan(b[1]) and b[2] == 20.0


def exact_products(v):
    """The products of each pair as whole numbers and the exponent of 2 they share."""
    m, e = np.frexp(v)
    m = (m * 2.0 ** 53).astype(np.int64)
    e = e.sum(axis=1) - 106
    low = int(e.min())
    return [int(a) * int(b) << int(x) - low for (a, b), x in zip(m, e)], low


@pytest.mark.parametrize("square", [True, False])
@pytest.mark.parametrize("outlier", [1.0, 1e2, 1e4, 1e6, 1e12])
@pytest.mark.parametrize("rows", [1, 107, 3000])
def test_lanes_of_a_warp_with_one_outlier(lib, rows, outlier, square):
    """Lanes share the reference of the warp's first rows. A term loses one unit of the
    sum at the addition and one at most at moves, each at most 2^-73 of the warp's largest
    product, and 3 * 2^-60 of itself; a lane's sum is rounded to 53 bits."""
    g = np.random.default_rng(rows)
    v = g.standard_normal((32 * rows, 2))
    v[5] *= outlier
    if square:
        v[:, 1] = v[:, 0]
    v = np.ascontiguousarray(v)
    out = np.empty(32)
    lib.warp_one(rows, v.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p))
    p, low = exact_products(v)
    scale = Fraction(2) ** low
    lane = [sum(p[k::32]) * scale for k in range(32)]
    bound = 2 * len(p) * max(map(abs, p)) * scale / 2 ** 73 + 3 * sum(map(abs, p)) * scale / 2 ** 60
    bound += sum(map(abs, lane)) / 2 ** 53
    assert abs(sum(Fraction(float(o)) for o in out) - sum(lane)) <= bound


@pytest.mark.parametrize("small", [3e-309, 1e-315, 4e-323])
@pytest.mark.parametrize("n", [1, 3, 200])
def test_subnormal_values(lib, n, small):
    """A subnormal value keeps its bits next to one that brings the product into range;
    bound of the sums above."""
    g = np.random.default_rng(n)
    v = g.standard_normal((n, 2)) * [small, 1e300]
    v[n // 2, 0] = np.sign(v[n // 2, 0]) * 5e-324
    p = [Fraction(float(x)) * Fraction(float(y)) for x, y in v]
    exact = sum(p)
    bound = 5 * n * Fraction(1, 2 ** 54) * max(map(abs, p)) + Fraction(1, 2 ** 53) * abs(exact)
    assert abs(Fraction(float(sums(lib, "one", v)[0])) - exact) <= bound
