"""The fixed-point functions of the FP64 kernels (csrc/ffrg_fx.cuh) on the CPU, where the header compiles as
plain C++, against 40-digit values: table coordinate of a log grid, regulator h(x) = x/(1 - e^{-x}), reciprocal.

Bounds: the results are rounded to a double (half an ulp, 2^-53 relative); fx_h's polynomial adds its coefficient
rounding (below 2^-55).  The coordinate is kept in units of at least 2^-53 of the coordinate per octave of y: u_scale
rounded to half a unit counts |log2 y| times, the offset, the table entry and the polynomial (three truncated
products) once each: (|log2 y|/2 + 5) 2^-53 octaves, plus the rounding of the weight to a double in [1, 2)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")
mpmath.mp.dps = 40
HERE = os.path.dirname(os.path.abspath(__file__))
SRC = r"""
#include "ffrg_fx.cuh"
using namespace ffrg;
static FxTables T;
extern "C" {
void init() { fx_build_tables(&T); }
double h(double x) { return fx_h(T, x); }
double flat(double x) { return fx_h_flat(x); }
double rcp(double x) { return fx_rcp(x); }
int grid(int n, double lo, double hi, FxGrid *g) { return fx_grid(n, lo, hi, g); }
int node(const FxGrid *g, double y, double *w1) {
  static FxLogEntry L[kFxLog];
  for (int j = 0; j < kFxLog; ++j) L[j] = fx_scaled(T.log[j], *g);
  int i;
  fx_node(*g, fx_log(L, *g, y) + g->uo, i, *w1);
  return i;
}
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(SRC)
    inc = os.path.join(HERE, "..", "paper_2412_13043_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", inc, str(d / "fx.cpp"), "-o", str(d / "fx.so")], check=True)
    lib = ctypes.CDLL(str(d / "fx.so"))
    for f in (lib.h, lib.rcp, lib.flat):
        f.restype, f.argtypes = ctypes.c_double, [ctypes.c_double]
    lib.grid.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_void_p]
    lib.node.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_void_p]
    lib.init()
    return lib


def _samples(lo, hi, n, seed):
    r = np.random.RandomState(seed)
    v = list(np.exp(r.uniform(np.log(lo), np.log(hi), n)))
    for e in range(int(np.log2(lo)) + 1, int(np.log2(hi))):   # both sides of the cell and octave edges
        v += [2.0 ** e, np.nextafter(2.0 ** e, 0), np.nextafter(2.0 ** e, np.inf), 2.0 ** e * (1 + 37 / 128)]
    return v


def test_regulator(fx):
    for x in _samples(1e-20, 1e4, 4000, 1) + list(np.arange(1, 128) / 128):
        ref = mpmath.mpf(x) / -mpmath.expm1(-mpmath.mpf(x))
        assert abs(fx.h(x) / ref - 1) < 1.5 * 2.0 ** -53, x
    for x in (0.0, -0.0, -1e-18, -1e-300, 5e-324):   # rounding of |q + p|^2 around 0
        assert fx.h(x) == 1.0
        assert fx.flat(x) == 1.0
    for f in (fx.h, fx.flat):
        assert f(float("inf")) == float("inf") and np.isnan(f(float("nan"))) and np.isnan(f(-float("nan")))
    for x in (0.3, np.nextafter(1, 0), 1.0, np.nextafter(1, 2), 700.0):
        assert fx.flat(x) == max(1.0, x)


def test_reciprocal(fx):
    for d in _samples(1e-300, 1e300, 4000, 2) + _samples(0.5, 4.0, 2000, 3):
        for s in (d, -d):
            assert abs(mpmath.mpf(fx.rcp(s)) * mpmath.mpf(s) - 1) < 1.02 * 2.0 ** -53, s
    for d in (0.0, -0.0, float("inf"), float("-inf"), 5e-324, 1e-309, 1.7e308):
        with np.errstate(divide="ignore", over="ignore"):
            assert fx.rcp(d) == np.float64(1.0) / np.float64(d)
    assert np.isnan(fx.rcp(float("nan")))


@pytest.mark.parametrize("n,lo,hi", [(2, 1e-3, 10.0), (3, 0.4, 0.9), (64, 1e-3, 10.0), (97, 1e-6, 1e3), (128, 1e-3, 10.0),
                                     (4096, 1e-3, 10.0)])
def test_coordinate(fx, n, lo, hi):
    g, w1 = ctypes.create_string_buffer(256), ctypes.c_double()
    assert fx.grid(n, lo, hi, g)
    scale = (n - 1) / mpmath.log(mpmath.mpf(hi) / mpmath.mpf(lo))
    for s in np.exp(np.random.RandomState(n).uniform(np.log(lo), np.log(hi), 300)):
        y = s * s
        u = scale * (mpmath.log(mpmath.mpf(y)) / 2 - mpmath.log(mpmath.mpf(lo)))
        if not 0 < u < n - 1:
            continue
        i = fx.node(g, y, ctypes.byref(w1))
        bound = (abs(np.log2(y)) / 2 + 5) * 2.0 ** -53 * float(mpmath.log(2) * scale / 2) + 2.0 ** -52
        assert abs(i + mpmath.mpf(w1.value) - 1 - u) < bound, (s, u)
    for y, want in ((0.0, 0), (-1e-20, 0), (lo * lo / 2, 0), (hi * hi * 2, n - 1), (float("inf"), n - 1)):
        assert fx.node(g, y, ctypes.byref(w1)) == want
        assert want or w1.value == 1.0


def test_grids_outside_fixed_point_are_refused(fx):
    g = ctypes.create_string_buffer(256)
    for n, lo, hi in ((64, 1e-20, 1.0), (64, 1e-3, 1e20), (2, 1.0, 1.0 + 1e-15)):
        assert not fx.grid(n, lo, hi, g)


@pytest.mark.parametrize("n,lo,hi", [(128, 1.0, 1.0 + 1e-9), (4096, 1.0, 1.000001), (4096, 1.0, 1.00001),
                                     (4096, 1.0, 1.0001), (4096, 1.0, 1.001), (4096, 1e-3, 1.001e-3), (64, 1.0, 1.000001),
                                     (64, 1.0, 1.0001), (2, 1.0, 1.0 + 1e-7), (4096, 2.0 ** 49, 2.0 ** 49.001)])
def test_nodes_of_narrow_grids_stay_in_the_row(fx, n, lo, hi):
    """Momenta far outside a narrow grid: the first or the last node, whatever their distance in nodes.  (A grid may
    be refused: the kernels then take the FP64 logarithm.)"""
    g, w1 = ctypes.create_string_buffer(256), ctypes.c_double()
    if not fx.grid(n, lo, hi, g):
        return
    for y in list(2.0 ** np.arange(-250.0, 251.0)) + [16.0, 4.0, 1e6, 1e30, 1e300, float("inf"), float("nan")]:
        assert fx.node(g, y, ctypes.byref(w1)) == (0 if y <= lo * lo else n - 1), y   # lo itself: the first node
    for y in (0.0, -0.0, -1.0, 5e-324):
        assert fx.node(g, y, ctypes.byref(w1)) == 0


def test_ordinary_grids_take_fixed_point(fx):
    g = ctypes.create_string_buffer(256)
    for n, lo, hi in ((4096, 1.0, 1.01), (4096, 1e-3, 10.0), (2, 0.999, 1.001), (256, 0.5, 0.6), (64, 1e-12, 1e12)):
        assert fx.grid(n, lo, hi, g)
