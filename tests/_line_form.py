"""The step's choice of line solver and its restart distance, from the host
headers of the library (line_tables.h, line_rule.h) through the host compiler."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "line_tables.h"
#include "line_rule.h"
using namespace chg;
template <typename T>
static MarchFactors fac(double ck) { return march_factors<T>(ck, kMarchMaxReach, std::ldexp(1.0, sizeof(T) == 8 ? -64 : -36)); }
extern "C" void factors(int fp64, double ck, double* out) {
    const MarchFactors f = fp64 ? fac<double>(ck) : fac<float>(ck);
    out[0] = f.l1; out[1] = f.l2; out[2] = f.dinv; out[3] = f.reach;
}
template <typename T>
static int query(const LineBox& b, double* us) {
    us[0] = scan_us<T>(b);
    const bool fits[5] = {true, sizeof(T) == 4 && tile_fits<T, 16>(b), tile_fits<T, 32>(b), sizeof(T) == 8 && tile_fits<T, 64>(b), march_fits<T>(b)};
    for (int f = 1; f < 5; ++f) us[f] = fits[f] ? march_us<T>(b, (LineForm)f) : -1.0;
    return choose_line_form<T>(b);
}
extern "C" int form(int fp64, int periodic, int dir, long nx, long ny, long nz, int reach, double* us) {
    const LineBox b{{nx, ny, nz}, dir, periodic != 0, reach, false};
    return fp64 ? query<double>(b, us) : query<float>(b, us);
}
"""
# (nz, ny, nx), precision and ck of boxes that take every form
BOXES = [((33, 33, 33), "f32", 0.02), ((33, 33, 36), "f32", 0.02), ((33, 65, 36), "f32", 0.02), ((36, 33, 257), "f32", 0.02),
         ((40, 34, 260), "f32", 0.02), ((400, 36, 36), "f32", 0.02), ((300, 33, 33), "f32", 0.25), ((33, 300, 33), "f32", 0.25),
         ((33, 300, 36), "f32", 0.25), ((64, 64, 301), "f32", 0.25), ((72, 66, 300), "f32", 0.25),
         ((40, 33, 33), "f64", 0.02), ((40, 33, 34), "f64", 0.02), ((64, 33, 33), "f64", 0.02), ((70, 500, 33), "f64", 0.02),
         ((70, 500, 36), "f64", 0.02), ((500, 40, 129), "f64", 0.02), ((500, 97, 65), "f64", 0.02), ((500, 97, 65), "f64", 3.0),
         ((96, 72, 72), "f64", 1.2), ((72, 97, 97), "f64", 1.2), ((70, 160, 33), "f64", 1.2), ((98, 100, 520), "f64", 0.25),
         ((98, 100, 517), "f64", 0.25),
         # lines as short as their restart
         ((200, 200, 8), "f32", 1e-4), ((128, 8, 33), "f32", 1e-4), ((8, 32, 32), "f32", 1e-4), ((128, 32, 16), "f64", 1e-4),
         ((128, 16, 32), "f64", 1e-4), ((16, 128, 32), "f64", 1e-4)]
NAMES = ("scan", "tile16", "tile32", "tile64", "march")
_lib = None


def lib():
    """The compiled headers, or None without a host compiler."""
    global _lib
    cxx = shutil.which("g++") or shutil.which("c++")
    if _lib is None and cxx:
        with tempfile.TemporaryDirectory() as d:
            src, so = os.path.join(d, "f.cpp"), os.path.join(d, "f.so")
            with open(src, "w") as f:
                f.write(SRC)
            subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I",
                            os.path.join(ROOT, "paper_2105_01865_gb300", "csrc"), src, "-o", so], check=True)
            _lib = ctypes.CDLL(so)
        _lib.factors.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_void_p]
        _lib.form.argtypes = [ctypes.c_int] * 3 + [ctypes.c_long] * 3 + [ctypes.c_int, ctypes.c_void_p]
    return _lib


def factors(prec, ck):
    """l1, l2, 1/u0 and the restart distance in rows."""
    out = np.empty(4)
    lib().factors(int(prec == "f64"), ck, out.ctypes.data)
    return out[0], out[1], out[2], int(out[3])


def form(prec, periodic, d, shape, reach):
    """(form taken, estimated us of each form that takes the lines) along direction d of a (nz, ny, nx) box."""
    us = np.empty(5)
    f = lib().form(int(prec == "f64"), int(periodic), d, shape[2], shape[1], shape[0], reach, us.ctypes.data)
    return NAMES[f], {n: t for n, t in zip(NAMES, us) if t >= 0}


def forms(prec, bc, shape, ck):
    """The forms of the x-, y- and z-solves of a substep with the operator I + ck [1, -4, 6, -4, 1]."""
    reach = factors(prec, ck)[3]
    return tuple(form(prec, bc[d] == 0, d, shape, reach)[0] for d in range(3))
