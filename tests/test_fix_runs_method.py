"""The integer differences and filters over runs of four (fix64.cuh), compiled for the host, against
exact rational arithmetic: smooth fields, fields that cross zero, steps and decays of up to a hundred
decades. A run is either refused (it then takes binary64) or at least as good as binary64, output by
output: the bound is one final rounding and a part of one unit in the last place (2^-53) of the
largest input of the output's own window.

Tenth difference over 1024: inputs and sum are within 2 units of 2^-62 of the run's power of two,
which a window passes by at most 2^7: 2^-54 of the window's largest input.
Gaussian filter: 11 units of 2^-62 (five products, each up to 1.5 short, the inputs' truncation and
the weights' rounding) against outputs of at least 2^-5: 2^-53.5 of the output.
Fourth differences: sixteen (the sum of the weights) units of 2^-59 against windows of at least 2^-5:
2^-50 of the largest of their five inputs, where binary64's four roundings reach 2^-50.4 on smooth
fields and 2^-48 on rough ones."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2210_05547_gb300", "csrc")
SHIM = """
#include "fix64.cuh"
using namespace hyp;
extern "C" int tenth(const double* p, double* out) {
    double x[RUN + 10], y[RUN];
    for (int k = 0; k < RUN + 10; ++k) x[k] = p[k];
    const bool ok = tenth_run(x, y);
    for (int k = 0; k < RUN; ++k) out[k] = y[k];
    return ok;
}
extern "C" int gauss(const double* p, double* out) {
    double x[RUN + 8], y[RUN];
    for (int k = 0; k < RUN + 8; ++k) x[k] = p[k];
    const int plain = gauss_fixed(x, y);
    for (int k = 0; k < RUN; ++k) out[k] = y[k];
    return plain;
}
extern "C" int fourth(const double* p, double* out) {
    double w[RUN + 4], r[4][RUN], dx[RUN], dy[RUN];
    for (int k = 0; k < RUN + 4; ++k) w[k] = p[2 * (RUN + 4) + k];
    for (int q = 0; q < 4; ++q)
        for (int k = 0; k < RUN; ++k) r[q][k] = p[(q + (q > 1)) * (RUN + 4) + k + 2];
    const double x[2] = {1, 0}, y[2] = {0, 1};
    const bool ok = fourth_run(w, r, x, dx) && fourth_run(w, r, y, dy);
    for (int k = 0; k < RUN; ++k) out[k] = dx[k], out[RUN + k] = dy[k];
    return ok;
}
"""
EPS = Fr(2) ** -53
GAUSS = [Fr(107, 103680), Fr(149, 12960), Fr(1997, 25920), Fr(3091, 12960), Fr(3565, 10368)]
GAUSS += GAUSS[-2::-1]
TENTH = [-1, 10, -45, 120, -210, 252, -210, 120, -45, 10, -1]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("runs")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run([gxx, "-O1", "-w", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _fields():
    s = np.arange(403.0)
    rng = np.random.default_rng(3)
    return {
        "smooth": 1 + 0.3 * np.sin(s / 20) + 0.1 * np.sin(s / 7),
        "binade": 1 + 0.02 * np.sin(s / 9),
        "zero": np.sin(s / 15),
        "noise": 1 + 1e-3 * rng.standard_normal(s.size),
        "step": 1e-9 + 0.5 * (1 + np.tanh((s - 200) / 2)),
        "spike": np.where(np.arange(403) % 37 == 5, 1.0, 1e-11),
        "decay": 10.0 ** (-100 * s / s.size),
        "top": np.where(rng.random(s.size) < 0.5, -1.0, 1.0) * np.nextafter(2.0, 1),
        "none": 0.0 * s,
        "small": 1e-280 * np.cos(s / 11),
    }


def _call(fn, x, n):
    x = np.ascontiguousarray(x)
    out = np.zeros(n)
    ok = fn(x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p))
    return ok, out


@pytest.mark.parametrize("name", _fields().keys())
def test_tenth_difference(lib, name):
    f = _fields()[name]
    taken = 0
    for a in range(0, f.size - 13):
        ok, got = _call(lib.tenth, f[a:a + 14], 4)
        if not ok:
            continue
        taken += 1
        for o in range(4):
            w = f[a + o:a + o + 11]
            exact = sum(Fr(float(v)) * c for v, c in zip(w, TENTH)) / 1024
            floor = Fr(2) ** -1022                       # below it results are rounded to it
            bound = abs(exact) * Fr(2) ** -53 + Fr(float(np.abs(w).max())) * Fr(2) ** -54 + floor
            assert abs(Fr(float(got[o])) - exact) <= bound, (a, o)
    assert taken == f.size - 13 or name in ("step", "spike", "decay")
    assert taken > f.size // 4


@pytest.mark.parametrize("name", _fields().keys())
def test_gaussian_filter(lib, name):
    f = _fields()[name]
    taken = 0
    for a in range(0, f.size - 11):
        plain, got = _call(lib.gauss, f[a:a + 12], 4)
        for o in range(4):
            if plain >> o & 1:
                continue
            taken += 1
            exact = sum(Fr(float(v)) * c for v, c in zip(f[a + o:a + o + 9], GAUSS))
            assert abs(Fr(float(got[o])) - exact) <= abs(exact) * EPS * Fr(171, 100), (a, o)
    n = 4 * (f.size - 11)
    assert taken == n if name in ("smooth", "binade", "noise", "none") else taken > n // 4


def _fourth_exact(w):
    w = [Fr(float(v)) for v in w]
    return w[0] - 4 * w[1] + 6 * w[2] - 4 * w[3] + w[4]


@pytest.mark.parametrize("across", ["like", "flat", "steep"])
@pytest.mark.parametrize("name", _fields().keys())
def test_fourth_differences(lib, name, across):
    """Five rows of a field that varies across the rows as along them, not at all, or by 10^3 a row."""
    f = _fields()[name]
    n = f.size - 12
    rows = {"like": [f[3 * j:n + 3 * j] for j in range(5)], "flat": [f[:n]] * 5,
            "steep": [f[:n] * 10.0 ** (3 * j) for j in range(5)]}[across]
    g = np.array(rows)
    taken = 0
    for a in range(0, n - 7):
        ok, got = _call(lib.fourth, g[:, a:a + 8], 8)
        if not ok:
            continue
        taken += 1
        for k in range(4):
            for w, v in ((g[2, a + k:a + k + 5], got[k]), (g[:, a + k + 2], got[4 + k])):
                exact = _fourth_exact(w)
                bound = EPS * abs(exact) + EPS * 8 * Fr(float(np.abs(w).max()))
                assert abs(Fr(float(v)) - exact) <= bound, (a, k)
    if across != "steep" and name in ("smooth", "binade", "noise", "top", "none"):
        assert taken == n - 7
    if across == "steep" and name not in ("none", "step", "spike"):
        assert taken == 0


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e290])
def test_inputs_out_of_range_are_refused(lib, bad):
    for k in range(14):
        x = np.ones(14)
        x[k] = bad
        assert not _call(lib.tenth, x, 4)[0]
        g = np.ones((5, 8))
        g[2, k % 8] = bad
        assert not _call(lib.fourth, g, 8)[0]
        assert k > 11 or _call(lib.gauss, x[:12], 4)[0] == 15
    assert _call(lib.gauss, np.full(12, 1e-300), 4)[0] == 15
    assert not _call(lib.tenth, np.full(14, 1e-300), 4)[0]
