"""The integer exponential, logarithm, reciprocal and roots of the closure (fix64.cuh), compiled for
the host: errors against long double over their ranges and at the edges of their reductions, and
the committed table against its generator.

Bounds, from the truncations listed beside each step of the header: the exponential's polynomial
keeps 2^-57 and the final rounding to binary64 adds half an ulp (0.5 + 2^-57 2^53 = 0.57 and the
reduced argument's 2^-54 for |x| up to 512: 0.65 ulp); the mantissas of the reciprocal and the root
are within 2^-60, so one rounding gives 0.51 ulp, two products 0.52; the logarithm is within 2^-54."""
import ctypes
import importlib.util
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2210_05547_gb300", "csrc")
SHIM = """
#include "fix64.cuh"
extern "C" void run(int fn, long n, const double* a, const double* b, double* out) {
    using namespace hyp;
    for (long i = 0; i < n; ++i) {
        if (fn == 0) out[i] = fix_exp(a[i]);
        if (fn == 1) out[i] = fix_div(a[i], b[i]);
        if (fn == 2) out[i] = fix_rcp(a[i]);
        if (fn == 3) out[i] = fix_sqrt(a[i]);
        if (fn == 4) out[i] = fix_rsqrt(a[i]);
        if (fn == 5) out[i] = f64_of_signed(log58(a[i]), 58);
    }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fix64")
    src, lib = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run([gxx, "-O1", "-w", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).run
    f.argtypes = [ctypes.c_int, ctypes.c_long] + [ctypes.c_void_p] * 3

    def call(fn, a, b=None):
        a = np.ascontiguousarray(a, dtype=np.float64)
        b = a if b is None else np.ascontiguousarray(b, dtype=np.float64)
        out = np.empty_like(a)
        f(fn, a.size, a.ctypes.data, b.ctypes.data, out.ctypes.data)
        return out
    return call


def _ulps(got, exact):
    return np.max(np.abs(got - exact) / np.spacing(np.abs(exact.astype(np.float64))))


def test_table_is_the_generators_output():
    spec = importlib.util.spec_from_file_location("gen", os.path.join(CSRC, "gen_fix_table.py"))
    gen = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(gen)
    assert open(os.path.join(CSRC, "fix_table.h")).read() == gen.render()


def test_exponential(run):
    rng = np.random.default_rng(1)
    k = np.arange(-60000, 60000) * (np.log(2.0) / 256)          # the reduction's breakpoints
    x = np.concatenate([rng.uniform(-511.9, 511.9, 200000), -rng.uniform(0, 45, 200000), k,
                        np.nextafter(k, np.inf), rng.uniform(-1e-5, 1e-5, 10000),
                        [0.0, -0.0, 5e-324, -5e-324, 511.9999, -511.9999]])
    assert _ulps(run(0, x), np.exp(x.astype(np.longdouble))) <= 0.65


def test_quotients_and_roots(run):
    rng = np.random.default_rng(2)
    edge = np.array([1.0, 2.0, np.nextafter(1.0, 2), np.nextafter(2.0, 1), np.nextafter(4.0, 1), 3.0])
    m = np.concatenate([1.0 + rng.uniform(0, 1, 200000), edge])
    b = np.ldexp(m, rng.integers(-119, 119, m.size)) * rng.choice([-1.0, 1.0], m.size)
    a = np.ldexp(1.0 + rng.uniform(0, 1, m.size), rng.integers(-119, 119, m.size))
    L = np.longdouble
    assert _ulps(run(1, a, b), a.astype(L) / b.astype(L)) <= 0.52
    assert _ulps(run(2, b), 1 / b.astype(L)) <= 0.51
    c = np.abs(b)
    assert _ulps(run(3, c), np.sqrt(c.astype(L))) <= 0.52
    assert _ulps(run(4, c), 1 / np.sqrt(c.astype(L))) <= 0.51


def test_logarithm(run):
    rng = np.random.default_rng(3)
    j = 1.0 + np.arange(128) / 128
    x = np.concatenate([np.exp(rng.uniform(np.log(2.0), np.log(2.0 ** 45), 200000)),
                        rng.uniform(50.0, 1e5, 200000), 1024.0 * j, np.nextafter(1024.0 * j, 0)])
    exact = np.log(x.astype(np.longdouble))
    err = np.abs(run(5, x) - exact)
    assert np.max(err - 0.5 * np.spacing(exact.astype(np.float64))) <= 2.0 ** -54
