"""The coefficient tables of the interval polynomials (poly_table.cu), on the
host: evaluated in 64 bits on the spectrum of each bucket they give the
interval's function ((1 + dt x / 2) / (1 - dt x / 2))^S to what is cut off and the FP32
rounding of the coefficients, on both sides of every line of the rule, and there
is no table where the function is not smooth."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1304_2062_gb300", "csrc",
                   "poly_table.cu")
BUCKETS, MOST = 8, 64


class Table(ctypes.Structure):
    _fields_ = [("reinsch", ctypes.c_int), ("len", ctypes.c_int), ("inv_beta", ctypes.c_float),
                ("m", ctypes.c_int * BUCKETS), ("h", ctypes.c_float * BUCKETS),
                ("c", (ctypes.c_float * MOST) * BUCKETS)]


@pytest.fixture(scope="module")
def make(tmp_path_factory):
    d = tmp_path_factory.mktemp("poly")
    src, lib = d / "t.cpp", d / "t.so"
    src.write_text(f'#include "{SRC}"\nextern "C" int make(double b, double T, int S, PolyTable *t) '
                   '{ return se2n_poly_make(b, T, S, *t); }\n')
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-o", str(lib), str(src)], check=True)
    fn = ctypes.CDLL(str(lib)).make
    fn.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_int, ctypes.POINTER(Table)]

    def call(beta, T, S):
        t = Table()
        return t if fn(beta, T, S, ctypes.byref(t)) else None
    return call


@pytest.mark.parametrize("beta", [0.004, 0.1, 0.25, 0.5, 3.0])
@pytest.mark.parametrize("T", [1e-4, 0.1, 0.5, 2.0, 5.0, 8.0, 13.0, 25.0, 50.0, 60.0])
def test_tables_give_the_interval(make, beta, T):
    for factor in (1, 2, 40):  # the largest admitted step, and smaller ones
        S = math.ceil(factor * T * (2 + 4 * beta) / 2)
        t = make(beta, T, S)
        if t is None:  # only where many coefficients are needed
            assert T * (2 + 4 * beta) > 140
            continue
        dt = T / S
        assert t.len == max(t.m) and 2 <= min(t.m) and t.len <= (MOST if t.reinsch else 32)
        for b in range(BUCKETS):
            w = 4 * beta + 2 * (b + 1) / BUCKETS
            x = -w * (0.5 - 0.5 * np.cos(np.linspace(0, np.pi, 401)))
            f = np.exp(2.0 * S * np.arctanh(np.maximum(0.5 * dt * x, -1 + 1e-16)))
            c = np.array(t.c[b][:t.m[b]], dtype=np.float64)
            assert not np.any(np.array(t.c[b][t.m[b]:]))
            u = x / beta / np.float64(t.h[b]) + 1.0   # (M + h) / h
            if t.reinsch:
                p = np.polynomial.chebyshev.chebval(u, c)
                size = np.abs(c).sum()
            else:  # f = 1 + x g(x), g by powers of M + h
                p = 1.0 + x / beta * np.polynomial.polynomial.polyval(u * t.h[b], c)
                size = np.max(np.abs(x / beta)) * np.sum(np.abs(c) * np.float64(t.h[b]) ** np.arange(len(c)))
                assert size < 25.0
            # cut off; half an ulp a coefficient; h half an ulp off moves x by as much of w
            slack = 2e-8 + 2.0 ** -24 * (size + np.max(np.abs(np.gradient(f, x))[1:-1]) * w + 1.0)
            assert np.max(np.abs(p - f)) <= slack, (beta, T, S, b, t.reinsch)


def test_no_table_where_the_function_is_not_smooth(make):
    assert make(0.25, 2.0, 2) is None      # dt (2 + 4 beta) = 3
    assert make(0.25, 2.0, 3) is not None  # 2
    assert make(10.0, 100.0, 100) is None
    assert make(0.25, 150.0, 3000) is None  # more than 64 coefficients
    assert make(1e-13, 2.0, 100) is None    # a_r^2 / beta too large for FP32 volumes
    assert make(1e-11, 2.0, 100) is not None
