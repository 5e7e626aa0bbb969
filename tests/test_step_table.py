"""The FP32 step table that the device makes of a pulse (dsp_steptable.h, compiled here for the host):
the running sum of its entries stays within half an ulp of an entry of the exact running sum however
long the run, and every entry is its step's value to an ulp."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1607_03062_gb300 import build as Bd

SHIM = r"""
#include "dsp_steptable.h"
extern "C" void table(const double *a, int64_t n, int per, double sdt, float *out)
{
    const int64_t blocks = (n + dsp::kTableBlock - 1) / dsp::kTableBlock;
    double *pre = new double[2 * (blocks + 1)];
    double *copy = new double[2 * n * per];
    dsp::copy_with_prefix(a, n, per, copy, pre);
    a = copy;
    const double h = per == 2 ? 0.5 * sdt : sdt;
    for (int c = 0; c < 2; ++c)
        for (int64_t g = blocks - 1; g >= 0; --g)  // any order
            dsp::table_block(g, n, h * pre[2 * g + c], h * pre[2 * g + 2 + c],
                             [&](int64_t k) {
                                 return per == 2 ? sdt * (0.5 * (a[4 * k + c] + a[4 * k + 2 + c]))
                                                 : sdt * a[2 * k + c];
                             },
                             [&](int64_t k, float f) { out[2 * k + c] = f; });
    delete[] pre;
    delete[] copy;
}
"""


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    d = tmp_path_factory.mktemp("steptable")
    (d / "shim.cpp").write_text(SHIM)
    lib = d / "libshim.so"
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    Bd.CSRC, str(d / "shim.cpp"), "-o", str(lib)], check=True)
    fn = ctypes.CDLL(os.fspath(lib)).table
    fn.restype = None

    def run(a, per, sdt):
        a = np.ascontiguousarray(a, np.float64)
        n = len(a)
        out = np.full((n, 2), np.nan, np.float32)
        fn(a.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(n), ctypes.c_int(per),
           ctypes.c_double(sdt), out.ctypes.data_as(ctypes.c_void_p))
        return out.astype(np.float64)
    return run


def tables(n):
    t = np.arange(n) / n
    rng = np.random.default_rng(2)
    jump = np.full(n, 0.37)
    jump[n // 3:] = 1.1
    spikes = np.full(n, 1e-9)
    spikes[::97] = 2.7
    return {"plateau": np.full(n, 0.7311), "top of a binade": np.full(n, 1.0 - 2.0 ** -26),
            "sine": 2.3 * np.sin(40 * np.pi * t), "tail": np.exp(-((t - 0.5) * 30) ** 2),
            "noise": rng.standard_normal(n), "jump": jump, "spikes": spikes, "zero": np.zeros(n)}


@pytest.mark.parametrize("per", [1, 2])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 1000, 100003])
def test_running_sum_keeps_to_the_exact_one(table, n, per):
    """Bounds: |F_n - S_n| <= q_n / 2, q_n the float spacing at the larger of the steps n and n + 1
    (twice it within 2^-20 of a power of two), or 2^-50 |S_n| where that is more, plus the rounding
    of the FP64 sums themselves, at most 16 of 2^-53 of the running sum (the values 2, sums inside a
    block 5 and outside 2, products 3); an entry is F_n - F_(n-1), so off by at most (q_n + q_(n-1))
    / 2."""
    sdt = -0.0113
    for name, col in tables(n).items():
        a = np.stack([col, -0.5 * col[::-1]], 1)
        if per == 2:
            a = np.stack([a, 1.25 * a], 1).reshape(n, 4)
        v = sdt * (0.5 * (a[:, :2] + a[:, 2:]) if per == 2 else a)
        f = table(a, per, sdt)
        exact = np.cumsum(v.astype(np.longdouble), axis=0)
        got = np.cumsum(f.astype(np.longdouble), axis=0)
        w = np.maximum(np.abs(v), np.abs(np.vstack([v[1:], v[-1:]])))
        q = np.spacing((w * (1 + 2.0 ** -20)).astype(np.float32)).astype(np.float64)
        q = np.maximum(q, 2.0 ** -50 * np.abs(exact).astype(np.float64))
        slack = 16 * 2.0 ** -53 * np.abs(exact).max()
        # steps 2^23 apart: their entry is rounded
        slack += 2.0 ** -24 * q.max() * np.sum(q[1:] > 4e6 * q[:-1])
        assert np.all(np.abs(got - exact) <= q / 2 + slack), (name, n)
        before = np.vstack([np.zeros((1, 2)), q[:-1]])
        assert np.all(np.abs(f - v) <= (q + before) / 2 + slack), (name, n)
