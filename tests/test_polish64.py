"""The FP64 con2prim polish of the mixed path (csrc/dg_polish64.cuh), compiled for the host: its
residual and Newton slope against 60-digit arithmetic."""
import ctypes
import os
import subprocess
from decimal import Decimal as Dec
from decimal import getcontext

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_00098_gb300", "csrc")
SRC = """
#include "dg_polish64.cuh"
extern "C" void run(long n, double g, const double *u, double *o)
{
    for (long i = 0; i < n; ++i) {
        const double *s = u + 4 * i;  // D, s2, tau, p
        const dg::PolishEval r = dg::sr_polish_eval(g, s[0], s[2] + s[0], s[1], s[2], s[3]);
        o[3 * i] = r.f;
        o[3 * i + 1] = r.fq / r.f / r.dq;
        o[3 * i + 2] = r.scale;
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("polish64")
    src, so = str(d / "t.cpp"), str(d / "t.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, src, "-o", so],
                   check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("g", [4.0 / 3.0, 5.0 / 3.0, 1.9, 2.0])
@pytest.mark.parametrize("W", [1.01, 2.0, 30.0, 1e3, 1e5])
def test_residual_and_slope_in_64_bits(lib, g, W):
    """1 - v^2 = 1/W^2 carries the rounding of v^2, some 2^-53 W^2 of it, and so do 1/W and the
    slope; the residual's rounding is some 2^-53 of its terms times W^2 (v^2's share).  A slope
    formed in FP32 is off by 2^-24 / f', 10^5 times more at W = 1e3 and g = 2."""
    getcontext().prec = 60
    r = np.random.RandomState(int(W) + int(100 * g))
    u, want = [], []
    for _ in range(60):
        rho, eps = 10.0 ** r.uniform(-6, 2), 10.0 ** r.uniform(-8, 8)
        p = (g - 1.0) * rho * eps
        v2 = 1.0 - 1.0 / W ** 2
        D, wh = rho * W, (rho * (1.0 + eps) + p) * W * W
        s2, tau = wh * wh * v2, wh - p - D
        if tau <= 0.0:
            continue
        q = p * r.uniform(0.9, 1.1)
        if not s2 < (tau + D + q) ** 2 * (1.0 - 0.1 / W ** 2):
            continue
        u.append([D, s2, tau, q])
        d, s, t, x, c = (Dec(float(z)) for z in (D, s2, tau, q, g))
        Ep = t + d + x
        V2 = s / (Ep * Ep)
        Wl = 1 / (1 - V2).sqrt()
        f = x - (c - 1) * (t - V2 * (Ep - d * Wl / (Wl + 1)))
        want.append([f, 1 / (1 - (c - 1) * V2 * (1 - d * Wl / Ep)), Wl * Wl])
    assert len(u) > 20
    a, o = np.array(u), np.empty((len(u), 3))
    lib.run(ctypes.c_long(len(u)), ctypes.c_double(g), a.ctypes.data_as(ctypes.c_void_p),
            o.ctypes.data_as(ctypes.c_void_p))
    for (f, inv, scale), (wf, winv, w2) in zip(o, want):
        bound = 16 * 2.0 ** -53 * float(w2)
        assert abs(Dec(float(f)) - wf) <= Dec(bound * scale)
        assert abs(Dec(float(inv)) / winv - 1) <= Dec(bound)
