"""The fixed-point exp and sin/cos of the FP64 structure factor, compiled for the host, against a 60-digit evaluation."""
import ctypes as C
import os
import shutil
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_2602_11709_gb300 import build as pkg_build

getcontext().prec = 60
PI = Decimal("3.14159265358979323846264338327950288419716939937510582097494")
EXP_N, SC_N = 1024, 512
SRC = r'''
#include "xrd_fx.cuh"
using namespace xrd;
extern "C" void host_exp(int n, const double* b, const double* s2, const uint64_t* tab, uint64_t* m, int* ex, double* out)
{
    for (int i = 0; i < n; i++) {
        const FxNum L = fx_log2e(b[i]), S = fx_num(s2[i]);
        m[i] = fx_exp2_neg(L.m, L.e, S.m, S.e, tab, ex[i]);
        out[i] = L.e == kFxSlow ? -1.0 : fx_exp_double(m[i], ex[i]);
    }
}
extern "C" void host_exp_sum(int n, const double* ab, const double* s2, const uint64_t* tab, double* out)
{
    for (int i = 0; i < n; i++) {
        uint64_t am[4], bm[4];
        int16_t ae[4], be[4];
        for (int j = 0; j < 4; j++) {
            int e;
            am[j] = fx_signed(ab[8 * i + 2 * j], e);
            ae[j] = (int16_t)e;
            const FxNum b = fx_log2e(ab[8 * i + 2 * j + 1]);
            bm[j] = b.m;
            be[j] = (int16_t)b.e;
        }
        out[i] = fx_exp_sum(am, ae, bm, be, fx_num(s2[i]), tab);
    }
}
extern "C" void host_sincos(int n, const uint64_t* P, const uint64_t* tab, int64_t* c, int64_t* s)
{
    for (int i = 0; i < n; i++) fx_sincos(P[i], (const ulonglong2*)tab, c[i], s[i]);
}
'''


def _sincos(x):
    """(sin, cos) of a Decimal 0 <= x <= 2 pi by the Taylor series."""
    t, k, s, c = Decimal(1), 0, Decimal(0), Decimal(1)
    while k < 90:
        k += 1
        t = t * x / k
        if k & 1:
            s += -t if k & 2 else t
        else:
            c += -t if k & 2 else t
    return s, c


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "t.cpp").write_text(SRC)
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(pkg_build.nvcc()))), "include")
    subprocess.run([shutil.which("g++"), "-O1", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I" + include,
                    "-I" + pkg_build.CSRC, str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    lib = C.CDLL(str(d / "t.so"))
    ln2 = Decimal(2).ln()
    exp = [min(int((-ln2 * j / EXP_N).exp() * 2 ** 64 + Decimal("0.5")), 2 ** 64 - 1) for j in range(EXP_N)]
    sc = []
    for j in range(SC_N + 1):
        s, c = _sincos(PI / 2 * j / SC_N)
        sc += [int(abs(c) * 2 ** 62 + Decimal("0.5")), int(s * 2 ** 62 + Decimal("0.5"))]
    lib.exp_tab, lib.sc_tab = np.array(exp, dtype=np.uint64), np.array(sc, dtype=np.uint64)
    return lib


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def _exp(fx, b, s2):
    """(m, n, double) of exp(-b s2) = m 2^(-64 - n)"""
    b, s2 = (np.ascontiguousarray(v, dtype=np.float64) for v in np.broadcast_arrays(b, s2))
    m, n, out = np.zeros(b.size, np.uint64), np.zeros(b.size, np.int32), np.zeros(b.size)
    fx.host_exp(b.size, _p(b), _p(s2), _p(fx.exp_tab), _p(m), _p(n), _p(out))
    return m, n, out


@pytest.mark.parametrize("s2", [1e-9, 1.0, 511.9, 512.0, 1023.9, 1024.0, 2047.0, 2048.0, 1e6, 1e300])
def test_zero_coefficient(fx, s2):
    """exp(-0 s^2) is 1 whatever s^2."""
    assert _exp(fx, [0.0, -0.0], s2)[2].tolist() == [1.0, 1.0]


def test_exp(fx):
    """Relative error of m below (1/2 + b s^2 / 128) 2^-53: the exponent is kept to 53 bits (0.35 of them), and of the
    product four of its 62 to 64 bits are lost, which grow with the exponent. The double is m rounded to nearest, zero
    below 2^-1021."""
    rng = np.random.default_rng(3)
    x = np.concatenate([10.0 ** rng.uniform(-12, 2.845, 3000), rng.uniform(0.0, 800.0, 1500), np.log(2.0) * np.arange(1, 1030)])
    s2 = 10.0 ** rng.uniform(-8, 6, x.size)
    b = x / s2
    for m, n, g, bi, si in zip(*_exp(fx, b, s2), b, s2):
        y = Decimal(float(bi)) * Decimal(float(si))
        ref, got = (-y).exp(), Decimal(int(m)) / Decimal(2) ** (64 + int(n))
        if ref < Decimal(2) ** -1020:
            assert got <= Decimal(2) ** -1020
        else:
            assert abs(got - ref) <= (Decimal("0.5") + y / 128) * Decimal(2) ** -53 * ref
        assert g == (np.ldexp(float((int(m) + 1024) >> 11), 11 - 64 - int(n)) if m else 0.0)
    assert _exp(fx, [1.0, 1e80], [1e4, 1e80])[2].tolist() == [0.0, 0.0]
    assert _exp(fx, [-1.0, 1e200, 1e-200, np.inf, np.nan], 1.0)[2].tolist() == [-1.0] * 5  # left to the library's exp


@pytest.mark.parametrize("form", ["positive", "signs", "spread", "zeros"])
@pytest.mark.parametrize("s2", [0.01, 1.0, 10.0, 25.0, 100.0, 1500.0])
def test_exp_sum(fx, form, s2):
    """sum_i a_i exp(-b_i s^2) with every term's own relative error, as in FP64, also where those of the largest a_i have
    decayed: the exponential's (1/2 + b s^2 / 128) 2^-53 and 2^-57 of the largest term each (two truncated products and
    the alignment), then the rounding of the sum. Exponentials below 2^-1021 and sums below 2^-1022 are zero."""
    rng = np.random.default_rng(5)
    ab = np.stack([rng.uniform(0.5, 4.0, (300, 4)), rng.uniform(0.05, 50.0, (300, 4))], axis=2)
    if form == "signs":
        ab[:, :, 0] *= rng.choice([-1.0, 1.0], (300, 4))
    elif form == "spread":
        ab[:, :, 0] *= 10.0 ** rng.integers(-80, 80, (300, 4))
    elif form == "zeros":
        ab[np.arange(300), rng.integers(0, 4, 300), 0] = 0.0
        ab[np.arange(300), rng.integers(0, 4, 300), 1] = 0.0
    ab, s, out = np.ascontiguousarray(ab), np.full(300, s2), np.zeros(300)
    fx.host_exp_sum(300, _p(ab), _p(s), _p(fx.exp_tab), _p(out))
    for c, g in zip(ab, out):
        y = [Decimal(float(b)) * Decimal(s2) for b in c[:, 1]]
        t = [Decimal(float(a)) * (-v).exp() for a, v in zip(c[:, 0], y)]
        lost = Decimal(2) ** -1022 + sum(abs(Decimal(float(a))) * Decimal(2) ** -1020 for a, v in zip(c[:, 0], y) if v > 707)
        unit = Decimal(2) ** -53
        bound = sum(abs(v) * (Decimal("0.5") + w / 128) * unit for v, w in zip(t, y)) + max(map(abs, t)) * unit / 4 + abs(sum(t)) * unit + lost
        assert abs(Decimal(float(g)) - sum(t)) <= bound


def test_sincos(fx):
    """Absolute error below 6.5e-18: x^3 is kept to 2^-56 from x^2 to 2^-48 and x to 2^-40 (5.5e-18 in x^3 / 6), the rest to
    2^-62. Exact at the quarter turns."""
    rng = np.random.default_rng(4)
    P = np.concatenate([rng.integers(0, 2 ** 64, 1500, dtype=np.uint64), (rng.integers(0, 2048, 500, dtype=np.uint64) << np.uint64(53))
                        - np.uint64(1), np.arange(4, dtype=np.uint64) << np.uint64(62)])
    c, s = np.zeros(P.size, np.int64), np.zeros(P.size, np.int64)
    fx.host_sincos(P.size, _p(P), _p(fx.sc_tab), _p(c), _p(s))
    unit, bound = Decimal(2) ** -62, Decimal("6.5e-18")
    for p, ci, si in zip(P, c, s):
        rs, rc = _sincos(2 * PI * int(p) / 2 ** 64)
        assert abs(int(ci) * unit - rc) <= bound and abs(int(si) * unit - rs) <= bound
    one = 2 ** 62
    assert list(zip(c[-4:].tolist(), s[-4:].tolist())) == [(one, 0), (0, one), (-one, 0), (0, -one)]
