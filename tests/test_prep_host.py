"""The root preparation (csrc/lcdm_prep.cuh) compiled for the host: status,
kind and roots against 60-digit roots, and the integrals on them against the
quadrature oracle."""
import ctypes
import os
import shutil
import subprocess

import mpmath as mp
import numpy as np
import pytest

import oracle

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2212_01937_gb300", "csrc")
CUDA = next((d for d in ("/usr/local/cuda/include",) if os.path.exists(os.path.join(d, "cuda_runtime.h"))), None)

C, T_H = 299792.458, 977.7922216807891


@pytest.fixture(scope="module")
def prep(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or CUDA is None:
        pytest.skip("g++ or the CUDA headers are missing")
    so = str(tmp_path_factory.mktemp("prep") / "libprep.so")
    subprocess.run([gxx, "-O2", "-w", "-x", "c++", "-std=c++17", "-shared", "-fPIC", "-I" + CUDA, "-I" + CSRC,
                    os.path.join(HERE, "prep_host.cpp"), "-o", so], check=True, capture_output=True)
    return ctypes.CDLL(so)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _rows(prep, P, near):
    P = np.ascontiguousarray(P, dtype=np.float64)
    st, kind, r = np.zeros(len(P), np.int32), np.zeros(len(P), np.int32), np.zeros((len(P), 4))
    prep.prep_rows(_ptr(P), ctypes.c_int64(len(P)), P.shape[1], ctypes.c_float(near), _ptr(st), _ptr(kind), _ptr(r))
    return st, kind, r


def _exact(P):
    """Real roots and those of the upper half-plane of the row's E^2(x), its
    coefficients as double precision forms them."""
    mp.mp.dps = 60
    Om, OL, Or = (float(v) for v in P[1:4])
    Ok = float(P[4]) if len(P) >= 5 else 1.0 - Om - OL - Or
    Os, Ox = (float(P[5]), float(P[6])) if len(P) == 7 else (0.0, 0.0)
    co = ([Or] if Or > 0 else []) + [Om, Ok + Os, Ox, OL]
    r = mp.polyroots([mp.mpf(c) for c in co], maxsteps=2000, extraprec=400)
    tiny = mp.mpf(10) ** -25
    return [x.real for x in r if abs(x.imag) <= tiny * abs(x)], [x for x in r if x.imag > tiny * abs(x)]


def _status(row, re, cx):
    """1: a real root at z >= 0; 5: two pairs; 3: the cubic's special root at x = 0."""
    if any(x >= 1 for x in re):
        return 1
    return 5 if len(cx) == 2 else 3 if row[3] == 0 and cx and re[0] == 0 else 0


def _check(prep, P, near):
    """Status, kind and the roots to 1e-13 (an isolated root is good to a few
    ulp, 1e-15; one of a pair is polished to the same, and its condition number,
    at most 1e5 where they are 1e-5 apart, multiplies the polish's residual of
    1e-32 only)."""
    st, kind, r = _rows(prep, P, near)
    for b, row in enumerate(P):
        re, cx = _exact(row)
        quartic = row[3] > 0
        assert st[b] == _status(row, re, cx), (row.tolist(), st[b])
        if len(cx) == 2:
            continue
        assert kind[b] == (0 if quartic else 2) + (0 if cx else 1), (row.tolist(), kind[b])
        got = ([r[b, 0]] if quartic else []) + [r[b, 1]] + ([complex(r[b, 2], r[b, 3])] if cx else [r[b, 2], r[b, 3]])
        for w in re + cx:
            w = complex(w)
            assert min(abs(g - w) for g in got) <= 1e-13 * abs(w), (row.tolist(), w, got)


def _double_root(rng, ncol, quartic):
    """A row with a double root x0: (Om, OL, Or, ...) by p(x0) = p'(x0) = 0."""
    while True:
        Om, Or = rng.uniform(0.05, 3.0), 10.0 ** rng.uniform(-6, -3) if quartic else 0.0
        Os, Ox = (rng.uniform(-0.05, 0.05), rng.uniform(-0.05, 0.05)) if ncol == 7 else (0.0, 0.0)
        if ncol > 4:
            x = rng.uniform(0.1, 4.0)
        else:   # with the closure: bisection
            f = lambda x: Or * x ** 4 + 0.5 * Om * x ** 3 - 0.5 * (4 * Or * x * x + 3 * Om * x) - (1 - Om - Or)
            g = np.linspace(0.01, 6.0, 400)
            v = f(g)
            k = np.nonzero(v[:-1] * v[1:] < 0)[0]
            if not k.size:
                continue
            k = rng.choice(k)
            a, b = g[k], g[k + 1]
            for _ in range(200):
                m = 0.5 * (a + b)
                a, b = (a, m) if f(a) * f(m) <= 0 else (m, b)
            x = a
        c = -(4 * Or * x ** 3 + 3 * Om * x * x + Ox) / (2 * x)
        OL = -(Or * x ** 4 + Om * x ** 3 + c * x * x + Ox * x)
        return [70.0, Om, OL, Or, c - Os, Os, Ox][:ncol]


@pytest.mark.parametrize("near", [0.1, 0.01])
@pytest.mark.parametrize("quartic", [True, False])
@pytest.mark.parametrize("ncol", [4, 5, 7])
def test_nearly_double_roots(prep, ncol, quartic, near):
    """Relative distances 1e-10 to 1e-5 of OL from the value at which two roots
    coincide, on both sides: the boundaries to no Big Bang (x0 > 1) and to
    recollapse (x0 < 1)."""
    rng = np.random.default_rng(11)
    P = []
    for i in range(60):
        row = _double_root(rng, ncol, quartic)
        row[2] *= 1.0 + 10.0 ** rng.uniform(-10, -5) * (1 if i % 2 else -1)
        P.append(row)
    _check(prep, np.array(P), near)


def _low_radiation(rng, ncol):
    """Om / Or from 1e4 to 1e7 (across the root sweeps' two ranges of
    coefficients) with OL from 1e-12 to 1."""
    Om = rng.uniform(0.05, 0.6)
    row = [70.0, Om, 10.0 ** rng.uniform(-12, 0), Om / 10.0 ** rng.uniform(4, 7)]
    return row + [10.0 ** rng.uniform(-6, 0), 10.0 ** rng.uniform(-6, -1), 10.0 ** rng.uniform(-6, -1)][:ncol - 4]


@pytest.mark.parametrize("near", [0.1, 0.01])
@pytest.mark.parametrize("ncol", [4, 5, 7])
def test_low_radiation(prep, ncol, near):
    rng = np.random.default_rng(12)
    _check(prep, np.array([_low_radiation(rng, ncol) for _ in range(100)]), near)


@pytest.mark.parametrize("row", [[70.0, 0.3, 1e-4, 7e-7],
                                 [70.0, 3.59100770371796, -5.521955913688765e-06, 1.0813750580855664e-05],
                                 [70.0, 1.1555128340131777, 4.6205600454127664e-08, 3.1582537844621348e-06,
                                  -0.9848739552881378],
                                 [70.0, 0.2462031973093668, -1.976969922057992e-25, 1e-05, 8.522853391548514e-10,
                                  4.967495035992166e-09, 0.0],
                                 [70.0, 0.8123634327126253, -4.790791447752325e-25, 1e-05, 1.09264510906137e-08,
                                  2.4156781053752366e-08, 0.0]])
def test_single_precision_range(prep, row):
    """A root of 3e5 to 1e6 whose closed-form start is not good (the sweeps'
    products), and three reals of 1e-8 (the discriminant)."""
    for near in (0.1, 0.01):
        _check(prep, np.array([row]), near)


def _zero_root(rng, quartic):
    """Omega_L0 = 0 beside Omega_x0: a single root at exactly x = 0."""
    return [70.0, rng.uniform(0.05, 0.6), 0.0, 10.0 ** rng.uniform(-6, -3) if quartic else 0.0,
            10.0 ** rng.uniform(-6, 0), 10.0 ** rng.uniform(-3, -1), 10.0 ** rng.uniform(-6, 0)]


@pytest.mark.parametrize("near", [0.1, 0.01])
@pytest.mark.parametrize("quartic", [True, False])
def test_zero_root(prep, quartic, near):
    rng = np.random.default_rng(13)
    _check(prep, np.array([_zero_root(rng, quartic) for _ in range(60)]), near)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_values_inside_the_recollapse_boundary(prep, prec):
    """Two real roots 2e-7 inside the boundary, at x = 0.372."""
    P = np.array([70.0, 2.1387452198383516, 0.055124236364160493, 1e-4])
    z = np.array([0.01, 0.1, 0.5, 1.0, 3.0, 10.0, 1100.0])
    if prec == "fp32":
        z = z.astype(np.float32).astype(np.float64)
    out = np.zeros((z.size, 4))
    assert prep.prep_pairs(_ptr(P), 4, int(prec == "fp64"), z.size, _ptr(z), _ptr(out)) == 0
    assert not out[:, 3].any()
    ref = oracle.quad_distances(P[None], z, np.array([0, z.size]))
    tol = np.array([1e-12] * 3 if prec == "fp64" else [2e-6, 2e-6, 1e-4])
    assert np.all(np.abs(out[:, :3] * np.array([C, T_H, C]) / P[0] / ref[:, :3] - 1).max(axis=0) <= tol)
