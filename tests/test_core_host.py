"""The pair core (csrc/lcdm_core.cuh), compiled for the host, against the
quadrature oracle: every root kind (quartic and cubic, conjugate pair and four
or three reals), all column counts, both precisions, from z = 1e-4 to 1100 and
beyond the scaling threshold of single precision, and the limit at infinity.

Bounds: values as in test_gpu_parity.py (FP64 1e-12; FP32 2e-6, X 1e-4);
gradients FP64 1e-9 + 1e-11/z, FP32 3e-5 + 2e-6/z (chi) and 1e-4 + 2e-6/z (t)
of the row's largest entry."""
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

# (H0, Om, OL, Or[, Ok[, Os, Ox]])
ROWS = {
    "quartic, pair": [70.0, 0.3, 0.7, 5e-5],
    "quartic, pair, open": [65.0, 0.3, 0.1, 5e-5],
    "quartic, pair, closed": [70.0, 0.3, 1.2, 1e-4],
    "quartic, pair, near the boundary": [70.0, 0.3, 1.7136, 5e-5],
    "quartic, reals, recollapsing": [70.0, 2.0, 0.01, 5e-5],
    "quartic, reals, negative Lambda": [70.0, 0.3, -0.2, 5e-5],
    "quartic, five columns": [70.0, 0.3, 0.6, 5e-5, 0.08],
    "quartic, seven columns": [70.0, 0.3, 0.6, 5e-5, 0.05, 0.03, 0.02],
    "cubic, pair": [70.0, 0.3, 0.7, 0.0],
    "cubic, open": [70.0, 0.2, 0.05, 0.0],
    "cubic, reals": [70.0, 0.3, -0.2, 0.0],
    "cubic, seven columns": [70.0, 0.3, 0.6, 0.0, 0.05, 0.03, 0.02],
}


@pytest.fixture(scope="module")
def core(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or CUDA is None:
        pytest.skip("g++ or the CUDA headers are missing")
    so = str(tmp_path_factory.mktemp("core") / "libcore.so")
    subprocess.run([gxx, "-O2", "-x", "c++", "-std=c++17", "-shared", "-fPIC", "-I" + CUDA, "-I" + CSRC,
                    os.path.join(HERE, "core_host.cpp"), "-o", so], check=True, capture_output=True)
    return ctypes.CDLL(so)


def _roots(P):
    """Labelled roots and their derivatives in 40 digits, rounded once."""
    mp.mp.dps = 40
    ncol, K = len(P), len(P) - 1
    Om, OL, Or = (mp.mpf(v) for v in P[1:4])
    Ok = mp.mpf(P[4]) if ncol >= 5 else 1 - Om - OL - Or
    Os, Ox = (mp.mpf(P[5]), mp.mpf(P[6])) if ncol == 7 else (mp.mpf(0), mp.mpf(0))
    quartic = P[3] > 0
    co = [Or, Om, Ok + Os, Ox, OL] if quartic else [Om, Ok + Os, Ox, OL]
    r = mp.polyroots(co, maxsteps=500, extraprec=200)
    tiny = mp.mpf(10) ** -25
    re = sorted([t.real for t in r if abs(t.imag) < tiny * abs(t)], key=lambda t: -abs(t))
    cx = [t for t in r if t.imag > tiny * abs(t)]
    A, rest = (re[0], re[1:]) if quartic else (mp.mpf(0), re)
    B, rest = rest[0], rest[1:]

    def d(k, x):
        b = [x ** 3, 1, x ** 4, x ** 2, x ** 2, x][k] - (x ** 2 if ncol == 4 else 0)
        return -b / (4 * Or * x ** 3 + 3 * Om * x ** 2 + 2 * (Ok + Os) * x + Ox)

    dr = np.zeros((K, 4))
    for k in range(K):
        dr[k, 0] = float(d(k, A)) if quartic else 0.0
        dr[k, 1] = float(d(k, B))
        if cx:
            dr[k, 2], dr[k, 3] = float(d(k, cx[0]).real), float(d(k, cx[0]).imag)
        else:
            dr[k, 2], dr[k, 3] = (float(d(k, x)) for x in rest)
    pair = [cx[0].real, cx[0].imag] if cx else rest
    return int(quartic), int(bool(cx)), np.array([float(v) for v in [A, B, *pair]]), dr


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("name", ROWS)
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_integrals_and_gradients(core, name, prec):
    P = np.array(ROWS[name])
    quartic, cpair, roots, dr = _roots(ROWS[name])
    K = len(P) - 1
    rng = np.random.default_rng(3)
    z = np.concatenate([rng.uniform(0.01, 10.0, 40), 10.0 ** rng.uniform(-4, np.log10(1100.0), 40)])
    if prec == "fp32":
        z = z.astype(np.float32).astype(np.float64)
    out, grad = np.zeros((z.size, 4)), np.zeros((z.size, 2, K))
    core.core_pairs(_ptr(P), len(P), quartic, cpair, _ptr(roots), _ptr(dr), int(prec == "fp64"), z.size, _ptr(z), _ptr(out),
                    _ptr(grad))
    assert not out[:, 3].any()
    ref, jac = oracle.quad_distances(P[None], z, np.array([0, z.size]), grad=True)
    scale = np.array([C, T_H, C]) / P[0]
    tol = np.array([1e-12] * 3 if prec == "fp64" else [2e-6, 2e-6, 1e-4])
    assert np.all(np.abs(out[:, :3] * scale / ref[:, :3] - 1).max(axis=0) <= tol)
    cols = [k for k in range(K) if quartic or k != 2]     # no Omega_r direction in a cubic
    for q, base in ((0, 3e-5), (1, 1e-4)):
        want = jac[:, q, 1:][:, cols]
        err = np.abs(grad[:, q][:, cols] * scale[q] - want).max(axis=1) / np.abs(want).max(axis=1)
        bound = 1e-9 + 1e-11 / z if prec == "fp64" else base + 2e-6 / z
        assert np.all(err <= bound), (q, (err / bound).max())


@pytest.mark.parametrize("z", [6.4e4, 6.6e4, 1e6, 1e9])
def test_very_large_redshifts(core, z):
    """Across the single-precision scaling threshold (65536) and far beyond:
    within 1e-4 of double precision (1 + z q carries the argument's rounding)."""
    P = np.array(ROWS["quartic, pair"])
    quartic, cpair, roots, dr = _roots(list(P))
    res = []
    for fp64 in (0, 1):
        zz, out, grad = np.array([float(np.float32(z))]), np.zeros((1, 4)), np.zeros((1, 2, 3))
        core.core_pairs(_ptr(P), 4, quartic, cpair, _ptr(roots), _ptr(dr), fp64, 1, _ptr(zz), _ptr(out), _ptr(grad))
        assert out[0, 3] == 0
        res.append(out[0, :2].copy())
    assert np.all(np.abs(res[0] / res[1] - 1) <= 1e-4)


@pytest.mark.parametrize("name", ["quartic, pair", "quartic, pair, open", "quartic, reals, recollapsing", "cubic, pair"])
def test_limit_at_infinity(core, name):
    P = np.array(ROWS[name])
    quartic, cpair, roots, dr = _roots(ROWS[name])
    out, grad = np.zeros(2), np.zeros((2, 3))
    core.core_limit(_ptr(P), quartic, cpair, _ptr(roots), _ptr(dr), _ptr(out), _ptr(grad))
    ref, jac = oracle.quad_limits(P[None], np.zeros(1), grad=True)
    scale = np.array([C, T_H]) / P[0]
    assert np.all(np.abs(out * scale / ref[0] - 1) <= 1e-12)
    cols = [0, 1, 2] if quartic else [0, 1]
    want = jac[0][:, 1:][:, cols]
    err = np.abs(grad[:, cols] * scale[:, None] - want).max(axis=1) / np.abs(want).max(axis=1)
    assert np.all(err <= 1e-9)
