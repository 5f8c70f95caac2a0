"""The pair core (csrc/lcdm_core.cuh), compiled for the host, at very large
redshifts, across the thresholds of its scaling (1e9 in double precision, 65536
in single), against 40-digit quadrature in u = 1 / (1 + z),
  chi = int du / sqrt(g), t = int u du / sqrt(g), X = int u^-2 du / sqrt(g),
  g(u) = u^4 E^2(1/u).
Bounds as at ordinary redshifts: FP64 1e-12 and, for gradients, 1e-9 of the
row's largest entry."""
import mpmath as mp
import numpy as np
import pytest

from test_core_host import ROWS, _ptr, _roots, core   # noqa: F401  (core: the fixture)

NAMES = ["quartic, pair", "quartic, reals, recollapsing", "cubic, pair", "quartic, seven columns"]


def _exact(P, z, grad):
    """chi, t, X and the density derivatives of chi and t."""
    mp.mp.dps = 40
    ncol = len(P)
    Om, OL, Or = (mp.mpf(v) for v in P[1:4])
    Ok = mp.mpf(P[4]) if ncol > 4 else 1 - Om - OL - Or
    Os, Ox = (mp.mpf(P[5]), mp.mpf(P[6])) if ncol == 7 else (mp.mpf(0), mp.mpf(0))
    g = lambda u: Or + u * (Om + u * (Ok + Os + u * (Ox + u * OL)))
    powers = [1, 4, 0, 2, 2, 3][:ncol - 1]
    dg = [lambda u, n=n: u ** n - (u * u if ncol == 4 else 0) for n in powers]
    lo = mp.sqrt(1 / (1 + mp.mpf(z)))   # u = v^2, decade by decade
    pts = [lo] + [mp.mpf(10) ** k for k in range(-58, 0, 2) if mp.mpf(10) ** k > 2 * lo] + [mp.mpf(1)]
    q = lambda f: mp.quad(lambda v: 2 * v * f(v * v), pts)
    val = [float(q(lambda u: w(u) / mp.sqrt(g(u)))) for w in (lambda u: 1, lambda u: u, lambda u: u ** -2)]
    if not grad:
        return np.array(val), None
    return np.array(val), np.array([[float(q(lambda u: -d(u) * w(u) / 2 * g(u) ** mp.mpf(-1.5))) for d in dg]
                                    for w in (lambda u: 1, lambda u: u)])


def _run(core, name, z, fp64):
    P = np.array(ROWS[name])
    quartic, cpair, roots, dr = _roots(ROWS[name])
    zz, out, grad = np.array([z]), np.zeros((1, 4)), np.zeros((1, 2, len(P) - 1))
    core.core_pairs(_ptr(P), len(P), quartic, cpair, _ptr(roots), _ptr(dr), fp64, 1, _ptr(zz), _ptr(out), _ptr(grad))
    return out[0], grad[0], [k for k in range(len(P) - 1) if quartic or k != 2]


@pytest.mark.parametrize("name", NAMES)
@pytest.mark.parametrize("z", [0.9e9, 1.1e9, 1e15, 1e19, 1e20, 1e29, 2e30, 1e100])
def test_double_precision(core, name, z):
    out, grad, cols = _run(core, name, z, 1)
    val, jac = _exact(ROWS[name], z, True)
    assert np.all(np.abs(out[:2] / val[:2] - 1) <= 1e-12)
    err = np.abs(grad[:, cols] - jac[:, cols]).max(axis=1) / np.abs(jac[:, cols]).max(axis=1)
    assert np.all(err <= 1e-9)


@pytest.mark.parametrize("name", NAMES)
@pytest.mark.parametrize("fp64,z", [(0, 6.4e4), (0, 6.6e4), (0, 1e9), (0, 1e12), (0, 1e15), (0, 1e18), (1, 0.9e9), (1, 1.1e9),
                                    (1, 1e20), (1, 2e30), (1, 1e100)])
def test_absorption_distance(core, name, fp64, z):
    """X grows like z: finite, and as accurate as at ordinary redshifts, FP64
    1e-12, FP32 1e-4."""
    z = z if fp64 else float(np.float32(z))
    out, _, _ = _run(core, name, z, fp64)
    val, _ = _exact(ROWS[name], z, False)
    assert abs(out[2] / val[2] - 1) <= (1e-12 if fp64 else 1e-4)
