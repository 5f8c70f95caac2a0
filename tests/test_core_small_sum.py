"""The pair core (csrc/lcdm_core.cuh), compiled for the host, where E^2(0), the
sum of the densities of a row that does not close, is small (the cosmologies of
general limits from a loitering redshift are alike): deviations of the arguments
over z^2 of up to 1e8.  Against 40-digit quadrature.

Bounds: values as for any row, FP64 1e-12 and FP32 2e-6 (X 1e-4), plus 2e-16 / S,
the rounding of the sum S itself.  Gradients are dominated by d / dS, from the roots
1 - O(S): FP32 as for any row, 3e-5 (t: 1e-4) + 2e-6 / z, plus 1e-6 / sqrt(S)."""
import functools

import mpmath as mp
import numpy as np
import pytest

from test_core_host import _ptr, _roots, core   # noqa: F401  (core: the fixture)

# (Om, OL, Or, and Ok = S - the others), dE^2/dx(1) > 0
BASE = {"pair": (0.3, 0.1, 5e-5), "reals": (0.9, -0.2, 1e-4), "cubic": (0.5, 0.2, 0.0)}
Z = np.array([0.1, 300.0], np.float32).astype(np.float64)


def _row(name, S):
    Om, OL, Or = BASE[name]
    return [70.0, Om, OL, Or, S - Om - OL - Or]


@functools.lru_cache(maxsize=None)
def _exact(P, z):
    mp.mp.dps = 40
    Om, OL, Or, Ok = (mp.mpf(v) for v in P[1:])
    E2 = lambda x: OL + x * x * (Ok + x * (Om + x * Or))
    d = [lambda x: x ** 3, lambda x: mp.mpf(1), lambda x: x ** 4, lambda x: x ** 2]
    w = [lambda x: mp.mpf(1), lambda x: 1 / x, lambda x: x * x]
    z = mp.mpf(z)
    pts = [mp.mpf(0)] + [z * mp.mpf(10) ** k for k in range(-14, 1)]
    q = lambda f: mp.quad(lambda s: f(1 + s), pts, maxdegree=5)
    return (np.array([float(q(lambda x: f(x) / mp.sqrt(E2(x)))) for f in w]),
            np.array([[float(q(lambda x: -f(x) * g(x) / 2 * E2(x) ** mp.mpf(-1.5))) for g in d] for f in w[:2]]))


@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("S", [1e-2, 1e-4, 1e-6, 1e-8, 1e-10])
@pytest.mark.parametrize("name", BASE)
def test_small_sum(core, name, S, fp64):
    P = _row(name, S)
    quartic, cpair, roots, dr = _roots(P)
    z = Z
    out, grad = np.zeros((z.size, 4)), np.zeros((z.size, 2, 4))
    core.core_pairs(_ptr(np.array(P)), 5, quartic, cpair, _ptr(roots), _ptr(dr), fp64, z.size, _ptr(z), _ptr(out), _ptr(grad))
    assert not out[:, 3].any()
    cols = [0, 1, 2, 3] if quartic else [0, 1, 3]
    for i, x in enumerate(z):
        val, jac = _exact(tuple(P), float(x))
        tol = (np.full(3, 1e-12) if fp64 else np.array([2e-6, 2e-6, 1e-4])) + 2e-16 / S
        assert np.all(np.abs(out[i, :3] / val - 1) <= tol), (x, out[i, :3] / val - 1)
        if not fp64 and S >= 1e-8:
            err = np.abs(grad[i][:, cols] - jac[:, cols]).max(axis=1) / np.abs(jac[:, cols]).max(axis=1)
            assert np.all(err <= np.array([3e-5, 1e-4]) + 2e-6 / x + 1e-6 / np.sqrt(S)), (x, err)
