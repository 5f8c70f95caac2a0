"""The root preparation on the GPU, with four lanes and with one lane per
cosmology (more than 16384 rows): status and values as test_prep_host.py has
them for the host build."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import COLS, TOL32, TOL64, _t
from test_prep_host import _double_root, _exact, _low_radiation, _status, _zero_root

pytestmark = pytest.mark.gpu


def _check(lib, P, well, z, prec, times):
    """Status of all rows, and d_C, t, X of the rows `well`, whose integrands are
    far from a root, to the bounds of any row."""
    rows, n = len(P), z.size
    P_, off = np.tile(P, (times, 1)), np.arange(rows * times + 1, dtype=np.int64) * n
    zz = np.tile(z, rows * times)
    zz = zz if prec == "fp64" else zz.astype(np.float32)
    got = lib.distances(_t(P_), _t(zz), _t(off), outputs=("d_C", "t", "X"), precision=prec)
    st = got["status"].cpu().numpy().reshape(times, rows)
    want = np.array([_status(row, *_exact(row)) for row in P])
    assert np.all(st == want), (P[(st != want).any(axis=0)].tolist(), want[(st != want).any(axis=0)])
    good = np.nonzero((want == 0) & well)[0]
    ref = oracle.quad_distances(P[good], np.tile(zz[:n].astype(np.float64), good.size),
                                np.arange(good.size + 1, dtype=np.int64) * n)
    tol = TOL64 if prec == "fp64" else TOL32
    for o in ("d_C", "t", "X"):
        v = got[o].double().cpu().numpy().reshape(times, rows, n)
        assert np.isnan(v[:, want != 0]).all()
        err = np.abs(v[:, good].reshape(times, -1) / ref[:, COLS[o]] - 1)
        assert err.max() <= tol[o], (o, err.max())


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("times", [1, 140])
@pytest.mark.parametrize("ncol", [4, 5, 7])
def test_nearly_double_roots(lib, ncol, times, prec):
    rng = np.random.default_rng(11)
    P = []
    for i in range(120):
        row = _double_root(rng, ncol, i % 4 < 2)
        row[2] *= 1.0 + 10.0 ** rng.uniform(-10, -5) * (1 if i % 2 else -1)
        P.append(row)
    P = np.array(P)
    # (values where the double root lies well below the range of integration)
    well = np.array([max(float(abs(x)) for x in re + cx if abs(x) < 20) < 0.8 for re, cx in map(_exact, P)])
    assert well.sum() >= 10
    _check(lib, P, well, np.array([0.01, 0.3, 1.0, 5.0, 300.0]), prec, times)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("times", [1, 140])
@pytest.mark.parametrize("ncol", [4, 5, 7])
def test_low_radiation(lib, ncol, times, prec):
    rng = np.random.default_rng(12)
    P = np.array([_low_radiation(rng, ncol) for _ in range(120)])
    _check(lib, P, np.full(len(P), True), np.array([0.01, 0.3, 1.0, 5.0, 300.0]), prec, times)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("times", [1, 140])
def test_zero_root(lib, times, prec):
    rng = np.random.default_rng(13)
    P = np.array([_zero_root(rng, i % 2) for i in range(120)])
    _check(lib, P, np.full(len(P), True), np.array([0.01, 0.3, 1.0, 5.0, 300.0]), prec, times)
