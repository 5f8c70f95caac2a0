"""Small E^2 at the lower limit on the GPU: general limits from a redshift at
which the universe loiters (next to the no-Big-Bang boundary), and rows whose
densities sum to little.  FP32 against FP64 on the same redshifts: values to
the bounds of any row, sums of derivatives finite and within 3e-5 + 1e-6 /
sqrt(E^2) of the row's largest (t: 1e-4 + ...)."""
import numpy as np
import pytest

from paper_2212_01937_gb300 import workloads
from test_gpu_parity import TOL32, _t

pytestmark = pytest.mark.gpu

OUTS = ("d_C", "t", "X")


def _compare(run, E2):
    for outs in (OUTS, ("d_C", "X")):
        a, b = run("fp32", outs, None), run("fp64", outs, None)
        assert not a["status"].any().item() and not b["status"].any().item()
        for o in outs:
            assert (a[o].double() / b[o] - 1).abs().max().item() <= TOL32[o], o
    for o, base in (("d_C", 3e-5), ("t", 1e-4)):
        a, b = (run(p, (), o)["grad"].cpu().numpy() for p in ("fp32", "fp64"))
        err = np.abs(a - b)[:, 1:].max(axis=1) / np.abs(b)[:, 1:].max(axis=1)
        assert np.all(err <= base + 2e-6 / 0.05 + 1e-6 / np.sqrt(E2)), (o, err)


@pytest.mark.parametrize("n", [7, 300])
def test_loitering(lib, n):
    rng = np.random.default_rng(14)
    P, z1, E2 = [], [], []
    while len(P) < 24:
        Om, Or = rng.uniform(0.05, 0.6), 10.0 ** rng.uniform(-5, -4)
        OL = workloads.ol_critical(Om, Or) * (1 - 10.0 ** rng.uniform(-8, -1))
        x = np.linspace(1.01, 8.0, 20000)
        e = Or * x ** 4 + Om * x ** 3 + (1 - Om - OL - Or) * x * x + OL
        if e.min() > 1e-8:
            P.append([70.0, Om, OL, Or])
            z1.append(x[e.argmin()] - 1)
            E2.append(e.min())
    P, z1 = np.array(P), np.array(z1)
    assert min(E2) < 1e-6
    z2 = (z1[:, None] + rng.uniform(0.05, 10.0, (len(P), n))).astype(np.float32).ravel()
    off = _t(np.arange(len(P) + 1, dtype=np.int64) * n)

    def run(prec, outs, cot):
        z = z2 if prec == "fp32" else z2.astype(np.float64)
        c = {cot: _t(np.ones_like(z))} if cot else None
        return lib.distances_between(_t(P), _t(z1), _t(z), off, outputs=outs, cot=c, precision=prec)

    _compare(run, np.array(E2))


@pytest.mark.parametrize("n", [7, 300])
def test_small_sum(lib, n):
    rng = np.random.default_rng(15)
    P, S = [], []
    while len(P) < 24:
        Om, OL, Or, s = rng.uniform(0.05, 1.0), rng.uniform(-0.3, 0.3), 10.0 ** rng.uniform(-5, -3), 10.0 ** rng.uniform(-8, -1)
        Ok = s - Om - OL - Or
        if 4 * Or + 3 * Om + 2 * Ok > 0.05:
            P.append([70.0, Om, OL, Or, Ok])
            S.append(s)
    P = np.array(P)
    z = rng.uniform(0.05, 10.0, len(P) * n).astype(np.float32)
    off = _t(np.arange(len(P) + 1, dtype=np.int64) * n)

    def run(prec, outs, cot):
        zz = _t(z if prec == "fp32" else z.astype(np.float64))
        if cot:
            return lib.distances_vjp(_t(P), zz, {cot: _t(np.ones(z.size, z.dtype if prec == "fp32" else np.float64))}, off,
                                     outputs=outs, precision=prec)
        return lib.distances(_t(P), zz, off, outputs=outs, precision=prec)

    _compare(run, np.array(S))


def test_small_sum_absorption(lib):
    """X far out: no product on the way flushes to zero (within 5e-6; 1e-6 is
    usual at sums of 1e-6 and more)."""
    rng = np.random.default_rng(16)
    P = []
    while len(P) < 300:
        Om, OL, Or, s = rng.uniform(0.05, 1.0), rng.uniform(-0.3, 0.3), 10.0 ** rng.uniform(-5, -3), 10.0 ** rng.uniform(-9, -6)
        Ok = s - Om - OL - Or
        if 4 * Or + 3 * Om + 2 * Ok > 0.05:
            P.append([70.0, Om, OL, Or, Ok])
    P, n = np.array(P), 8
    z = (10.0 ** rng.uniform(1.5, 3, len(P) * n)).astype(np.float32)
    off = _t(np.arange(len(P) + 1, dtype=np.int64) * n)
    a, b = (lib.distances(_t(P), _t(v), off, outputs=("X",), precision=p)["X"]
            for v, p in ((z, "fp32"), (z.astype(np.float64), "fp64")))
    assert (a.double() / b - 1).abs().max().item() <= 5e-6
