"""General limits: a pair with z2 < z1 adds nothing to the gradient, whatever
outputs are differentiated."""
import numpy as np
import pytest

from paper_2212_01937_gb300 import workloads
from test_gpu_parity import _t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("names", [("mu",), ("d_C", "t", "d_M", "d_L", "mu"), ("X",), ("X", "mu"), ("X", "t", "d_M", "d_L", "mu")])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_outside_pairs_add_nothing(lib, prec, names):
    b = workloads.general_batch(B=3, n=1, seed=8)
    rng = np.random.default_rng(1)
    n, z1 = 60, np.array([0.3, 1.0, 2.5])
    z2 = z1[:, None] + rng.uniform(0.05, 2.0, (3, n))
    out = rng.random((3, n)) < 0.3
    z2[out] = (z1[:, None] * rng.uniform(0.0, 0.9, (3, n)))[out]
    dt = np.float64 if prec == "fp64" else np.float32
    cot = {o: rng.uniform(0.5, 1.5, (3, n)).astype(dt) for o in names}
    ins = ~out

    def run(m):
        off = np.concatenate([[0], np.cumsum(m.sum(axis=1))]).astype(np.int64)
        return lib.distances_between(_t(b.params), _t(z1), _t(z2[m].astype(dt)), _t(off), outputs=(),
                                     cot={o: _t(c[m]) for o, c in cot.items()}, precision=prec)["grad"].cpu().numpy()

    a, c = run(np.ones_like(out)), run(ins)
    # the same pairs in another order of summation (FP32: per-pair results may take another path, 3e-5)
    assert np.all(np.abs(a - c) <= (1e-12 if prec == "fp64" else 3e-5) * np.abs(c).max(axis=1, keepdims=True))
