"""A pair that does not converge beside pairs that do: which of a row's pairs
are evaluated does not depend on when a warp enters the row."""
import numpy as np
import pytest
import torch

from test_gpu_parity import TOL32, TOL64, _t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deterministic", [False, True])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("outs", [("d_C",), ("d_C", "t"), ("X",)])
def test_bad_pair_seen_before_the_row_is_entered(lib, outs, prec, deterministic):
    """One warp per SM.  The second row starts at the end of the second warp's
    range; its NaN redshift is the first pair of the third warp, which marks the
    row long before the second warp gets there."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    chunk = 6400
    n, start, bad = sms * chunk, 2 * chunk - 100, 2 * chunk
    P = np.array([[70.0, 0.3, 0.7, 5e-5], [68.0, 0.32, 0.6, 9e-5]])
    off = np.array([0, start, n])
    z = np.random.default_rng(3).uniform(0.05, 2.0, n).astype(np.float32)
    z[bad] = 0.5
    zb = z.copy()
    zb[bad] = np.nan
    dt = np.float64 if prec == "fp64" else np.float32
    cot = {o: np.ones(n, dt) for o in outs}
    for c in cot.values():
        c[bad] = 0.0
    res = [lib.distances_vjp(_t(P), _t(v.astype(dt)), {o: _t(c) for o, c in cot.items()}, _t(off), outputs=outs, precision=prec,
                             block=32, blocks_per_sm=1, deterministic=deterministic) for v in (z, zb)]
    a, b = res
    assert a["status"].tolist() == [0, 0] and b["status"].tolist() == [0, 4]
    keep = np.arange(n) != bad
    for o in outs:
        va, vb = a[o].double().cpu().numpy(), b[o].double().cpu().numpy()
        assert np.isnan(vb[bad])
        assert np.abs(vb[keep] / va[keep] - 1).max() <= 2 * (TOL64 if prec == "fp64" else TOL32)[o]
    ga, gb = a["grad"].cpu().numpy(), b["grad"].cpu().numpy()
    # (the second warp's 100 pairs are 1e-4 of the row's sum)
    assert np.all(np.abs(ga - gb) <= 1e-5 * np.abs(ga).max(axis=1, keepdims=True))
