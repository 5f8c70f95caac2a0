"""Very large redshifts on the GPU, with small ones beside them (in one thread
of the packed kernel, rows of 256 and more): FP64 against 40-digit quadrature,
FP32 against FP64, to the bounds of ordinary redshifts."""
import numpy as np
import pytest

from test_core_host import ROWS
from test_core_large_z import NAMES, _exact
from test_gpu_parity import TOL32, TOL64, _t

pytestmark = pytest.mark.gpu

OUTS = ("d_C", "t", "X")
SCALE = np.array([299792.458, 977.7922216807891, 299792.458])


@pytest.mark.parametrize("name", NAMES)
def test_double_precision(lib, name):
    P = np.array([ROWS[name]])
    z = np.array([0.5, 0.9e9, 1.1e9, 1e15, 1e19, 1e25, 2e30])
    got = lib.distances(_t(P), _t(z), _t(np.array([0, z.size])), outputs=OUTS, precision="fp64")
    assert int(got["status"][0]) == 0
    for i, x in enumerate(z):
        val, _ = _exact(ROWS[name], float(x), False)
        for q, o in enumerate(OUTS):
            assert abs(got[o][i].item() / (val[q] * SCALE[q] / P[0, 0]) - 1) <= TOL64[o], (x, o)


@pytest.mark.parametrize("n", [40, 300])
@pytest.mark.parametrize("name", NAMES)
def test_single_precision(lib, name, n):
    P = np.array([ROWS[name]] * 2)
    rng = np.random.default_rng(8)
    z = np.where(rng.random(2 * n) < 0.5, 10.0 ** rng.uniform(-2, 3, 2 * n), 10.0 ** rng.uniform(4, 18, 2 * n)).astype(np.float32)
    off = _t(np.array([0, n, 2 * n]))
    for outs in (OUTS, ("d_C", "X")):
        got = lib.distances(_t(P), _t(z), off, outputs=outs, precision="fp32")
        ref = lib.distances(_t(P), _t(z.astype(np.float64)), off, outputs=outs, precision="fp64")
        assert got["status"].tolist() == [0, 0]
        for o in outs:
            assert (got[o].double() / ref[o] - 1).abs().max().item() <= TOL32[o], o
