"""lcdm_roots: the kind of a row whose roots are not labelled is 0."""
import numpy as np
import pytest

from test_gpu_parity import _t

pytestmark = pytest.mark.gpu


def test_kind(lib):
    P = np.array([[70.0, 0.3, 0.7, 5e-5], [70.0, 2.0, 0.01, 5e-5], [70.0, 0.3, 0.7, 0.0], [70.0, 0.3, -0.2, 0.0],
                  [-1.0, 0.3, 0.7, 5e-5], [70.0, np.nan, 0.7, 5e-5], [70.0, 0.0, 0.7, 0.0], [70.0, 0.3, 0.7, -1e-4]])
    r = lib.roots(_t(P))
    assert r["status"].tolist() == [0, 0, 0, 0, 2, 2, 2, 2]
    assert r["kind"].tolist() == [0, 1, 2, 3, 0, 0, 0, 0]
