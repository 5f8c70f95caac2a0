"""What the size queries ask for."""
import ctypes

import pytest

from test_abi import cdll   # noqa: F401  (the fixture)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("B", [1, 3, 4096])
def test_sizes(cdll, B, prec):
    from paper_2212_01937_gb300.lcdm import Opts
    i64, opts = ctypes.c_int64, ctypes.byref(Opts(4, prec, 0, 0, 0))

    def size(f, *n):
        b = ctypes.c_size_t()
        assert f(i64(B), *(i64(v) for v in n), opts, ctypes.byref(b)) == 0
        return b.value

    records = size(cdll.lcdm_workspace_size)
    # both kinds of records: the core's (260 numbers) and the X-tangent kernel's (120
    # doubles, in single precision also their two halves)
    assert records >= B * (260 * (4 if prec else 8) + 120 * 8 * (2 if prec else 1))
    # the redshift derivatives take the records alone, however many pairs
    assert size(cdll.lcdm_loglike_dz_workspace_size, 10) == size(cdll.lcdm_loglike_dz_workspace_size, 10 ** 6) == records
    # limits works in double precision whatever the precision asked for
    assert size(cdll.lcdm_between_workspace_size, 0) >= records + B * (4 * 4 + 1 + 2 + 4) * 8
