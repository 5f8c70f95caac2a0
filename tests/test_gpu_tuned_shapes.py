"""A tuned launch shape belongs to the kernel that it was tuned for."""
import numpy as np
import pytest
import torch

from paper_2212_01937_gb300 import workloads
from test_gpu_parity import _t

pytestmark = pytest.mark.gpu


def test_tuned_lane_map_stays_with_its_kernel(lib):
    """The packed kernel (rows of 1024), tuned with the interleaved lane map, and
    the kernel of short rows (128), as many pairs in all: the latter's sums, in
    deterministic mode, are bit for bit those of the default map."""
    rng = np.random.default_rng(0)

    def batch(B, n):
        b = workloads.general_batch(B=B, n=1, seed=9)
        z = rng.uniform(0.01, 3.0, B * n).astype(np.float32)
        # (over sixteen decades, so that the sums round and show their order)
        c = (rng.normal(size=B * n) * 10.0 ** rng.uniform(-8, 8, B * n)).astype(np.float32)
        return _t(b.params), _t(z), {"d_C": _t(c)}, _t(np.arange(B + 1, dtype=np.int64) * n)

    P, z, cot, off = batch(24, 1024)
    assert lib.autotune(P, z, off, outputs=("d_C",), cot=cot, lane_map="interleaved")["lane_map"] == "interleaved"
    P, z, cot, off = batch(192, 128)
    kw = dict(outputs=("d_C",), precision="fp32", deterministic=True, block=64, blocks_per_sm=1)
    by_map = {m: lib.distances_vjp(P, z, cot, off, lane_map=m, **kw)["grad"] for m in ("contiguous", "interleaved", "tuned")}
    assert not torch.equal(by_map["contiguous"], by_map["interleaved"])
    assert torch.equal(by_map["tuned"], by_map["contiguous"])
