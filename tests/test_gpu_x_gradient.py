"""Calls that differentiate X beside other work (value-only outputs, redshift
derivatives): one root preparation, whose records of both kinds serve the
launches; results as those of the calls apart."""
import numpy as np
import pytest
import torch

from paper_2212_01937_gb300 import workloads
from test_gpu_parity import TOL32, TOL64, _t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("B,n", [(1, 1), (5, 70), (3, 300), (16500, 3)])
def test_one_preparation(lib, B, n, prec):
    b = workloads.general_batch(B=min(B, 500), n=1, seed=4)
    P, off = _t(np.tile(b.params, (B // 500 + 1, 1))[:B]), _t(np.arange(B + 1, dtype=np.int64) * n)
    dt = torch.float64 if prec == "fp64" else torch.float32
    z = _t(np.random.default_rng(1).uniform(0.05, 3.0, B * n)).to(dt)
    cot = {"X": _t(np.random.default_rng(2).normal(size=B * n)).to(dt)}

    def launches(f):
        k = lib.launch_count()
        r = f()
        return r, lib.launch_count() - k

    both, k = launches(lambda: lib.distances_vjp(P, z, cot, off, outputs=("t", "X"), precision=prec))
    assert k == 3   # preparation, t, X with its gradient
    dz, k = launches(lambda: lib.distances_vjp(P, z, cot, off, outputs=("t", "X"), grad_z=True, precision=prec))
    assert k == 5   # the same, the redshift derivatives, and the rows that did not converge
    jac, k = launches(lambda: lib.distances_jac(P, z, off, outputs=("t", "X"), jac_outputs=("X",), precision=prec))
    assert k == 3
    t = lib.distances(P, z, off, outputs=("t",), precision=prec)["t"]
    x = lib.distances_vjp(P, z, cot, off, outputs=("X",), precision=prec)
    ref = lib.distances_vjp(P, z.double(), {"X": cot["X"].double()}, off, grad_z=True, precision="fp64")["grad_z"]
    tol = TOL64 if prec == "fp64" else TOL32
    for r in (both, dz, jac):
        assert int(r["status"].abs().sum()) == 0
        # (the roots of the X-tangent kernel's preparation are polished from a wider separation on)
        assert (r["t"] / t - 1).abs().max().item() <= 2 * tol["t"]
        assert torch.equal(r["X"], x["X"])
    for r in (both, dz):
        assert (r["grad"] - x["grad"]).abs().max().item() <= 1e-11 * x["grad"].abs().max().item()
    assert ((dz["grad_z"].double() - ref).abs() / ref.abs()).max().item() <= (1e-11 if prec == "fp64" else 4e-6)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_host_route(lib, prec):
    b = workloads.general_batch(B=40, n=30, seed=6)
    dt = torch.float64 if prec == "fp64" else torch.float32
    z, cot = torch.tensor(b.z).to(dt), torch.ones(b.z.size, dtype=dt)
    P, off = torch.tensor(b.params), torch.tensor(b.offsets)
    call = lib.HostVJP(40, z.numel(), outputs=("t", "X"), precision=prec, nchunks=1)
    k = lib.launch_count()
    r = call(P, z, {"X": cot}, off)
    assert lib.launch_count() - k == 3
    d = lib.distances_vjp(P.cuda(), z.cuda(), {"X": cot.cuda()}, off.cuda(), outputs=("t", "X"), precision=prec)
    for o in ("t", "X"):
        assert torch.equal(r[o], d[o].cpu())
    assert (r["grad"] - d["grad"].cpu()).abs().max().item() <= 1e-11 * d["grad"].abs().max().item()
