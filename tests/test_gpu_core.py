"""Routes of the pair kernels at the sizes where they change: two pairs in a
thread (single precision, mean row length of 256 and more) against one, for
row lengths around the batch and pair sizes, both lane maps and the shared
layout; the redshift derivatives in each kernel that gives them; general
limits; and rows with a non-finite redshift.

The reference is the FP64 path on the same (single-precision) redshifts, which
test_gpu_parity.py, test_gpu_between.py and test_bhm.py hold to the oracle at
1e-12 (gradients 1e-9 of the row).  Bounds are the FP32 path's per pair: values
as TOL32 (mu 1e-5 mag); a row's gradient sum_n cot_n d_n is within
sum_n |cot_n| jac_tol(z_n) max_k |d_nk| of it."""
import numpy as np
import pytest
import torch

from paper_2212_01937_gb300 import workloads

from test_gpu_parity import TOL32, _t, jac_tol

pytestmark = pytest.mark.gpu

VALS = ("d_C", "t", "d_M", "d_L", "mu")


def _close(got, ref, name, mask=None):
    got, ref = got.double().cpu().numpy(), ref.cpu().numpy()
    if mask is not None:
        got, ref = got[mask], ref[mask]
    if name == "mu":
        fin = np.isfinite(ref)
        assert np.array_equal(fin, np.isfinite(got))
        assert np.abs(got[fin] - ref[fin]).max() <= 2e-5
        return
    err = np.abs(got - ref) / np.maximum(np.abs(ref), 1e-30)
    assert err[ref != 0].max() <= TOL32[name], (name, err[ref != 0].max())
    assert not got[ref == 0].any()


def _batch(lens, seed, ncol=4, radiation=True):
    b = workloads.general_batch(B=len(lens), n=1, seed=seed)
    rng = np.random.default_rng(seed)
    P = b.params.copy()
    # redshifts to 3 and moderate curvature: no pair near an antipode
    P[:, 2] = np.minimum(P[:, 2], 0.9)
    if not radiation:
        P[:, 3] = 0.0
    if ncol == 5:
        P = np.concatenate([P, (1.0 - P[:, 1:4].sum(axis=1) + 0.02)[:, None]], axis=1)
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    z = rng.uniform(0.01, 3.0, offs[-1]).astype(np.float32)
    z[::211] = 0.0
    return P, z, offs, rng


def _grad_bound(lib, P, z, offs, cot, ncol):
    """FP64 gradient and the bound of its FP32 counterpart, per row and entry."""
    z64 = z.astype(np.float64)
    jac = lib.distances_jac(_t(P), _t(z64), _t(offs), outputs=(), jac_outputs=tuple(cot), precision="fp64")["jac"]
    rows = np.repeat(np.arange(len(P)), np.diff(offs))
    g, bound = np.zeros((len(P), ncol)), np.zeros(len(P))
    for o, c in cot.items():
        J, c = jac[o].cpu().numpy(), c.astype(np.float64)
        np.add.at(g, rows, c[:, None] * J)
        Jf = np.where(np.isfinite(J), J, 0.0)
        np.add.at(bound, rows, np.abs(c) * jac_tol("fp32", np.maximum(z64, 1e-2), o) * np.abs(Jf).max(axis=1))
    return g, bound[:, None]


# mean length >= 256: packed; the lengths around 32, 64 and an odd batch, with
# empty and single-pair rows between
LENS = [1024, 257, 0, 1, 63, 64, 65, 31, 33, 2000, 1500, 95, 97, 1]


@pytest.mark.parametrize("lane_map", ["contiguous", "interleaved"])
@pytest.mark.parametrize("ncol,radiation", [(4, True), (5, True), (4, False)])
def test_two_pairs_in_a_thread(lib, lane_map, ncol, radiation):
    P, z, offs, rng = _batch(LENS, 23, ncol, radiation)
    assert z.size >= 256 * len(LENS)
    z64 = z.astype(np.float64)
    cot = {o: rng.normal(size=z.size).astype(np.float32) for o in VALS}
    ref = lib.distances(_t(P), _t(z64), _t(offs), outputs=VALS, precision="fp64")
    for outputs in (VALS, ("d_C", "mu")):
        got = lib.distances(_t(P), _t(z), _t(offs), outputs=outputs, precision="fp32", lane_map=lane_map)
        for o in outputs:
            _close(got[o], ref[o], o)
    for names in (VALS, ("d_C", "mu")):
        cc = {o: cot[o] for o in names}
        got = lib.distances_vjp(_t(P), _t(z), {o: _t(c) for o, c in cc.items()}, _t(offs), outputs=names,
                                precision="fp32", lane_map=lane_map)
        for o in names:
            _close(got[o], ref[o], o)
        g, bound = _grad_bound(lib, P, z, offs, cc, ncol)
        got_g = got["grad"].cpu().numpy()
        assert np.array_equal(np.isnan(got_g), np.isnan(g))
        ok = np.isfinite(g)
        assert np.all((np.abs(got_g - g) <= bound)[ok])


@pytest.mark.parametrize("names", [("X",), ("t", "X", "mu")])
@pytest.mark.parametrize("ncol,radiation", [(4, True), (5, True), (4, False)])
def test_two_pairs_in_a_thread_absorption(lib, names, ncol, radiation):
    """X beside a pair that needs another number of steps (z over five decades
    in random order) and beside a NaN; general limits."""
    P, z, offs, rng = _batch(LENS, 29, ncol, radiation)
    z = np.where(z > 0, 10.0 ** rng.uniform(-3, 0.5, z.size), 0.0).astype(np.float32)
    bad = z.copy()
    bad[5] = np.nan
    z64 = z.astype(np.float64)
    ref = lib.distances(_t(P), _t(z64), _t(offs), outputs=names, precision="fp64")
    for lane_map in ("contiguous", "interleaved"):
        got = lib.distances(_t(P), _t(z), _t(offs), outputs=names, precision="fp32", lane_map=lane_map)
        nan = lib.distances(_t(P), _t(bad), _t(offs), outputs=names, precision="fp32", lane_map=lane_map)
        for o in names:
            _close(got[o], ref[o], o)
            assert np.isnan(nan[o][5].item())
            nan[o][5] = got[o][5]
            _close(nan[o], ref[o], o)
    z1 = _t(rng.uniform(0.0, 0.5, len(P)))
    z2 = (z + z1.cpu().numpy()[np.repeat(np.arange(len(P)), np.diff(offs))] + 0.05).astype(np.float32)
    got = lib.distances_between(_t(P), z1, _t(z2), _t(offs), outputs=names, precision="fp32")
    ref = lib.distances_between(_t(P), z1, _t(z2.astype(np.float64)), _t(offs), outputs=names, precision="fp64")
    for o in names:
        _close(got[o], ref[o], o)


@pytest.mark.parametrize("n", [255, 256, 1001])
def test_shared_layout_loglike(lib, n):
    """Below and from the packed kernel's line on; a shared redshift set."""
    P, z, _, rng = _batch([n], 5)
    P = np.concatenate([P, P * [1.01, 0.97, 1.0, 1.0]])
    z = np.maximum(z, 0.01).astype(np.float32)
    mu = lib.distances(_t(P[:1]), _t(z.astype(np.float64)), outputs=("mu",), precision="fp64")["mu"].cpu().numpy()
    m = (mu - 19.3 + rng.normal(0, 0.1, n)).astype(np.float32)
    kw = dict(M=-19.3, sigma=0.1, layout="shared", want_mu=True)
    a = lib.gauss_loglike(_t(P), _t(z), _t(m), precision="fp32", **kw)
    b = lib.gauss_loglike(_t(P), _t(z.astype(np.float64)), _t(m.astype(np.float64)), precision="fp64", **kw)
    _close(a["mu"], b["mu"], "mu")
    r = np.abs(np.tile(m.astype(np.float64), 2) - b["mu"].cpu().numpy() + 19.3) / 0.1
    # d loglike = |r| / sigma d mu, d mu <= 2e-5, plus the sums' own rounding
    bound = (r.reshape(2, n) * 2e-5 / 0.1 + 1e-6 * (1 + r.reshape(2, n) ** 2)).sum(axis=1)
    assert np.all(np.abs(a["loglike"].cpu().numpy() - b["loglike"].cpu().numpy()) <= bound)
    ga, gb = a["grad"].cpu().numpy(), b["grad"].cpu().numpy()
    jac = lib.distances_jac(_t(P), _t(z.astype(np.float64)), outputs=(), jac_outputs=("mu",), layout="shared",
                            precision="fp64")["jac"]["mu"].cpu().numpy().reshape(2, n, 4)
    big = np.abs(jac).max(axis=2)
    # the residual's error times the derivative, and the residual times the derivative's error
    gbound = ((2e-5 / 0.01 + r.reshape(2, n) / 0.1 * (3e-5 + 2e-6 / z)) * big).sum(axis=1)
    assert np.all(np.abs(ga - gb) <= gbound[:, None])


@pytest.mark.parametrize("lens", [[40, 1, 0, 33], [700, 300]])
@pytest.mark.parametrize("names", [("mu",), ("d_C", "t", "d_M", "d_L", "mu"), ("X", "d_C")])
def test_redshift_derivatives(lib, lens, names):
    """Beside the sums, beside the X-tangent kernel, and without a parameter
    gradient (alone, and with t and X among the outputs)."""
    P, z, offs, rng = _batch(lens, 31)
    z = np.maximum(z, 0.01).astype(np.float32)
    cot = {o: rng.normal(size=z.size).astype(np.float32) for o in names}
    ref = lib.distances_vjp(_t(P), _t(z.astype(np.float64)), {o: _t(c.astype(np.float64)) for o, c in cot.items()}, _t(offs),
                            grad_z=True, precision="fp64")
    import oracle
    d = oracle.dout_dz(P, z.astype(np.float64), offs)
    cols = {"d_C": 0, "t": 1, "X": 2, "d_M": 3, "d_L": 4, "mu": 5}
    want = sum(cot[o].astype(np.float64) * d[:, cols[o]] for o in names)
    size = sum(np.abs(cot[o].astype(np.float64) * d[:, cols[o]]) for o in names)
    assert np.all(np.abs(ref["grad_z"].cpu().numpy() - want) <= 1e-11 * size)
    for outputs in ((), ("t", "mu")):
        got = lib.distances_vjp(_t(P), _t(z), {o: _t(c) for o, c in cot.items()}, _t(offs), outputs=outputs, grad_z=True,
                                precision="fp32")
        assert np.all(np.abs(got["grad_z"].double().cpu().numpy() - want) <= 4e-6 * size)
        assert np.all(np.isfinite(got["grad"].cpu().numpy()))
    # values and redshift derivatives only (no parameter gradient), through the C interface
    import ctypes
    for prec, tol in (("fp64", 1e-11), ("fp32", 4e-6)):
        for outputs in ((), ("t", "X")):
            c = lib.Call(_t(P), _t(z), _t(offs), precision=prec)
            out, vp = c.out_buffers(outputs)
            cc = {o: _t(v).to(c.dtype) for o, v in cot.items()}
            cp = lib._VP6(*[(cc[o].data_ptr() if o in cc else None) for o in lib.OUTS])
            gz = torch.empty(c.npairs, dtype=c.dtype, device=c.device)
            ws = lib.loglike_dz_workspace(c)
            lib._check(lib.load().lcdm_distances_vjp_dz(*c.common(), cp, vp, None, lib._ptr(gz), lib._ptr(c.status),
                                                        ctypes.byref(c.opts), lib._ptr(ws), ws.numel(),
                                                        lib._stream(c.device)))
            torch.cuda.synchronize()
            assert np.all(np.abs(gz.double().cpu().numpy() - want) <= tol * size)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("lens", [[50, 60], [600, 500]])
def test_non_finite_redshift(lib, prec, lens):
    """One NaN redshift: its outputs are NaN, the pair beside it is not, the
    row's status is bad and all the row's redshift derivatives are NaN; the
    other row is untouched."""
    P, z, offs, rng = _batch(lens, 7)
    z = np.maximum(z, 0.01).astype(np.float32)
    bad = z.copy()
    bad[10] = np.nan
    dt = torch.float64 if prec == "fp64" else torch.float32
    m = torch.full((z.size,), 22.0, dtype=dt, device="cuda:0")
    res = [lib.gauss_loglike(_t(P), _t(v).to(dt), m, _t(offs), grad_z=True, want_mu=True, precision=prec) for v in (z, bad)]
    torch.cuda.synchronize()
    a, b = res
    assert b["status"].tolist()[0] != 0 and b["status"].tolist()[1] == 0
    mu_a, mu_b = a["mu"].cpu().numpy(), b["mu"].cpu().numpy()
    assert np.isnan(mu_b[10]) and np.all(np.isfinite(np.delete(mu_b, 10)))
    assert np.abs(np.delete(mu_b - mu_a, 10)).max() <= 2e-5
    gz = b["grad_z"].cpu().numpy()
    assert np.all(np.isnan(gz[:lens[0]])) and np.all(np.isfinite(gz[lens[0]:]))


@pytest.mark.parametrize("lens", [[40, 1, 33], [700, 300, 400]])
@pytest.mark.parametrize("names", [("d_C", "t", "d_M", "d_L", "mu"), ("X", "mu")])
def test_general_limits_routes(lib, lens, names):
    """Mapped in the pair kernels, and by the pair maps where X has tangents."""
    P, z, offs, rng = _batch(lens, 41)
    z1 = np.array([0.0, 0.7, 2.5])
    rows = np.repeat(np.arange(3), lens)
    z2 = (z1[rows] + np.maximum(z, 0.01)).astype(np.float32)
    z2[5] = z1[0]                 # an empty interval
    z2[-3] = 0.1                  # z2 < z1
    cot = {o: rng.normal(size=z.size).astype(np.float32) for o in names if o != "X" or len(names) == 2}
    kw = dict(outputs=names)
    a = lib.distances_between(_t(P), _t(z1), _t(z2), _t(offs), cot={o: _t(c) for o, c in cot.items()}, precision="fp32", **kw)
    b = lib.distances_between(_t(P), _t(z1), _t(z2.astype(np.float64)), _t(offs),
                              cot={o: _t(c.astype(np.float64)) for o, c in cot.items()}, precision="fp64", **kw)
    inside = z2 >= z1[rows]
    for o in names:
        assert np.all(np.isnan(a[o].cpu().numpy()[~inside]))
        _close(a[o], b[o], o, inside)
    ga, gb = a["grad"].cpu().numpy(), b["grad"].cpu().numpy()
    # per pair within 1e-4 + 2e-6/z' (X: 1e-3); hundreds of pairs of either sign
    # leave a sum of a few times their root-mean-square, against errors of which
    # all but a few are a hundredth of the bound
    assert np.all(np.abs(ga - gb) <= (2e-2 if "X" in names else 3e-3) * np.abs(gb).max(axis=1, keepdims=True) + 1e-6)
    v = lib.distances_between(_t(P), _t(z1), _t(z2), _t(offs), precision="fp32", **kw)
    for o in names:
        _close(v[o], b[o], o, inside)
