"""Workloads of the distance library, as its users run them.

Each case is one call (or one forward and backward pass) of the public Python
interface on seeded synthetic inputs of this repository's own configurations
(``workloads.py``: the flat radiationless cosmology, the general batch, the
ragged batch, the precision-stress set, general limits, ages, the supernova
model's latent redshifts) or of generic sizes.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes a case's inputs on the GPU, ``run`` makes one pass,
``exact`` gives the same outputs by Gauss-Legendre quadrature of the defining
integrals in 64 bits (plain torch), ``work`` the bytes and operations that
one pass cannot do without.

Gradients are taken through ``distances_autograd`` with float32 parameter
tensors, PyTorch's default type and the interface's default precision.
"""
import math

import numpy as np
import torch

from paper_2212_01937_gb300 import lcdm

C_KMS = 299792.458
HUBBLE_GYR = 977.7922216807891
ORDER = ("d_C", "t", "X", "d_M", "d_L", "mu")
COMMON = {"layout": "dense", "ncol": 4, "precision": "fp32", "cosmo": "general", "zmin": 1e-4, "zmax": 10.0,
          "grads": "", "outputs": "d_C,t,X,mu", "zlog": False, "zgrad": False}


def listed():
    return [
        # one step of a fit to a handful of standard candles: the smallest
        # call, bounded by launches and by the root solve's latency
        case("fit_1x64", "autograd", 1, 64, outputs="mu", grads="mu", zmin=0.01, zmax=1.5),
        # one flat radiationless cosmology, 10^4 redshifts in double precision
        # (the plain use of the method: a distance table)
        case("flat_fp64_1x10000", "forward", 1, 10_000, cosmo="flat", precision="fp64", outputs="d_C,mu",
             zmin=0.01, zmax=2.0),
        # the general batch of the benchmark: four outputs, three of them
        # differentiated
        case("general_4096x1024", "autograd", 4096, 1024, layout="csr", grads="d_C,t,mu"),
        # ragged rows of 1 to 10^5 redshifts (posterior samples with their own
        # data sets), distance moduli and their gradient
        case("ragged_16384", "autograd", 16384, 5, layout="ragged", outputs="mu", grads="mu", zmax=3.0),
        # forward values close to flatness and to the no-Big-Bang boundary,
        # z from 1e-4 to 1100, explicit curvature column: the largest batch
        # (no mu: these universes are seen past their antipodes, where it diverges)
        case("stress_10000x10000", "forward", 10_000, 10_000, cosmo="stress", ncol=5, outputs="d_C,t,X", zmax=1100.0,
             zlog=True),
        # latent redshifts of the supernova model: gradients with respect to
        # every redshift and to the cosmology, radiationless, 4 guide samples
        case("latent_4x1000000", "autograd", 4, 1_000_000, cosmo="radiationless", outputs="mu", grads="mu",
             zmin=0.01, zmax=1.5, zgrad=True),
        # guide samples over one shared supernova set, an odd number of both
        case("samples_251x100003", "autograd", 251, 100_003, layout="shared", outputs="mu", grads="mu", zmin=0.01,
             zmax=1.5),
        # distances between two redshifts (a lens or absorber at z1 per row)
        case("between_4096x1024", "between", 4096, 1024, outputs="d_C,t,mu"),
        # ages and particle horizons with their gradients, double precision
        case("limits_65536", "limits", 65536, 0, precision="fp64"),
        # the general batch in double precision
        case("general_fp64_1024x1024", "forward", 1024, 1024, precision="fp64", layout="csr"),
        # the Gaussian log-likelihood of magnitudes and its gradient in double
        # precision (a final posterior evaluation)
        case("loglike_fp64_64x10000", "loglike", 64, 10_000, layout="shared", precision="fp64", zmin=0.01, zmax=1.5),
        # per-pair Jacobians (Fisher matrices), explicit curvature column
        case("fisher_500x1000", "jac", 500, 1000, ncol=5, outputs="d_C,mu", zmax=3.0),
    ]


def case(name, op, B, n, **kw):
    c = dict(COMMON, name=name, op=op, B=int(B), n=int(n))
    c.update(kw)
    return c


def draw(rng):
    def logi(lo, hi):
        return max(int(lo), min(int(hi), int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    op = rng.choice(("autograd", "autograd", "autograd", "forward", "forward", "jac", "between", "limits", "loglike"))
    if op == "limits":
        c = case("", op, logi(1, 131072), 0, precision="fp64")
    elif op == "loglike":
        B = logi(1, 300)
        c = case("", op, B, logi(1, 600_000 // B), layout=rng.choice(("shared", "dense")), precision="fp64", zmin=0.01,
                 zmax=1.5)
    elif op == "jac":
        p = rng.choice(("fp32", "fp32", "fp64"))
        B = logi(1, 2000)
        c = case("", op, B, logi(1, (1_000_000 if p == "fp32" else 150_000) // B), ncol=rng.choice((4, 5, 7)),
                 precision=p, outputs=rng.choice(("d_C,mu", "d_C,t,mu", "mu")), zmax=rng.uniform(1.0, 10.0))
        if c["ncol"] == 7:
            c["cosmo"] = "mixture"
    elif op == "between":
        B = logi(1, 16384)
        c = case("", op, B, logi(1, 8_000_000 // B), precision=rng.choice(("fp32", "fp32", "fp32", "fp64")),
                 outputs=rng.choice(("d_C,t,mu", "d_C,d_M,mu", "d_C")))
        if c["precision"] == "fp64":
            c["n"] = max(1, c["n"] // 10)
    elif op == "forward":
        p = rng.choice(("fp32", "fp32", "fp64"))
        B = logi(1, 16384)
        c = case("", op, B, logi(1, max(2, (50_000_000 if p == "fp32" else 1_000_000) // B)), precision=p,
                 layout=rng.choice(("dense", "csr", "shared")), cosmo=rng.choice(("general", "general", "radiationless")),
                 outputs=rng.choice(("d_C,t,X,mu", "d_C,mu", "d_C,t", "d_M,d_L", "X")), zmax=rng.choice((2.0, 10.0, 1100.0)))
        c["zlog"] = c["zmax"] > 100.0
        if c["cosmo"] == "radiationless" and "X" in c["outputs"]:
            c["outputs"] = "d_C,t,mu"   # X of a nearly empty radiationless universe is ill-conditioned
    else:
        B = logi(1, 16384)
        layout = rng.choice(("dense", "csr", "shared", "ragged"))
        c = case("", op, B, logi(1, max(2, 40_000_000 // B)), layout=layout, zmax=rng.choice((1.5, 3.0, 10.0)), zmin=0.01,
                 ncol=rng.choice((4, 4, 5)), cosmo=rng.choice(("general", "general", "radiationless")))
        c["outputs"], c["grads"] = rng.choice((("mu", "mu"), ("mu", "mu"), ("d_C,t,mu", "d_C,t,mu"),
                                               ("d_C,t,X,mu", "d_C,t,mu"), ("d_C,d_L", "d_C,d_L")))
        if layout == "ragged":
            # n is the largest exponent of a row's length, as in the ragged batch
            c["n"] = max(1, min(5, int(math.log10(max(10, 40_000_000 // B)))))
        elif layout != "shared":
            c["zgrad"] = rng.random() < 0.4
        if c["cosmo"] == "radiationless" and "X" in c["outputs"]:
            c["outputs"] = "d_C,t,mu"
    c.pop("name")
    return c


# ------------------------------------------------------------------ inputs ---
def cosmologies(kind, B, ncol, rng, zmax):
    """[B, ncol] parameter rows of a kind; all rows have a Big Bang and, but
    for the stress set, no antipode of the observer within zmax (mu diverges there)."""
    if kind == "flat":
        return np.tile(np.array([[70.0, 0.3, 0.7, 0.0]]), (B, 1))
    if kind == "stress":
        # half within 1e-6 of flatness, half just inside the no-Big-Bang boundary
        H0, Om, Or = rng.uniform(60, 80, B), rng.uniform(0.05, 0.6, B), 10.0 ** rng.uniform(-5, -4, B)
        Ok = rng.uniform(-1e-6, 1e-6, B)
        OL = 1.0 - Om - Or - Ok
        edge = np.arange(B) % 2 == 1
        OLc = critical_OL(Om, Or) * (1.0 - rng.uniform(1e-9, 1e-6, B))
        OL = np.where(edge, OLc, OL)
        Ok = np.where(edge, 1.0 - Om - OL - Or, Ok)
        return np.stack([H0, Om, OL, Or, Ok], axis=1)
    rows = np.zeros((0, ncol))
    a = np.linspace(0.0, 1.0, 257)[1:]
    while rows.shape[0] < B:
        m = 5 * (B - rows.shape[0]) // 4 + 16
        H0, Om, OL = rng.uniform(60, 80, m), rng.uniform(0.05, 0.6, m), rng.uniform(0.0, 1.2, m)
        Or = 10.0 ** rng.uniform(-5, -4, m) if kind != "radiationless" else np.zeros(m)
        Os = rng.uniform(-0.05, 0.2, m) if ncol == 7 else np.zeros(m)
        Ox = rng.uniform(-0.05, 0.2, m) if ncol == 7 else np.zeros(m)
        Ok = 1.0 - Om - OL - Or - Os - Ox
        Q = np.min(Or[:, None] / a + Om[:, None] + (Ok + Os)[:, None] * a + Ox[:, None] * a ** 2
                   + OL[:, None] * a ** 3, axis=1)
        ok = (Q > 1e-3) & (np.sqrt(np.maximum(-Ok, 0.0)) * horizon(Om, OL, Or, Ok + Os, Ox, zmax) < 2.6)
        if ncol == 7:
            r = roots_x(np.stack([H0, Om, OL, Or, Ok, Os, Ox], axis=1))
            ok &= np.sum(np.abs(r.imag) < 1e-9 * np.abs(r), axis=1) >= 2
        cols = [H0, Om, OL, Or, Ok, Os, Ox][:ncol]
        rows = np.concatenate([rows, np.stack(cols, axis=1)[ok]])
    return rows[:B]


def horizon(Om, OL, Or, Oks, Ox, zmax):
    """H0 / c times the comoving distance to zmax per row, by the midpoint rule in log(1 + z)."""
    n = 96
    h = math.log1p(zmax) / n
    x = np.exp((np.arange(n) + 0.5) * h)
    E2 = (((Or[:, None] * x + Om[:, None]) * x + Oks[:, None]) * x + Ox[:, None]) * x + OL[:, None]
    return h * np.sum(x / np.sqrt(np.maximum(E2, 1e-6)), axis=1)


def critical_OL(Om, Or):
    """Largest Omega_L0 (closure) with a Big Bang: E^2 has a double root at
    a in (0, 1), where Q = Q' = 0 is linear in (Om, OL); bisection on a."""
    def solve(a):
        # Om (a - a^2) + OL (a^4 - a^2) = -(Or + (1 - Or) a^2);  Om (1 - 2a) + OL (4 a^3 - 2a) = -2 (1 - Or) a
        A, B_, C, D = a - a * a, a ** 4 - a * a, 1 - 2 * a, 4 * a ** 3 - 2 * a
        e, f = -(Or + (1 - Or) * a * a), -2 * (1 - Or) * a
        det = A * D - B_ * C
        return (e * D - B_ * f) / det, (A * f - e * C) / det
    lo, hi = np.full_like(Om, 1e-3), np.full_like(Om, 0.999)   # Om grows with a on the loitering branch
    for _ in range(80):
        mid = 0.5 * (lo + hi)
        up = solve(mid)[0] < Om
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
    return solve(0.5 * (lo + hi))[1]


def densities(P):
    """Columns (Om, OL, Or, Ok, Os, Ox) of parameter rows, double precision numpy."""
    P = np.asarray(P, dtype=np.float64)
    Ok = P[:, 4] if P.shape[1] >= 5 else 1.0 - P[:, 1] - P[:, 2] - P[:, 3]
    z = np.zeros(P.shape[0])
    return P[:, 1], P[:, 2], P[:, 3], Ok, (P[:, 5] if P.shape[1] == 7 else z), (P[:, 6] if P.shape[1] == 7 else z)


def roots_x(P):
    """Roots of E^2 in x = 1 + z, [B, 4] complex (approximate: for choosing coordinates only)."""
    Om, OL, Or, Ok, Os, Ox = densities(P)
    out = np.zeros((P.shape[0], 4), dtype=np.complex128)
    for quartic in (True, False):
        rows = np.nonzero((Or > 0) == quartic)[0]
        if not rows.size:
            continue
        c = [OL, Ox, Ok + Os, Om, Or][:5 if quartic else 4]
        n = len(c) - 1
        M = np.zeros((rows.size, n, n))
        M[:, np.arange(1, n), np.arange(n - 1)] = 1.0
        for k in range(n):
            M[:, k, n - 1] = -c[k][rows] / c[n][rows]
        out[rows, :n] = np.linalg.eigvals(M)
    return out


def lengths(c, rng):
    if c["layout"] == "ragged":
        # the set of lengths belongs to the case, their order to the seed
        own = np.random.default_rng([c["B"], c["n"]])
        return rng.permutation(np.floor(10.0 ** own.uniform(0.0, float(c["n"]), c["B"])).astype(np.int64))
    return np.full(c["B"], c["n"], dtype=np.int64)


def device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def normals(n, gen, dtype, dev):
    return torch.randn(n, generator=gen, dtype=dtype, device=dev)


def inputs(c, seed):
    """The tensors of a case: params, z, offsets, and what its op needs beside them."""
    dev = device()
    rng = np.random.default_rng([int(seed), c["B"], c["n"], c["ncol"]])
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + c["B"] + c["n"])
    T = torch.float64 if c["precision"] == "fp64" else torch.float32
    P = cosmologies(c["cosmo"], c["B"], c["ncol"], rng, c["zmax"] + (3.0 if c["op"] == "between" else 0.0))
    s = {"case": c, "params": torch.tensor(P, dtype=torch.float64, device=dev)}
    if c["op"] == "limits":
        z1 = np.where(np.arange(c["B"]) % 2 == 0, rng.uniform(0, 10, c["B"]),
                      10.0 ** rng.uniform(1.0, math.log10(1100.0), c["B"]))
        s["z1"] = torch.tensor(z1, device=dev)
        s["cot_chi"], s["cot_t"] = (normals(c["B"], gen, torch.float64, dev) for _ in range(2))
        return s
    lens = lengths(c, rng)
    nz = c["n"] if c["layout"] == "shared" else int(lens.sum())
    u = torch.rand(nz, generator=gen, dtype=T, device=dev)
    if c["zlog"]:
        z = torch.exp(u * (math.log(c["zmax"]) - math.log(c["zmin"])) + math.log(c["zmin"]))
    else:
        z = u * (c["zmax"] - c["zmin"]) + c["zmin"]
    if c["op"] == "between":
        z1 = rng.uniform(0.0, 3.0, c["B"])
        s["z1"] = torch.tensor(z1, device=dev)
        z = (z + torch.repeat_interleave(s["z1"].to(T), c["n"])).to(T)
    s["z"] = z
    s["lens"] = lens
    if c["layout"] in ("csr", "ragged"):
        s["offsets"] = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int64, device=dev)
    if c["op"] == "loglike":
        q0 = 0.5 * 0.3 - 0.7
        mu = 5.0 * torch.log10(C_KMS * z / 70.0 * (1.0 + 0.5 * (1.0 - q0) * z)) + 25.0
        s["m_obs"] = mu - 19.3 + 0.1 * normals(nz, gen, T, dev)
    if c["op"] == "autograd":
        npairs = c["B"] * c["n"] if c["layout"] == "shared" else nz
        s["params"] = s["params"].to(torch.float32).requires_grad_()
        if c["zgrad"]:
            s["z"] = z.requires_grad_()
        # gradients that arrive from the rest of the model: standardised residuals
        s["cot"] = {o: normals(npairs, gen, T, dev) for o in c["grads"].split(",")}
    return s


def prepare(c, seed):
    return inputs(dict(COMMON, **c), seed)


# -------------------------------------------------------------------- a pass ---
def run(s):
    c = s["case"]
    outs = tuple(c["outputs"].split(","))
    layout = "csr" if c["layout"] == "ragged" else c["layout"]
    kw = {"layout": layout, "precision": c["precision"]}
    if c["op"] == "forward":
        return lcdm.distances(s["params"], s["z"], s.get("offsets"), outputs=outs, **kw)
    if c["op"] == "jac":
        return lcdm.distances_jac(s["params"], s["z"], s.get("offsets"), outputs=outs, **kw)
    if c["op"] == "between":
        return lcdm.distances_between(s["params"], s["z1"], s["z"], s.get("offsets"), outputs=outs, **kw)
    if c["op"] == "limits":
        return lcdm.limits(s["params"], s["z1"], s["cot_chi"], s["cot_t"], grad=True)
    if c["op"] == "loglike":
        return lcdm.gauss_loglike(s["params"], s["z"], s["m_obs"], s.get("offsets"), M=-19.3, sigma=0.1, grad=True, **kw)
    res = lcdm.distances_autograd(s["params"], s["z"], s.get("offsets"), outputs=outs, **kw)
    out = dict(zip(outs, res))
    wrt = [s["params"]] + ([s["z"]] if c["zgrad"] else [])
    g = torch.autograd.grad([out[o] for o in s["cot"]], wrt, [s["cot"][o] for o in s["cot"]])
    out = {o: v.detach() for o, v in out.items()}
    out["grad"] = g[0]
    if c["zgrad"]:
        out["grad_z"] = g[1]
    return out


# ---------------------------------------------------------------- 64 bits ---
def gauss(n, dev):
    x, w = np.polynomial.legendre.leggauss(n)
    return torch.tensor(x, device=dev), torch.tensor(w, device=dev)


def coordinates(P):
    """Per row (x0, d) of the map x = x0 + d sinh(u): the complex roots of E^2 sit at u = +-i pi/2."""
    r = roots_x(P)
    cplx = np.abs(r.imag) > 1e-12 * np.abs(r)
    k = np.argmin(np.where(cplx, np.abs(r - 1.0), np.inf), axis=1)
    pick = r[np.arange(r.shape[0]), k]
    any_c = cplx.any(axis=1)
    return np.where(any_c, pick.real, 0.0), np.where(any_c, np.maximum(np.abs(pick.imag), 1e-9), 1.0)


def du_of(a, b, ba):
    """asinh(b) - asinh(a) for b - a = ba >= 0, without cancellation."""
    ca, cb = torch.sqrt(1.0 + a * a), torch.sqrt(1.0 + b * b)
    same = a * b > 0
    close = torch.asinh(torch.where(same, ba * (a + b) / torch.where(same, b * ca + a * cb, torch.ones_like(a)), 0.0 * a))
    return torch.where(same, close, torch.asinh(b) - torch.asinh(a))


def curvature_map(D, Ok):
    """S_k(D), dS/dD, dS/dOk."""
    u = Ok * D * D
    small = u.abs() < 1e-2
    r = torch.sqrt(torch.where(small, torch.ones_like(u), Ok.abs()))
    y = r * D
    pos = Ok > 0
    S = torch.where(pos, torch.sinh(y), torch.sin(y)) / r
    SD = torch.where(pos, torch.cosh(y), torch.cos(y))
    Sk = (D * SD - S) / torch.where(small, torch.ones_like(u), 2.0 * Ok)
    s = sd = sk = torch.zeros_like(u)
    for i in range(8, -1, -1):
        s = 1.0 / math.factorial(2 * i + 1) + u * s
        sd = 1.0 / math.factorial(2 * i) + u * sd
        if i:
            sk = i / math.factorial(2 * i + 1) + u * sk
    return torch.where(small, D * s, S), torch.where(small, sd, SD), torch.where(small, D ** 3 * sk, Sk)


class Pairs:
    """Distances of a chunk of pairs by quadrature: the outputs `names`, their
    derivatives with respect to the parameters (those in `tangents`) and to z."""

    def __init__(self, row, x1, z, names, tangents, ncol, nodes, want_dz=False):
        # row: columns (H0, Om, OL, Or, Ok, Os, Ox, x0, d) of each pair; x1 = 1 + lower limit; z: the interval's length
        H0, Om, OL, Or, Ok, Os, Ox, x0, d = row.unbind(1)
        dev = z.device
        y, w = gauss(nodes, dev)
        a, b = (x1 - x0) / d, (x1 + z - x0) / d
        ua, du = torch.asinh(a), du_of(a, b, z / d)
        e = torch.exp((ua + 0.5 * du)[:, None] + 0.5 * du[:, None] * y)
        ie = 1.0 / e
        x = x0[:, None] + d[:, None] * (0.5 * (e - ie))
        jac = (0.25 * d * du)[:, None] * (e + ie)
        E2 = (((Or[:, None] * x + Om[:, None]) * x + (Ok + Os)[:, None]) * x + Ox[:, None]) * x + OL[:, None]
        iE = torch.rsqrt(E2)
        f0 = iE * jac
        wanted = set(names) | set(tangents)
        dist = wanted & {"d_C", "d_M", "d_L", "mu"}
        power = {"chi": None, "t": -1, "X": 2}
        kinds = (["chi"] if dist else []) + (["t"] if "t" in wanted else []) + (["X"] if "X" in wanted else [])
        I, dI = {}, {}
        g = -0.5 * f0 * iE * iE if tangents else None
        for k in kinds:
            m = None if power[k] is None else (1.0 / x if power[k] < 0 else x * x)
            I[k] = (f0 if m is None else f0 * m) @ w
            if tangents and (k != "chi" and k in tangents or k == "chi" and dist & set(tangents)):
                gk = g if m is None else g * m
                x2 = x * x
                basis = [x2 * x, None, x2 * x2, x2, x2, x][:ncol - 1]
                cl = (gk * x2) @ w if ncol == 4 else 0.0
                dI[k] = [(gk @ w if q is None else (gk * q) @ w) - cl for q in basis]
        DH, tH = C_KMS / H0, HUBBLE_GYR / H0
        s, x2_ = x1, x1 + z
        self.v, self.d, self.dz = {}, {}, {}
        iEz = torch.rsqrt((((Or * x2_ + Om) * x2_ + Ok + Os) * x2_ + Ox) * x2_ + OL)
        if dist:
            D = I["chi"]
            S, SD, Sk = curvature_map(D, Ok)
            self.v["d_C"], self.v["d_M"] = DH * D, DH * S
            fac = x2_ / (s * s)
            self.v["d_L"] = fac * self.v["d_M"]
            self.v["mu"] = 5.0 * torch.log10(self.v["d_L"]) + 25.0
            if "chi" in dI:
                dOk = [-1.0 if ncol == 4 else (1.0 if k == 3 else 0.0) for k in range(ncol - 1)]
                dC = dI["chi"]
                dM = [SD * q + Sk * o for q, o in zip(dC, dOk)]
                self.d["d_C"] = [-self.v["d_C"] / H0] + [DH * q for q in dC]
                self.d["d_M"] = [-self.v["d_M"] / H0] + [DH * q for q in dM]
                self.d["d_L"] = [fac * q for q in self.d["d_M"]]
                self.d["mu"] = [5.0 / math.log(10.0) * q / self.v["d_M"] for q in self.d["d_M"]]
            if want_dz:
                self.dz["d_C"], self.dz["d_M"] = DH * iEz, DH * SD * iEz
                self.dz["d_L"] = self.v["d_M"] + x2_ * self.dz["d_M"]
                self.dz["mu"] = 5.0 / math.log(10.0) * (1.0 / x2_ + SD * iEz / S)
        for k, pre in (("t", tH), ("X", DH)):
            if k in I:
                self.v[k] = pre * I[k]
                if k in dI:
                    self.d[k] = [-self.v[k] / H0] + [pre * q for q in dI[k]]
                if want_dz:
                    self.dz[k] = pre * iEz * (1.0 / x2_ if k == "t" else x2_ * x2_)


def exact(c, seed):
    c = dict(COMMON, **c)
    with torch.no_grad():
        s = inputs(c, seed)
        return exact_limits(c, s) if c["op"] == "limits" else exact_pairs(c, s)


def exact_pairs(c, s):
    P = s["params"].detach().double()
    dev, B, ncol = P.device, c["B"], c["ncol"]
    Pn = P.cpu().numpy()
    x0, d = coordinates(Pn)
    cols = np.stack([Pn[:, 0], *densities(Pn), x0, d], axis=1)
    rows = torch.tensor(cols, device=dev)
    z = s["z"].detach().double()
    z1 = s["z1"] if c["op"] == "between" else torch.zeros(B, dtype=torch.float64, device=dev)
    shared = c["layout"] == "shared"
    npairs = B * c["n"] if shared else z.numel()
    offs = torch.tensor(np.concatenate([[0], np.cumsum(s["lens"])]), device=dev)
    outs = c["outputs"].split(",")
    fp64 = c["precision"] == "fp64"
    nodes = 96 if (fp64 or c["cosmo"] == "stress") else 48
    if c["op"] == "loglike":
        names, tang = ["mu"], ["mu"]
    elif c["op"] == "jac":
        names, tang = outs, outs
    else:
        names, tang = outs, list(s.get("cot", {}))
    T = torch.float64 if fp64 else torch.float32
    keep = outs if c["op"] != "loglike" else []
    out = {o: torch.empty(npairs, dtype=torch.float64, device=dev) for o in keep}
    jac = {o: torch.empty(npairs, ncol, dtype=torch.float64, device=dev) for o in (outs if c["op"] == "jac" else [])}
    grad = torch.zeros(B, ncol, dtype=torch.float64, device=dev)
    ll = torch.zeros(B, dtype=torch.float64, device=dev)
    gz = torch.empty(npairs if c["zgrad"] else 0, dtype=torch.float64, device=dev)
    step = 2 ** 24 // nodes
    for p0 in range(0, npairs, step):
        p1 = min(npairs, p0 + step)
        p = torch.arange(p0, p1, device=dev)
        b = torch.div(p, c["n"], rounding_mode="floor") if shared else torch.searchsorted(offs, p, right=True) - 1
        zi = p - b * c["n"] if shared else p
        zp = z[zi] - z1[b]
        q = Pairs(rows[b], 1.0 + z1[b], zp, names, tang, ncol, nodes, c["zgrad"])
        for o in keep:
            out[o][p0:p1] = q.v[o]
        for o in jac:
            jac[o][p0:p1] = torch.stack(q.d[o], dim=1)
        if c["op"] == "loglike":
            r = (s["m_obs"][zi].double() - q.v["mu"] + 19.3) / 0.1
            ll.index_add_(0, b, -0.5 * r * r - math.log(0.1 * math.sqrt(2.0 * math.pi)))
            grad.index_add_(0, b, torch.stack([r / 0.1 * g for g in q.d["mu"]], dim=1))
        elif "cot" in s:
            g = 0.0
            for o, ct in s["cot"].items():
                g = g + torch.stack(q.d[o], dim=1) * ct[p0:p1].double()[:, None]
            grad.index_add_(0, b, g)
            if c["zgrad"]:
                gz[p0:p1] = sum(ct[p0:p1].double() * q.dz[o] for o, ct in s["cot"].items())
        del q
    # a radiationless universe has no Omega_r direction in the cubic reduction
    norad = torch.tensor(Pn[:, 3] == 0.0, device=dev)
    if c["op"] == "jac":
        out["jac"] = jac
    if c["op"] == "loglike":
        grad[norad, 3] = float("nan")
        out = {"loglike": ll, "grad": grad}
    if c["op"] == "autograd":
        grad[norad, 3] = float("nan")
        out["grad"] = grad
        if c["zgrad"]:
            out["grad_z"] = gz
    else:
        out["status"] = None
    return out


def exact_limits(c, s):
    """chi(z1, inf) and t(z1, inf) as integrals over a = 1 / (1 + z) = v^2, v = v0 sinh(u)."""
    Pn = s["params"].cpu().numpy()
    dev = s["params"].device
    Om, OL, Or, Ok, Os, Ox = (torch.tensor(v, device=dev)[:, None] for v in densities(Pn))
    H0 = s["params"][:, 0]
    v0 = torch.sqrt(Or / Om)
    vend = torch.sqrt(1.0 / (1.0 + s["z1"]))[:, None]
    uend = torch.asinh(vend / v0)
    y, w = gauss(48, dev)
    panels = 8
    chi = torch.zeros_like(H0)
    age = torch.zeros_like(H0)
    dchi, dage = [0.0] * 3, [0.0] * 3
    for k in range(panels):
        u = uend * ((k + 0.5 + 0.5 * y) / panels)
        v = v0 * torch.sinh(u)
        a = v * v
        jac = 2.0 * v * v0 * torch.cosh(u) * uend * (0.5 / panels)
        Q = Or + a * (Om + a * ((Ok + Os) + a * (Ox + a * OL)))
        iQ = torch.rsqrt(Q)
        f = iQ * jac
        chi = chi + f @ w
        age = age + (f * a) @ w
        g = -0.5 * f * iQ * iQ
        for j, b in enumerate((a, a ** 4, torch.ones_like(a))):
            q = g * (b - a * a)
            dchi[j] = dchi[j] + q @ w
            dage[j] = dage[j] + (q * a) @ w
    DH, tH = C_KMS / H0, HUBBLE_GYR / H0
    cc, ct = s["cot_chi"], s["cot_t"]
    g = [-(cc * DH * chi + ct * tH * age) / H0] + [cc * DH * x + ct * tH * t for x, t in zip(dchi, dage)]
    return {"chi_inf": DH * chi, "t_inf": tH * age, "grad": torch.stack(g, dim=1), "status": None}


# -------------------------------------------------------------------- work ---
#: floating-point operations per pair and integral that the reduction to
#: Carlson integrals cannot do without (Carlson's duplication in single
#: precision, one shared sequence, real symmetric functions of the root pair;
#: twice the steps in double precision); a gradient at twice the value's work
#: (reverse mode), whatever the number of parameters.
FLOPS = {"chi": 120.0, "t": 90.0, "X": 160.0, "map": 40.0}


def work(c):
    c = dict(COMMON, **c)
    es = 8 if c["precision"] == "fp64" else 4
    two = 2.0 if c["precision"] == "fp64" else 1.0
    root = 1500.0
    if c["op"] == "limits":
        # rows in; age, horizon, gradient out; value and gradient of two integrals per row
        return {"bytes": c["B"] * 8.0 * (4 + 3 + 2 + 4), "flops": c["B"] * (root + two * 3.0 * (FLOPS["chi"] + FLOPS["t"]))}
    B, ncol = c["B"], c["ncol"]
    if c["layout"] == "ragged":
        # expected length of a row: floor(10^U(0, n))
        npairs = nz = B * (10.0 ** c["n"] - 1.0) / (c["n"] * math.log(10.0))
    else:
        npairs = float(B) * c["n"]
        nz = c["n"] if c["layout"] == "shared" else npairs
    outs = c["outputs"].split(",") if c["op"] != "loglike" else ["mu"]
    grads = outs if c["op"] in ("jac", "loglike") else [o for o in c["grads"].split(",") if o]
    flops = 0.0
    for names, f in ((outs, 1.0), (grads, 2.0)):
        dist = [o for o in names if o not in ("t", "X")]
        flops += f * ((FLOPS["chi"] if dist else 0.0) + (FLOPS["map"] if set(dist) - {"d_C"} else 0.0)
                      + (FLOPS["t"] if "t" in names else 0.0) + (FLOPS["X"] if "X" in names else 0.0))
    nbytes = es * nz + 8.0 * B * ncol
    if c["op"] == "loglike":
        nbytes += es * nz + 8.0 * B * (1 + ncol)
    else:
        nbytes += es * npairs * len(outs)
    if c["op"] == "jac":
        nbytes += es * npairs * ncol * len(outs)
    if c["op"] == "autograd":
        nbytes += es * npairs * len(grads) + 4.0 * B * ncol + (es * npairs if c["zgrad"] else 0.0)
    return {"bytes": nbytes, "flops": B * root + two * npairs * flops}
