"""What a program that uses this library has it do, as cases to be timed.

Each case is one call, or one short sequence of calls, through the public
functions of paper_1308_5351_gb300 (gnk.Boundary, gnk.Batch, gnk.slit_map,
gnk.slit_map_adjoint, autograd.fbie).  `listed()` gives the cases, `draw()`
more of the same ranges, `prepare()` the inputs, `run()` one pass, `work()`
what the pass cannot do without, and `exact()` the same outputs from dense
FP64 matrices or sums in plain torch, or from a closed form.

Closed form: for unbounded G with A = 1, f(z) = sum_k w_k / (z - z_k) with
every z_k inside a hole is analytic in G and vanishes at infinity, so
gamma = Re f(eta) + c_k on boundary k has mu = Im f(eta) and h = -c_k.
"""
import math

import numpy as np
import torch

from paper_1308_5351_gb300 import autograd as AG
from paper_1308_5351_gb300 import domains as Dm
from paper_1308_5351_gb300 import gnk as G

PREC = {"fp64": G.GNK_PREC_FP64, "df32": G.GNK_PREC_DF32, "fmm": G.GNK_PREC_FMM,
        "mixed": G.GNK_PREC_MIXED, "mixed_df": G.GNK_PREC_MIXED_DF, "mixed_fmm": G.GNK_PREC_MIXED_FMM}
DENSE_MAX = 17000  # nodes up to which exact() forms the dense matrices
FMM_ORDER = 32
STEPS = 20         # GMRES steps that work() counts for one solve


def listed():
    return [
        # One product of an own iteration on the smallest domain (connectivity 3): latency and launches.
        {"name": "apply_768_fp64", "kind": "apply", "op": "IminusN", "geom": "circles3", "m1": 3, "n": 256,
         "prec": "fp64"},
        # The whole FBIE computation of a new small domain with default options (FP64, tol 1e-12).
        {"name": "fbie_768_fp64", "kind": "fbie", "geom": "circles3", "m1": 3, "n": 256, "prec": "fp64",
         "tol": 1e-12, "restart": 20},
        # The operator M with direct FP64 sums on an ordinary domain, n not a power of two.
        {"name": "apply_M_16000_fp64", "kind": "apply", "op": "M", "geom": "ellipses", "m1": 16, "n": 1000,
         "prec": "fp64"},
        # Direct sums in mixed precision: FP32 inner products, double-float refinement.
        {"name": "fbie_16384_mixed_df", "kind": "fbie", "geom": "ellipses", "m1": 16, "n": 1024,
         "prec": "mixed_df", "tol": 1e-12, "restart": 20},
        # One Cauchy sum with complex weights by the FMM (a caller's own use of E w).
        {"name": "sum_65536_fmm", "kind": "sum", "geom": "ellipses", "m1": 64, "n": 1024, "prec": "fmm"},
        # The benchmark's step: a new 64-ellipse domain, build, tree, solve to 1e-10, h, free.
        {"name": "fbie_65536_fmm", "kind": "fbie", "geom": "ellipses", "m1": 64, "n": 1024, "prec": "fmm",
         "tol": 1e-10, "restart": 20},
        # High connectivity with close boundaries, the largest size: 1024 curves, N = 524,288.
        {"name": "fbie_524288_fmm", "kind": "fbie", "geom": "close", "m1": 1024, "n": 512, "prec": "fmm",
         "tol": 1e-10, "restart": 30},
        # The adjoint equation on a handle that is kept, for a new right-hand side; ragged n, odd m+1.
        {"name": "adjoint_16830_fmm", "kind": "adjoint", "geom": "ellipses", "m1": 33, "n": 510, "prec": "fmm",
         "tol": 1e-12, "restart": 20},
        # A conformal map of an unbounded five-circle domain onto a slit domain, at 20,000 points of G.
        {"name": "slit_5120", "kind": "slit", "geom": "ex4", "m1": 5, "n": 1024, "prec": "fmm", "tol": 1e-12,
         "points": 20000},
        # The same kind of map for a bounded domain by the adjoint route: m + 1 solves.
        {"name": "slit_adjoint_2560", "kind": "slit_adjoint", "geom": "ex2", "m1": 5, "n": 512, "prec": "fmm",
         "tol": 1e-12, "points": 3000},
        # Gradient of a loss of mu, h, h_k: forward and backward, 16 stars and 4 graded polygons.
        {"name": "gradient_40960_fmm", "kind": "gradient", "geom": "stars", "m1": 20, "n": 2048, "prec": "fmm",
         "tol": 1e-12, "restart": 30},
        # Many domains of uneven size with m+1 right-hand sides each, solved together (default precision).
        {"name": "batch_24", "kind": "batch", "count": 24, "m1": 16, "n": 512, "prec": "mixed_df", "tol": 1e-10,
         "restart": 20},
    ]


def _log_int(rng, lo, hi, step=1):
    hi -= hi % step
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step
    return max(lo, min(hi, v))


def draw(rng):
    kind = rng.choice(["apply", "apply", "sum", "fbie", "fbie", "fbie_fmm", "fbie_fmm", "adjoint", "slit",
                       "slit_adjoint", "gradient", "batch"])
    if kind == "apply":
        m1 = _log_int(rng, 2, 32)
        return {"kind": "apply", "op": rng.choice(["IminusN", "M", "adjoint"]), "geom": "ellipses", "m1": m1,
                "n": _log_int(rng, 64, 16384 // m1 if m1 > 8 else 2048, 2),
                "prec": rng.choice(["fp64", "fp64", "df32"])}
    if kind == "sum":
        m1 = _log_int(rng, 4, 128)
        return {"kind": "sum", "geom": "ellipses", "m1": m1, "n": _log_int(rng, 64, 1024, 2),
                "prec": rng.choice(["fp64", "fmm", "fmm"]) if m1 <= 16 else "fmm"}
    if kind == "fbie":
        return {"kind": "fbie", "geom": "ellipses", "m1": _log_int(rng, 2, 16), "n": _log_int(rng, 128, 1024, 2),
                "prec": rng.choice(["fp64", "mixed_df", "mixed_df", "mixed"]), "tol": 1e-12, "restart": 20}
    if kind == "fbie_fmm":
        if rng.random() < 0.3:
            g = rng.randint(8, 30)
            return {"kind": "fbie", "geom": "close", "m1": g * g, "n": _log_int(rng, 64, 512, 2), "prec": "fmm",
                    "tol": 1e-10, "restart": 30}
        return {"kind": "fbie", "geom": "ellipses", "m1": _log_int(rng, 8, 256), "n": _log_int(rng, 256, 1024, 2),
                "prec": "fmm", "tol": 1e-10, "restart": 20}
    if kind == "adjoint":
        return {"kind": "adjoint", "geom": "ellipses", "m1": _log_int(rng, 2, 64), "n": _log_int(rng, 128, 1024, 2),
                "prec": "fmm", "tol": 1e-12, "restart": 20}
    if kind == "slit":
        return {"kind": "slit", "geom": rng.choice(["ex2", "ex4"]), "m1": 5, "n": _log_int(rng, 256, 2048, 2),
                "prec": "fmm", "tol": 1e-12, "points": _log_int(rng, 500, 30000)}
    if kind == "slit_adjoint":
        return {"kind": "slit_adjoint", "geom": "ex2", "m1": 5, "n": _log_int(rng, 256, 2048, 2), "prec": "fmm",
                "tol": 1e-12, "points": _log_int(rng, 500, 10000)}
    if kind == "gradient":
        return {"kind": "gradient", "geom": "stars", "m1": 20, "n": _log_int(rng, 512, 2048, 2), "prec": "fmm",
                "tol": 1e-12, "restart": 30}
    return {"kind": "batch", "count": rng.randint(4, 24), "m1": rng.randint(4, 16), "n": rng.choice([256, 512]),
            "prec": "mixed_df", "tol": 1e-10, "restart": 20}


# --------------------------------------------------------------------- inputs
def _domain(case, seed):
    geom, m1, n = case["geom"], case["m1"], case["n"]
    r = np.random.default_rng([seed, 11])
    if geom == "circles3":  # the unit circle with two holes, moved and sized a little by the seed
        d = r.uniform(-0.02, 0.02, 4)
        return Dm.build_domain([Dm.Circle(0j, 1.0, ccw=True), Dm.Circle(0.45 + d[0], 0.2 + d[2]),
                                Dm.Circle(-0.45 + d[1], 0.2 + d[3])], n, bounded=True, alpha=0.05j)
    if geom == "ellipses":  # semi-axes U[0.1, 0.4], gaps >= 0.05, box scaled to the connectivity
        return Dm.build_domain(Dm.random_ellipses(r, m1, 4.0 * math.sqrt(m1 / 64.0) + (0.5 if m1 != 64 else 0.0)), n,
                               bounded=False)
    if geom == "close":
        g = math.isqrt(m1)
        return Dm.close_curves(seed=[seed, 12], n=n, grid=g, squares=max(1, m1 // 32))
    if geom == "stars":
        return Dm.stars_and_polygons(seed=[seed, 13], n=n)
    eps = 0.1 * r.uniform(0.8, 1.2)
    return Dm.ex2_circles(eps, n, alpha=_alpha(case, seed)) if geom == "ex2" else Dm.ex4_circles(eps, n)


def _alpha(case, seed):
    r = np.random.default_rng([seed, 14])
    d = complex(r.uniform(-0.02, 0.02), r.uniform(-0.02, 0.02))
    return d if case["geom"] == "ex2" else 2.5 + d


def _theta(case, seed):
    th = np.where(np.random.default_rng([seed, 15]).uniform(size=case["m1"]) < 0.6, math.pi / 2, 0.0)
    if case["geom"] == "ex2":
        th[0] = math.pi / 2
    return th


def _points(case, seed, d):
    """Points of G for the five-circle domains, at least 0.02 from every circle."""
    r = np.random.default_rng([seed, 16])
    R = 0.98 if case["geom"] == "ex2" else 3.0
    out, have = [], 0
    while have < case["points"]:
        z = r.uniform(-R, R, 4 * case["points"]) + 1j * r.uniform(-R, R, 4 * case["points"])
        if case["geom"] == "ex2":
            z = z[np.abs(z) < R]
        for cv in d.curves[1 if case["geom"] == "ex2" else 0:]:
            z = z[np.abs(z - cv.centre) > cv.radius + 0.02]
        out.append(z)
        have += z.size
    return np.concatenate(out)[: case["points"]]


def _poles(d, seed):
    """Poles in up to 8 holes, weights of the size of the hole, and c_k."""
    r = np.random.default_rng([seed, 17])
    k = r.choice(d.m1, size=min(8, d.m1), replace=False)
    size = np.array([d.curves[i].bbox_radius() for i in k])
    w = size * (r.normal(size=k.size) + 1j * r.normal(size=k.size))
    return np.array([d.holes[i] for i in k]), w, r.normal(size=d.m1)


def _has_closed_form(case):
    return case["geom"] in ("ellipses", "close", "stars") and case["m1"] * case["n"] > DENSE_MAX


def _gamma(case, seed, d):
    if not _has_closed_form(case):  # log|eta - alpha|, alpha in a hole or the domain's own point
        k = int(np.random.default_rng([seed, 18]).integers(d.m1))
        return Dm.gamma_log(d, d.holes[k])
    p, w, c = _poles(d, seed)
    return Dm.f_poles(p, w)(d.et).real + np.repeat(c, d.n)


def _dev(*arrays):
    return [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in arrays]


def _vector(seed, n, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 7 + 3)
    return torch.randn(n, dtype=dtype, device="cuda", generator=g)


def _boundary_precision(prec):
    if prec in ("fmm", "mixed_fmm"):
        return G.GNK_PREC_FMM
    return G.GNK_PREC_DF32 if prec in ("df32", "mixed_df") else G.GNK_PREC_FP64


def _batch(case, seed):
    ns = [n for n in (128, 256, 512) if n <= case["n"]]
    sizes = np.random.default_rng([case["count"], case["m1"], case["n"]])  # the seed moves the curves only
    r = np.random.default_rng([seed, 19])
    doms = []
    for _ in range(case["count"]):
        m1, n = int(sizes.integers(2, case["m1"] + 1)), int(sizes.choice(ns))
        doms.append(Dm.build_domain(Dm.random_ellipses(r, m1, 4.0 * math.sqrt(m1 / 64.0) + 0.5), n, bounded=False))
    gam = np.concatenate([Dm.gamma_log(d, a) for d in doms for a in d.holes])
    return doms, gam


def prepare(case, seed):
    kind, prec = case["kind"], PREC[case["prec"]]
    if kind == "batch":
        doms, gam = _batch(case, seed)
        b = G.Batch(doms, [d.m1 for d in doms], device="cuda")
        return {"case": case, "b": b, "gam": _dev(gam)[0]}
    d = _domain(case, seed)
    s = {"case": case, "prec": prec}
    if kind in ("apply", "sum", "adjoint"):  # the handle is kept: many products or right-hand sides
        adj = kind == "adjoint" or case.get("op") == "adjoint"
        s["b"] = G.Boundary.from_domain(d, adjoint=adj, device="cuda", precision=_boundary_precision(case["prec"]))
        if kind == "apply":
            s["x"] = _vector(seed, d.N)
        elif kind == "sum":
            s["w"] = _vector(seed, d.N, torch.complex128)
        else:
            s["gam"] = _dev(Dm.gamma_log(d, d.holes[0]))[0]
        return s
    if kind in ("slit", "slit_adjoint"):  # the call takes the domain's host arrays
        return dict(s, d=d, alpha=_alpha(case, seed), theta=_theta(case, seed), z=_points(case, seed, d))
    s["m1"], s["n"], s["bounded"] = d.m1, d.n, d.bounded
    s["et"], s["etp"], s["A"], s["gam"] = _dev(d.et, d.etp, d.A, _gamma(case, seed, d))
    if kind == "gradient":
        for k in ("et", "etp", "A", "gam"):
            s[k].requires_grad_(True)
        s["g"] = [_vector(seed + 1, d.N) / d.N, _vector(seed + 2, d.N) / d.N, _vector(seed + 3, d.m1)]
    return s


# ------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "apply":
        return getattr(s["b"], "apply_" + case["op"])(s["x"], s["prec"])
    if kind == "sum":
        return s["b"].cauchy_sum(s["w"], s["prec"])
    if kind == "adjoint":
        return s["b"].solve_adjoint_ie(s["gam"], tol=case["tol"], restart=case["restart"], precision=s["prec"])[0]
    if kind == "fbie":
        with G.Boundary(s["m1"], s["n"], s["et"], s["etp"], s["A"], bounded=s["bounded"],
                        precision=_boundary_precision(case["prec"]) | G.GNK_BUILD_DEFER) as b:
            mu, h, hk, _ = b.fbie(s["gam"], tol=case["tol"], restart=case["restart"], precision=s["prec"])
        return {"mu": mu, "h": h, "hk": hk}
    if kind == "slit":
        w, hk, wz, _ = G.slit_map(s["d"], s["alpha"], s["theta"], s["z"], precision=s["prec"], tol=case["tol"])
        return {"w": w, "hk": hk, "wz": wz}
    if kind == "slit_adjoint":
        w, psi, params, omega, wz, _ = G.slit_map_adjoint(s["d"], s["alpha"], s["theta"], s["z"],
                                                          precision=s["prec"], tol=case["tol"])
        return {"w": w, "psi": psi, "params": params, "omega": omega, "wz": wz}
    if kind == "batch":
        mu, h, hk, _, _ = s["b"].fbie(s["gam"], tol=case["tol"], restart=case["restart"], precision=PREC[case["prec"]])
        return {"mu": mu, "h": h, "hk": hk}
    leaves = [s["et"], s["etp"], s["A"], s["gam"]]
    out = AG.fbie(*leaves, s["m1"], s["n"], bounded=s["bounded"], precision=s["prec"], tol=case["tol"],
                  restart=case["restart"])
    grads = torch.autograd.grad(list(out), leaves, s["g"])
    return {"out": [o.detach() for o in out], "grads": list(grads)}


# ----------------------------------------------------------------------- work
def _product(N, prec):
    """(bytes, flops) of one Cauchy sum: nodes and weights in, sums out; direct
    sums 16 flops a pair, the FMM P coefficients a node up and down and its
    near field (9 boxes of 64 nodes)."""
    flops = 16.0 * N * N if prec != "fmm" else N * (2 * 8.0 * FMM_ORDER + 16.0 * 9 * 64)
    return 48.0 * N, flops


def work(case):
    if case["kind"] == "batch":
        m1, n, c = (case["m1"] + 2) / 2, 0.58 * case["n"], case["count"]
        by, fl = _product(m1 * n, "mixed_df")
        return {"bytes": c * m1 * by, "flops": c * m1 * STEPS * fl}
    N, prec = case["m1"] * case["n"], case["prec"]
    by, fl = _product(N, prec)
    if case["kind"] in ("apply", "sum"):
        return {"bytes": by, "flops": fl}
    fl *= STEPS
    if case["kind"] == "slit_adjoint":
        fl *= case["m1"]
    if case["kind"] in ("slit", "slit_adjoint"):
        by, fl = by + 32.0 * case["points"], fl + 24.0 * N * case["points"]
    if case["kind"] == "gradient":
        by, fl = 3 * by, 2 * fl
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------- exact values
def _sum_at(z, et, w, skip=False):
    """sum_j w_j / (z_i - et_j) in complex128, j = i left out with skip; w (N, R)."""
    out = torch.empty((z.numel(), w.shape[1]), dtype=torch.complex128, device=z.device)
    rows = max(1, (1 << 27) // et.numel())
    for a in range(0, z.numel(), rows):
        d = z[a:a + rows, None] - et[None, :]
        if skip:
            d[torch.arange(d.shape[0]), torch.arange(a, a + d.shape[0])] = math.inf
        out[a:a + rows] = d.reciprocal_() @ w
    return out


def _circulant(x, n):
    k = torch.arange(n, device=x.device, dtype=torch.float64)
    lam = torch.where(k < n / 2, 2 * k / n, 2 * (k - n) / n)
    lam[n // 2] = 0.0
    return torch.fft.ifft(1j * lam * torch.fft.fft(x.reshape(-1, n))).real.reshape(-1)


class _Dense:
    """The discrete operators from their definitions."""

    def __init__(self, m1, n, et, etp, A):
        self.m1, self.n, self.et, self.etp, self.A = m1, n, et, etp, A
        self.q = etp / A
        N = et.numel()
        eye = torch.eye(N, dtype=torch.bool, device=et.device)
        d = (et[:, None] - et[None, :]).masked_fill(eye, 1.0)
        self.E = (1.0 / d).masked_fill(eye, 0.0)
        self.one = self.E @ self.q

    def K_times(self, x):
        n, A = self.n, self.A
        return 2 * x - (2.0 / n) * (A * self.one).imag * x + (2.0 / n) * (A * (self.E @ (self.q * x))).imag

    def M_times(self, x):
        n, A = self.n, self.A
        return (-(2.0 / n) * (A * (self.E @ (self.q * x))).real + (2.0 / n) * (A * self.one).real * x
                + _circulant(x, n))

    def K(self):
        m = (2.0 / self.n) * (self.A[:, None] * self.E * self.q[None, :]).imag
        m.diagonal().copy_(2.0 - (2.0 / self.n) * (self.A * self.one).imag)
        return m

    def adjoint(self, etpp, Ap, c):
        n = self.n
        r = torch.where(self.etp.abs() > 0, etpp / self.etp - Ap / self.A, torch.zeros_like(self.etp)).imag
        e = 1 - c - (2.0 / n) * (self.E @ self.etp).imag + (2.0 / n) * r
        m = (2.0 / n) * (self.q[:, None] * self.E * self.A[None, :]).imag
        m.diagonal().copy_(e)
        m.view(self.m1, n, self.m1, n).diagonal(dim1=0, dim2=2).add_(1.0 / n)
        return m

    def fbie(self, gam):
        mu = torch.linalg.solve(self.K(), -self.M_times(gam))
        h = (self.M_times(mu) - self.K_times(gam)) / 2
        return mu, h, h.reshape(self.m1, self.n).mean(1)


def _exact_slit(case, seed, d):
    alpha, th, z = _alpha(case, seed), _theta(case, seed), _points(case, seed, d)
    rot = np.repeat(np.exp(1j * (math.pi / 2 - th)), d.n)
    lg = np.log(np.abs(d.et - alpha)) + 1j * np.unwrap(np.angle(d.et - alpha).reshape(d.m1, d.n), axis=1).reshape(-1)
    A = rot * (d.et - alpha) if d.bounded else rot
    et, etp, A, gam, z = _dev(d.et, d.etp, A, -(rot * lg).real, z)
    D = _Dense(d.m1, d.n, et, etp, A)
    mu, h, hk = D.fbie(gam)
    f = (gam + h + 1j * mu) / A
    s = _sum_at(z, et, torch.stack([f * etp, etp], 1))
    if d.bounded:
        fz = s[:, 0] / s[:, 1]
        w, wz = [torch.exp(-hk[0]) * (t - alpha) * torch.exp((t - alpha) * v) for t, v in ((et, f), (z, fz))]
    else:
        fz = -s[:, 0] / (d.n * 1j) / (1 - s[:, 1] / (d.n * 1j))
        w, wz = [(t - alpha) * torch.exp(v) for t, v in ((et, f), (z, fz))]
    if case["kind"] == "slit":
        return {"w": w, "hk": hk, "wz": wz}
    Ap = torch.as_tensor(rot * d.etp, device="cuda")
    rhs = torch.zeros(d.N, dtype=torch.float64, device="cuda")
    rhs[: d.n] = 1.0
    psi = torch.linalg.solve(D.adjoint(_dev(d.etpp)[0], Ap, d.c), rhs)
    return {"w": w, "psi": psi, "params": None, "omega": None, "wz": wz}


def _exact_gradient(case, seed, d):
    s = prepare(case, seed)
    p = [s[k] for k in ("et", "etp", "A", "gam")]
    with torch.no_grad():
        D = _Dense(d.m1, d.n, *p[:3])
        mu, h, hk = D.fbie(p[3])
        g_mu, g_h = s["g"][0], s["g"][1] + torch.repeat_interleave(s["g"][2], d.n) / d.n
        K = D.K()
    x = torch.zeros(d.N, dtype=torch.float64, device="cuda", requires_grad=True)
    Mt = torch.autograd.grad(D.M_times(x), x, g_h)[0]
    lam = torch.linalg.solve(K.T, g_mu + Mt / 2)
    del K, D
    D = _Dense(d.m1, d.n, *p[:3])
    loss = (-(lam * (D.K_times(mu) + D.M_times(p[3]))).sum() + (g_h * (D.M_times(mu) - D.K_times(p[3]))).sum() / 2)
    return {"out": [mu, h, hk], "grads": list(torch.autograd.grad(loss, p))}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        doms, gam = _batch(case, seed)
        out, at = [], 0
        for d in doms:
            et, etp, A = _dev(d.et, d.etp, d.A)
            D = _Dense(d.m1, d.n, et, etp, A)
            lu = torch.linalg.lu_factor(D.K())
            for _ in range(d.m1):
                g = _dev(gam[at:at + d.N])[0]
                at += d.N
                mu = torch.linalg.lu_solve(*lu, -D.M_times(g)[:, None])[:, 0]
                h = (D.M_times(mu) - D.K_times(g)) / 2
                out.append((mu, h, h.reshape(d.m1, d.n).mean(1)))
        return {k: torch.cat([o[i] for o in out]) for i, k in enumerate(("mu", "h", "hk"))}
    N = case["m1"] * case["n"]
    d = _domain(case, seed)
    if kind == "sum":
        if N > 131072:
            return None
        return _sum_at(*_dev(d.et, d.et), _vector(seed, N, torch.complex128)[:, None], skip=True)[:, 0]
    if kind == "fbie" and _has_closed_form(case):
        if case["geom"] == "close" or case["n"] < 512:  # the discretisation's own error is the larger one there
            return None
        p, w, c = _poles(d, seed)
        mu, h, hk = _dev(Dm.f_poles(p, w)(d.et).imag, np.repeat(-c, d.n), -c)
        return {"mu": mu, "h": h, "hk": hk}
    if N > (12000 if kind == "gradient" else DENSE_MAX):
        return None
    if kind in ("slit", "slit_adjoint"):
        return _exact_slit(case, seed, d)
    if kind == "gradient":
        return _exact_gradient(case, seed, d)
    D = _Dense(d.m1, d.n, *_dev(d.et, d.etp, d.A))
    if kind == "apply":
        x = _vector(seed, N)
        if case["op"] == "adjoint":
            return D.adjoint(*_dev(d.etpp, d.Ap), d.c) @ x
        return D.K_times(x) if case["op"] == "IminusN" else D.M_times(x)
    if kind == "adjoint":
        return torch.linalg.solve(D.adjoint(*_dev(d.etpp, d.Ap), d.c), _dev(Dm.gamma_log(d, d.holes[0]))[0])
    mu, h, hk = D.fbie(_dev(_gamma(case, seed, d))[0])
    return {"mu": mu, "h": h, "hk": hk}
