"""Performance cases: the work that a user of the library has it do, through the binding's calls.

Each case names one call on one problem; `run` makes the call and `exact` evaluates what it returns
in 64 bits from the paper's formulas with plain torch.  Where the call takes a vector, `prepare` draws
the vector and keeps the context of one atmosphere, as a Krylov solver or a synthesis run around the
call does; the solves and the setup draw the atmosphere itself.

  operator    y = (Id - Lambda Sigma) x, the step of every Krylov iteration
  transpose   y = (Id - Lambda Sigma)^T x, the step of the adjoint solve behind the field gradient
  precond     P^-1 y, beside the operator in every Krylov iteration
  solve       the whole preconditioned solve of one problem
  batch       the same for several independent ragged problems at once
  emergent    Stokes profiles along lines of sight off the angular grid, from a solution
  setup       a new atmosphere: tables, redistribution tiles, preconditioner, then its right-hand
              side and a first apply (what a field fit or an atmosphere grid pays at each point)

The full 70-height Mg II problem takes a minute to set up; its heights are independent in the
contraction, so the large cases keep its frequencies and directions and take a few heights.
"""
import functools
import math

import numpy as np
import torch

from paper_2505_20968_gb300 import inputs
from paper_2505_20968_gb300.binding import PRD, solve_batch

LOS_MU, LOS_CHI = (1.0, 0.1, 0.43), (0.0, 0.0, 0.7)   # disc centre, limb, one inclined view
TOL, MAX_ITER, RESTART = 1e-10, 600, 60               # the tolerance of the repository's solves


def listed():
    return [
        # the two-level slab in FP64: a few thousand points, nothing but launches and latency
        dict(name="slab_fp64", do="operator", atom="slab", prec="fp64", aa=False, nz=20, nnu=21, n_mu=1, n_chi=4),
        # a reduced Mg II problem, as the tests and gradient fits use: small, odd frequency count
        dict(name="mgii_small", do="operator", atom="mgii", prec="fp32", aa=False, nz=10, nnu=27, n_mu=2, n_chi=4),
        # the headline problem's frequencies and directions
        dict(name="mgii_full_grid", do="operator", atom="mgii", prec="fp32", aa=False, nz=8, nnu=200, n_mu=4, n_chi=8),
        # the split-BF16 precision at an odd frequency count of a ragged batch's range
        dict(name="mgii_bf16x3", do="operator", atom="mgii", prec="fp32_bf16x3", aa=False, nz=4, nnu=163, n_mu=4,
             n_chi=8),
        # H I Ly-alpha, the workload with most directions (96)
        dict(name="hi_full_grid", do="operator", atom="hi", prec="fp32", aa=False, nz=4, nnu=150, n_mu=6, n_chi=8),
        # the angle-averaged approximation: one class of all direction pairs
        dict(name="hi_angle_averaged", do="operator", atom="hi", prec="fp32", aa=True, nz=8, nnu=91, n_mu=4, n_chi=8),
        # backward direction, FP64 throughout
        dict(name="mgii_transpose", do="transpose", atom="mgii", prec="fp64", aa=False, nz=6, nnu=48, n_mu=2, n_chi=4),
        # the preconditioner on a tall atmosphere
        dict(name="mgii_precond", do="precond", atom="mgii", prec="fp32", aa=False, nz=20, nnu=100, n_mu=2, n_chi=4),
        # whole solves: one problem, and a ragged batch
        dict(name="mgii_solve", do="solve", atom="mgii", prec="fp32", aa=False, nz=6, nnu=26, n_mu=2, n_chi=4),
        dict(name="mgii_batch", do="batch", atom="mgii", prec="fp32", aa=False, nz=3, nnu=14, n_mu=2, n_chi=4, n=4),
        # what a synthesis run asks of a solution
        dict(name="mgii_emergent", do="emergent", atom="mgii", prec="fp32", aa=False, nz=4, nnu=41, n_mu=2, n_chi=4),
        # a new point of a fit
        dict(name="mgii_setup", do="setup", atom="mgii", prec="fp32", aa=False, nz=4, nnu=60, n_mu=2, n_chi=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["operator"] * 6 + ["transpose", "precond", "solve", "batch", "emergent", "setup"])
    if do == "operator":
        atom, prec = rng.choice([("mgii", "fp32"), ("mgii", "fp32"), ("hi", "fp32"), ("mgii", "fp32_bf16x3"),
                                 ("hi", "fp32_bf16x3"), ("slab", "fp64"), ("slab", "fp32"), ("mgii", "fp64")])
        aa = rng.random() < 0.2
        n_mu, n_chi = rng.choice([(1, 4), (2, 4), (2, 6), (3, 5), (4, 8)] + ([] if aa else [(6, 8)]))
        nnu = _log_int(rng, 12, 60 if prec == "fp64" else 100 if aa else 220)
        # work grows with heights x scattering angles x frequencies^2 (and FP64's rate is low): no more
        # than the largest listed case
        per_z = (2 * n_mu * n_chi) ** 1.6 * nnu ** 2 * (1 if atom == "slab" else 5) * (8 if prec == "fp64" else 1)
        top = 8 if aa else min(24, max(2, int(8 * 64 ** 1.6 * 200 ** 2 * 5 / per_z)))
        return dict(do=do, atom=atom, prec=prec, aa=aa, nz=_log_int(rng, 2, top), nnu=nnu, n_mu=n_mu, n_chi=n_chi)
    n_mu, n_chi = rng.choice([(2, 4), (2, 5), (3, 4)])
    c = dict(do=do, atom=rng.choice(["mgii", "hi"]), prec=rng.choice(["fp32", "fp64"]), aa=False, n_mu=n_mu,
             n_chi=n_chi)
    if do == "transpose":
        c.update(nz=_log_int(rng, 3, 12), nnu=_log_int(rng, 14, 64))
    elif do == "precond":
        c.update(nz=_log_int(rng, 5, 24), nnu=_log_int(rng, 20, 110))
    elif do == "solve":
        c.update(nz=_log_int(rng, 4, 8), nnu=_log_int(rng, 14, 32))
    elif do == "batch":
        c.update(prec="fp32", nz=_log_int(rng, 2, 4), nnu=_log_int(rng, 14, 18), n=rng.randint(2, 5))
    elif do == "emergent":
        c.update(nz=_log_int(rng, 3, 8), nnu=_log_int(rng, 14, 48))
    else:
        c.update(nz=_log_int(rng, 3, 6), nnu=_log_int(rng, 14, 60))
    return c


DRAWN_ATMOSPHERE = ("solve", "batch", "setup")   # the others draw the vector of a kept context


def _problem(case, seed, more=0):
    seed = seed if case["do"] in DRAWN_ATMOSPHERE else 2
    nz, nnu = case["nz"] + more % 5, case["nnu"] + more % 6
    mode = inputs.MODE_AA if case["aa"] else inputs.MODE_AD
    dirs = dict(n_mu_half=case["n_mu"], n_chi=case["n_chi"])
    wing = max(6, int(round(0.3 * nnu)))
    if case["atom"] == "slab":
        # the slab has no drawn part: its depth and thermalisation vary with the seed
        r = np.random.default_rng(seed)
        cfg = inputs.twolevel_slab(n_z=nz, n_x=nnu, tau_max=10 ** r.uniform(3, 5), eps=10 ** r.uniform(-4.5, -3),
                                   a=10 ** r.uniform(-3.3, -2.7), **dirs)
    elif case["atom"] == "mgii":
        core = (nnu - wing) // 2
        cfg = inputs.mgii(n_z=nz, n_core_each=core, n_wing=nnu - 2 * core, seed=seed, **dirs)
    else:
        cfg = inputs.hi_lya(n_z=nz, n_core=nnu - wing, n_wing=wing, seed=seed, **dirs)
    cfg["quad"]["mode"] = mode
    return dict(cfg, precision=case["prec"])


def _vector(case, cfg, seed, nO):
    """A Stokes field: the Planck function of each height times (0.3 .. 1), polarised to a few per cent."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.as_tensor(cfg["atm"]["W_T"], device="cuda", dtype=torch.float64)
    shape = (len(w), nO, len(cfg["quad"]["grid"]), 4)
    x = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)
    x[..., 0] = 0.3 + 0.7 * x[..., 0]
    x[..., 1:] = 0.1 * (x[..., 1:] - 0.5)
    x = x * w[:, None, None, None]
    return x if case["prec"] == "fp64" else x.float()


def _directions(case):
    return 2 * case["n_mu"] * case["n_chi"]


@functools.lru_cache(maxsize=1)
def _context(case):
    return PRD(_problem(dict(case), 0))


def prepare(case, seed):
    if case["do"] == "batch":
        return dict(do="batch", P=[PRD(_problem(case, seed + 17 * i, i)) for i in range(case["n"])])
    cfg = _problem(case, seed)
    s = dict(do=case["do"], x=_vector(case, cfg, seed, _directions(case)))
    if case["do"] == "setup":
        s["cfg"] = cfg
    elif case["do"] == "solve":
        s["P"] = PRD(cfg)
    else:
        s["P"] = _context(tuple((k, v) for k, v in case.items() if k != "name"))
    return s


def run(s):
    do = s["do"]
    if do == "operator":
        return s["P"].apply_operator(s["x"])
    if do == "transpose":
        return s["P"].apply_operator_T(s["x"])
    if do == "precond":
        return s["P"].apply_preconditioner(s["x"])
    if do == "solve":
        return s["P"].solve(tol=TOL, max_iter=MAX_ITER, restart=RESTART)[0]
    if do == "batch":
        return solve_batch(s["P"], tol=TOL, max_iter=MAX_ITER, restart=RESTART)[0]
    if do == "emergent":
        return s["P"].emergent_stokes(s["x"], LOS_MU, LOS_CHI)
    P = PRD(s["cfg"])
    out = [P.rhs(), P.apply_operator(s["x"])]
    P.close()
    return out


def work(case):
    mu, chi, _ = _angles(case["n_mu"], case["n_chi"], _full_rule(case))
    n = _unit(mu, chi)
    th = _theta(n[:, None], n[None])
    cls = np.unique(np.round(th, 9), return_inverse=True)[1].reshape(th.shape)
    if case["aa"]:
        cls = np.zeros_like(cls)
    ncls = float(cls.max() + 1)
    outs = float(sum(len(np.unique(np.nonzero(cls == c)[0])) for c in range(int(ncls))))
    ntrip, ntile = (3, 4) if case["atom"] == "slab" else (18, 20)
    nz, N, nO = case["nz"], case["nnu"], len(mu)
    esz = 8 if case["prec"] == "fp64" else 4
    # one apply: every redistribution tile once, the vector in and out, the formal solver's 10 coefficients
    apply_b = nz * ncls * ntile * N * 2 * N * esz + nz * nO * N * (8 + 10) * esz
    apply_f = 2.0 * nz * ntile * N * 2 * N * 4 * outs
    vec = nz * nO * N * 4 * esz
    do = case["do"]
    if do in ("operator", "transpose"):
        return {"bytes": apply_b, "flops": apply_f}
    if do == "precond":   # three sweeps of an N x N product and a scalar formal solution per height
        return {"bytes": 2 * vec + nz * N * N * 8 * 2 + nz * nO * N * 4 * esz, "flops": 3 * nz * (4.0 * N * N + 60 * nO * N)}
    if do in ("solve", "batch"):   # about 20 Krylov steps, each an apply
        k = 20 * case.get("n", 1)
        return {"bytes": k * (apply_b + 4 * vec), "flops": k * apply_f}
    # quadrature rows: about 50 panels of 8 nodes, some 200 FP64 operations each
    angles = len(LOS_MU) * nO if do == "emergent" else ncls
    rows = nz * angles * ntrip * N
    return {"bytes": vec + rows * 2 * N * esz, "flops": rows * 50 * 8 * 200.0}


# ------------------------------------------------------------------ 64-bit values
# The discrete problem of Eq. linear_system evaluated with plain torch in FP64: Sect. 2-4 and
# App. B, E.  The redistribution integrals are panel quadratures over breakpoints of their own.

def _full_rule(case):
    return case["atom"] == "slab" and case["n_mu"] == 1


def _angles(n_mu, n_chi, full):
    if full:
        mu, w = np.polynomial.legendre.leggauss(2 * n_mu)
    else:
        x, wx = np.polynomial.legendre.leggauss(n_mu)
        p = 0.5 * (x + 1.0)
        mu, w = np.concatenate([-p[::-1], p]), np.concatenate([0.5 * wx[::-1], 0.5 * wx])
    chi = 2.0 * np.pi * np.arange(n_chi) / n_chi
    return np.repeat(mu, n_chi), np.tile(chi, len(mu)), np.repeat(0.5 * w, n_chi) / n_chi


def _unit(mu, chi):
    s = np.sqrt(1.0 - mu * mu)
    return np.stack([s * np.cos(chi), s * np.sin(chi), mu], -1)


def _theta(a, b):
    th = 2.0 * np.arctan2(np.linalg.norm(a - b, axis=-1), np.linalg.norm(a + b, axis=-1))
    th = np.where(th < 1e-10, 0.0, th)
    return np.where(np.abs(th - np.pi) < 1e-10, np.pi, th)


class _Faddeeva:
    """w(z) for Im z >= 0: Weideman's rational series (SIAM J. Numer. Anal. 31, 1994) with 64
    terms, and the Laplace continued fraction beyond |z| = 8."""

    def __init__(self, n=64):
        m = 2 * n
        k = np.arange(-m + 1, m)
        self.L = math.sqrt(n / math.sqrt(2.0))
        t = self.L * np.tan(k * math.pi / m / 2)
        f = np.concatenate([[0.0], np.exp(-t * t) * (self.L ** 2 + t * t)])
        self.a = np.real(np.fft.fft(np.fft.fftshift(f)))[1:n + 1][::-1] / (2 * m)

    def __call__(self, x, y):
        z = torch.complex(x, y.expand_as(x).contiguous())
        d = self.L - 1j * z
        Z = (self.L + 1j * z) / d
        p = torch.zeros_like(Z)
        for a in self.a:
            p = p * Z + float(a)
        near = 2 * p / d ** 2 + 1.0 / (math.sqrt(math.pi) * d)
        zf = torch.where(z.abs() > 8, z, torch.full_like(z, 8.0 + 8.0j))
        c = torch.zeros_like(zf)
        for k in range(24, 0, -1):
            c = (0.5 * k) / (zf - c)
        return torch.where(z.abs() > 8, (1j / math.sqrt(math.pi)) / (zf - c), near)


_W = _Faddeeva()
_SIG = np.array([[[1, 0], [0, 1]], [[1, 0], [0, -1]], [[0, 1], [1, 0]], [[0, -1j], [1j, 0]]])
_GL = np.polynomial.legendre.leggauss(10)


def _t(v):
    return torch.as_tensor(np.asarray(v), device="cuda")


def _spline_map(u):
    """Second derivatives of the natural cubic spline on u as a linear map of the node values."""
    n = len(u)
    h = np.diff(u)
    T = np.eye(n)
    D = np.zeros((n, n))
    for i in range(1, n - 1):
        T[i, i - 1:i + 2] = h[i - 1], 2 * (h[i - 1] + h[i]), h[i]
        D[i, i - 1:i + 2] = 6 / h[i - 1], -6 / h[i - 1] - 6 / h[i], 6 / h[i]
    return np.linalg.solve(T, D)


def _spline_basis(u, Q, x):
    """[len(x), N]: the spline through unit values, continued by its end values."""
    n = len(u)
    j = np.clip(np.searchsorted(u, x, side="right") - 1, 0, n - 2)
    h = u[j + 1] - u[j]
    t = np.clip((x - u[j]) / h, 0.0, 1.0)
    s = 1 - t
    B = ((h * h / 6) * (s ** 3 - s))[:, None] * Q[j] + ((h * h / 6) * (t ** 3 - t))[:, None] * Q[j + 1]
    r = np.arange(len(x))
    B[r, j] += s
    B[r, j + 1] += t
    return B


def _rows(u, Q, a, theta, s_in, s_out, un, kind):
    """Integrals over u' of the kernel against the cardinal splines, one row per entry of the
    (equal-length) arrays: kind 2, F(theta, u' + s_in, un + s_out) (Eq. G); kind 3, the incident
    bracket W(u' + s_in) + W(u' + s_out)^* of Eq. RIIIQKKp over the grid's span."""
    N, ut = len(u), _t(u)
    out = []
    gx, gw = _t(_GL[0]), _t(_GL[1])
    per = max(1, int(3e6 / ((N + 70) * 10)))
    for c0 in range(0, len(un), per):
        th, si, so, x0 = (_t(v[c0:c0 + per])[:, None] for v in (theta, s_in, s_out, un))
        R = len(x0)
        x = x0 + so
        P, M = torch.zeros(2, 2, 2, R, N, dtype=torch.float64, device="cuda")   # moments: end, Re | Im, interval
        if kind == 2:
            s2, c2 = torch.sin(th / 2), torch.cos(th / 2)
            back, fwd = th == math.pi, th == 0.0
            c2 = torch.where(back, torch.zeros_like(c2), c2)
            g = torch.where(fwd, torch.ones_like(s2), 2 * s2)
            mid, far = x - si, -x - si
            lo, hi = mid - 6.5 * g, mid + 6.5 * g
            hv = torch.maximum(c2, torch.full_like(c2, a))
            near = torch.cat([mid + 0.5 * g * torch.arange(-13, 14, device="cuda"), far], 1)
            for k in range(18):
                near = torch.cat([near, far - hv * 2.0 ** k, far + hv * 2.0 ** k], 1)
        else:
            lo, hi = ut[0].expand(R, 1), ut[-1].expand(R, 1)
            off = [sg * a * 2.0 ** k for k in range(18) for sg in (-1, 1)] + [0.0] + [0.5 * k for k in range(-12, 13)]
            near = torch.cat([-s + torch.tensor(off, device="cuda", dtype=torch.float64) for s in (si, so)], 1)
        b = torch.cat([lo, hi, ut.expand(R, N), near], 1)
        b = torch.sort(torch.minimum(torch.maximum(b, lo), hi), 1)[0]
        half, cen = 0.5 * (b[:, 1:] - b[:, :-1]), 0.5 * (b[:, 1:] + b[:, :-1])
        j = torch.searchsorted(ut, cen.contiguous(), right=True)        # 0 left of the grid .. N right of it
        up = cen[..., None] + half[..., None] * gx
        wq = half[..., None] * gw
        if kind == 2:
            x3, si3, th3 = x[..., None], si[..., None], th[..., None]
            xp = up + si3
            c3 = torch.where(back | fwd, torch.ones_like(c2), c2)[..., None]
            g3 = g[..., None]
            F = torch.exp(-((x3 - xp) / g3) ** 2) * _W((x3 + xp) / (2 * c3), a / c3) / (g3 * c3)
            v, d = 0.5 * (x3 + xp), x3 - xp
            Fb = torch.exp(-0.25 * d * d) / (2 * math.sqrt(math.pi)) * torch.complex(a / (v * v + a * a), v / (v * v + a * a))
            F = torch.where(back[..., None], Fb, F)
            # forward scattering: sqrt(pi) W(a, x) delta(u' - (x - s_in)); one point in its interval
            F = torch.where((th3 == 0.0), torch.zeros_like(F), F)
        else:
            aa = torch.full_like(up, a)
            F = _W(up + si[..., None], aa) + _W(up + so[..., None], aa).conj()
        F = F * wq

        def add(F, up, j):
            i0 = (j - 1).clamp(0, N - 2)
            h = (ut[i0 + 1] - ut[i0])[..., None]
            t = ((up - ut[i0][..., None]) / h).clamp(0.0, 1.0)
            s = 1 - t
            k6 = h * h / 6
            for m, wts in ((P, (s, t)), (M, (k6 * (s ** 3 - s), k6 * (t ** 3 - t)))):
                for q in (0, 1):
                    v = (F * wts[q]).sum(-1)
                    m[q, 0].scatter_add_(1, i0, v.real)
                    m[q, 1].scatter_add_(1, i0, v.imag)
        add(F, up, j)
        if kind == 2 and bool(fwd.any()):
            p = x - si
            D = torch.where(fwd, math.sqrt(math.pi) * _W(x, torch.full_like(x, a)), torch.zeros_like(x, dtype=torch.complex128))
            add(D[..., None], p[..., None], torch.searchsorted(ut, p.contiguous(), right=True))
        Py, Pm = (m[0] + torch.cat([m.new_zeros(2, R, 1), m[1][..., :N - 1]], -1) for m in (P, M))
        out.append(torch.complex(*(Py + Pm @ _t(Q))))
    return torch.cat(out)


class _Exact:
    MUB, C, KB, AMU = 1.39962449361e10, 2.99792458e8, 1.380649e-23, 1.66053906660e-27

    def __init__(self, case, cfg):
        self.cfg, self.aa = cfg, case["aa"]
        atm, at, q = cfg["atm"], cfg["atom"], cfg["quad"]
        self.mu, self.chi, self.w = _angles(case["n_mu"], case["n_chi"], _full_rule(case))
        self.nz, self.N, self.nO = len(atm["z_km"]), len(q["grid"]), len(self.mu)
        E = np.array(at["E_u_cm"]) * 2.99792458e10
        self.S2 = 1 if at["twoS"] == 0 else 2
        self.nu0 = E[0] if self.S2 == 1 else (2 * E[0] + 4 * E[1]) / 6
        vD = np.sqrt(2 * self.KB * atm["T_K"] / (at["mass_amu"] * self.AMU) + (atm["xi_kms"] * 1e3) ** 2)
        self.vD, self.dnu = vD / 1e3, self.nu0 * vD / self.C
        g = q["grid"]
        nu = self.C / (g * 1e-10) if q["grid_kind"] == inputs.GRID_LAMBDA else self.nu0 - g * self.dnu[0]
        self.u = (self.nu0 - nu) / self.dnu[:, None]
        self.Q = [_spline_map(u) for u in self.u]
        self.grid = self._side(self.mu, self.chi)

    def _states(self, iz):
        at, B = self.cfg["atom"], self.cfg["atm"]["B_G"][iz]
        E, nl = np.array(at["E_u_cm"]) * 2.99792458e10, self.MUB * 1e-4 * B
        ms = [0.0] if self.S2 == 1 else [-0.5, 0.5]
        basis = [(m, s) for m in (-1, 0, 1) for s in ms]
        zeta = 0.0 if self.S2 == 1 else (E[1] - E[0]) / 1.5
        H = np.diag([E[0] + zeta * (1 + m * s) - self.nu0 + nl * (m + at["g_s"] * s) for m, s in basis])
        for i, (m, s) in enumerate(basis):
            for k, (m2, s2) in enumerate(basis):
                if self.S2 == 2 and abs(m - m2) == 1 and m + s == m2 + s2:
                    H[i, k] = 0.5 * zeta * math.sqrt(2.0)
        Eu, V = np.linalg.eigh(H)
        D = np.zeros((3, len(basis), len(ms)))
        for b, (m, s) in enumerate(basis):
            D[m + 1, :, ms.index(s)] = V[b]
        return Eu, np.array([nl * at["g_s"] * s for s in ms]), D

    def _amps(self, iz, D, mu, chi):
        tb, cb = self.cfg["atm"]["thetaB"][iz], self.cfg["atm"]["chiB"][iz]
        R = np.array([[np.cos(tb) * np.cos(cb), np.cos(tb) * np.sin(cb), -np.sin(tb)], [-np.sin(cb), np.cos(cb), 0],
                      [np.sin(tb) * np.cos(cb), np.sin(tb) * np.sin(cb), np.cos(tb)]])
        s = np.sqrt(1 - mu * mu)
        e = np.stack([np.stack([-np.sin(chi), np.cos(chi), 0 * mu], -1),
                      np.stack([mu * np.cos(chi), mu * np.sin(chi), -s], -1)], 1)             # [dir, 2, 3]
        r = 1 / math.sqrt(2.0)
        eq = np.array([[r, 1j * r, 0], [0, 0, 1], [-r, 1j * r, 0]])
        return np.einsum("qx,xy,day,qul->daul", eq, R, e, D)

    def _side(self, mu, chi):
        """Everything of the output directions (mu, chi): per height the comoving emissivity matrix
        from the grid's comoving field, the frame changes, K, and the Kirchhoff factor."""
        atm, N = self.cfg["atm"], self.N
        no, ng = _unit(mu, chi), _unit(self.mu, self.chi)
        th = _theta(no[:, None], ng[None])
        key = np.round(th, 9)
        ths, cls = np.unique(key, return_inverse=True)
        cls = cls.reshape(th.shape)
        ths = np.array([th[cls == c][0] for c in range(len(ths))])
        if self.aa:
            x, w = np.polynomial.legendre.leggauss(48)
            x = np.concatenate([(x + 1) / 4 * np.pi, (x + 3) / 4 * np.pi])
            aw = np.concatenate([w, w]) * np.pi / 8 * np.sin(x)
            ths, cls = x, np.zeros_like(cls)
        S = dict(mu=mu, S=[], K=[], back=[], inn=[], f=[])
        for iz in range(self.nz):
            u, Q, a = self.u[iz], self.Q[iz], float(atm["a"][iz])
            Eu, El, D = self._states(iz)
            nu_, nl = len(Eu), len(El)
            sh = (Eu[:, None] - El) / self.dnu[iz]
            A, Ag = self._amps(iz, D, mu, chi), self._amps(iz, D, self.mu, self.chi)
            # tiles G[class, k, l, l'] of the couplings that exist
            idx = [(c, k, l, m) for c in range(len(ths)) for k in range(nu_) for l in range(nl) for m in range(nl)
                   if np.any(D[:, k, l]) and np.any(D[:, k, m])]
            c_, k_, l_, m_ = (np.repeat(v, N) for v in np.array(idx).T)
            rows = _rows(u, Q, a, ths[c_], sh[k_, l_], sh[k_, m_], np.tile(u, len(idx)), 2)
            G = torch.zeros(len(ths), nu_, nl, nl, N, N, dtype=torch.complex128, device="cuda")
            ii = np.array(idx).T
            G[ii[0], ii[1], ii[2], ii[3]] = rows.view(len(idx), N, N)
            if self.aa:
                G = torch.einsum("c,cklmnp->klmnp", _t(aw).to(G.dtype), G)[None]
            Gt = 4 * np.pi * self.dnu[iz] * a
            de = 2j * np.pi * (Eu[:, None] - Eu)
            eps, rE = atm["eps"][iz], atm["r_el"][iz]
            al = (1 - eps) * (1 - rE) / (1 + de / Gt)
            be = (1 - eps) / (1 + de / (Gt * (1 - rE)))
            # Tr(sig_i M(u) sig_j M(v)^+) split into outgoing and incoming factors
            O = np.einsum("dbvm,iba,daum->duvmi", A, _SIG, A.conj())
            I = np.einsum("ebvl,jab,eaul->euvlj", Ag.conj(), _SIG, Ag)
            wk = self.w * atm["k_line"][iz]
            Y = _t(np.einsum("duvmi,euvlj,uv,e->devlmij", O, I, al, wk) * 3 / (4 * np.pi * self.S2))
            M = torch.zeros(len(mu), N, 4, self.nO, N, 4, dtype=torch.float64, device="cuda")
            for d in range(len(mu)):
                for e in range(self.nO):
                    M[d, :, :, e] = torch.einsum("vlmij,vlmnp->nipj", Y[d, e], G[cls[d, e]]).real
            # R_III: separable
            ku, kv, kl = (v.ravel() for v in np.meshgrid(np.arange(nu_), np.arange(nu_), np.arange(nl), indexing="ij"))
            rin = _rows(u, Q, a, 0.0 * ku, sh[kv, kl], sh[ku, kl], 0.0 * ku, 3).view(nu_, nu_, nl, N)
            w = _W(_t(u[:, None, None] + sh), _t(np.full((1,), a)))                          # [n, k, l]
            prof = w[:, None].expand(-1, nu_, -1, -1) + w[:, :, None].expand(-1, -1, nu_, -1).conj()
            cf = 3 / (16 * np.pi * self.S2) * (be - al)
            Od = torch.einsum("duvmi,nuvm->uvdni", _t(O), prof)
            Id = torch.einsum("euvlj,uvlp->uvepj", _t(I * wk[:, None, None, None, None]), rin)
            M += torch.einsum("uv,uvdni,uvepj->dniepj", _t(cf), Od, Id).real
            # K, thermal emissivity
            v = atm["v_kms"][iz] / self.vD[iz]
            ub, ug = no @ v, ng @ v
            wk_ = _W(_t(u[None, :, None, None] + ub[:, None, None, None] + sh), _t(np.full((1,), a)))
            kap = torch.einsum("daul,dbul,dnul->dnab", _t(A.conj()), _t(A), wk_.conj())
            kap = kap * atm["k_line"][iz] / (2 * math.sqrt(math.pi) * self.S2)
            sg = _t(_SIG)
            K = 0.5 * (torch.einsum("iab,dnbc,jca->dnij", sg, kap, sg) + torch.einsum("iab,jbc,dnac->dnij", sg, sg, kap.conj())).real
            back = torch.stack([_t(_spline_basis(u, Q, u + b)) for b in ub])
            inn = torch.stack([_t(_spline_basis(u, Q, u - b)) for b in ug])
            W = float(atm["W_T"][iz])
            flat = torch.zeros(self.nO, N, 4, dtype=torch.float64, device="cuda")
            flat[..., 0] = W
            num = torch.einsum("dnp,dp->dn", back, torch.einsum("dnepj,epj->dn", M[:, :, 0], flat))
            S["S"].append(M)
            S["K"].append(K)
            S["back"].append(back)
            S["inn"].append(inn)
            S["f"].append((1 - eps) * W * K[..., 0, 0] / num)
        S["K"] = torch.stack(S["K"])
        return S

    def sigma(self, x, S):
        out = []
        for iz in range(self.nz):
            It = torch.einsum("enp,epj->enj", S["inn"][iz], x[iz])
            eb = torch.einsum("dniepj,epj->dni", S["S"][iz], It)
            e = torch.einsum("dnp,dpi->dni", S["back"][iz], eb)
            out.append(torch.cat([e[..., :1] * S["f"][iz][..., None], e[..., 1:]], -1))
        return torch.stack(out)

    def thermal(self, S):
        atm = self.cfg["atm"]
        return _t(atm["eps"] * atm["W_T"])[:, None, None, None] * S["K"][..., :, 0]

    def formal(self, eps, S, boundary):
        """DELO-linear along every direction of S (Sect. 3), both senses at once by flipping heights."""
        z = _t(np.asarray(self.cfg["atm"]["z_km"], float))
        up = S["mu"] > 0
        out = [None] * len(up)
        eye = torch.eye(4, dtype=torch.float64, device="cuda")
        for sense in (True, False):
            d = np.nonzero(up == sense)[0]
            if not len(d):
                continue
            flip = (lambda v: v) if sense else (lambda v: torch.flip(v, (0,)))
            K, e, zz = flip(S["K"][:, d]), flip(eps[:, d]), flip(z)
            eta = K[..., 0, 0]
            Kp, Sv = K / eta[..., None, None] - eye, e / eta[..., None]
            amu = _t(np.abs(S["mu"][d]))[:, None]
            I = torch.zeros_like(Sv[0])
            if boundary and sense:
                I = torch.cat([torch.full_like(I[..., :1], float(self.cfg["atm"]["W_T"][0])), I[..., 1:]], -1)
            rows = [I]
            for p in range(1, self.nz):
                t = 0.5 * (eta[p - 1] + eta[p]) * (zz[p] - zz[p - 1]).abs() / amu
                w0 = -torch.expm1(-t)
                ser = t / 2 - t ** 2 / 6 + t ** 3 / 24 - t ** 4 / 120 + t ** 5 / 720 - t ** 6 / 5040
                b = torch.where(t < 0.02, ser, 1 - w0 / t)
                sea = t / 2 - t ** 2 / 3 + t ** 3 / 8 - t ** 4 / 30 + t ** 5 / 144 - t ** 6 / 840
                a = torch.where(t < 0.02, sea, w0 - b)
                rhs = torch.exp(-t)[..., None] * I - a[..., None] * (Kp[p - 1] @ I[..., None])[..., 0] + a[..., None] * Sv[p - 1] + b[..., None] * Sv[p]
                I = torch.linalg.solve(eye + b[..., None, None] * Kp[p], rhs[..., None])[..., 0]
                rows.append(I)
            r = flip(torch.stack(rows))
            for n, i in enumerate(d):
                out[i] = r[:, n]
        return torch.stack(out, 1)

    def operator(self, x):
        return x - self.formal(self.sigma(x, self.grid), self.grid, False)


def exact(case, seed):
    # solves stop anywhere below their tolerance and the preconditioner is an approximate inverse
    # of the framework's own: no value in 64 bits to hold them to
    if case["do"] in ("solve", "batch", "precond"):
        return None
    # the quadrature's kernel evaluations and the dense height matrices: beyond these it takes minutes
    nO, N = _directions(case), case["nnu"]
    per_z = N * (96 if case["aa"] else nO ** 1.6 / 3) * (3 if case["atom"] == "slab" else 18)
    if case["nz"] * per_z * (N + 70) * 10 > 1.2e9 or (nO * N * 4) ** 2 * 8 * case["nz"] > 20e9:
        return None
    cfg = _problem(case, seed)
    x = _vector(case, cfg, seed, nO).double()
    X = _Exact(case, cfg)
    if case["do"] == "operator":
        return X.operator(x)
    if case["do"] == "transpose":
        v = torch.zeros_like(x, requires_grad=True)
        return torch.autograd.grad(X.operator(v), v, x)[0]
    if case["do"] == "setup":
        return [X.formal(X.thermal(X.grid), X.grid, True), X.operator(x)]
    S = X._side(np.array(LOS_MU), np.array(LOS_CHI))
    return X.formal(X.sigma(x, S) + X.thermal(S), S, True)[-1]
