"""Performance cases of the column-by-column MALI library, run through the Python binding's public calls.

Each case is one call (or the few calls) a user's program makes on columns it holds on the GPU:

* ``iterate`` -- ``Context.iterate``: MALI iterations with Ng acceleration from the LTE start, mixed precision or
  all FP64, linear or Bezier formal solver, lines in complete or (``prd``) partial redistribution; populations out.
  ``tol`` 0 runs exactly ``maxiter`` iterations (a bounded slice of a long run); ``tol`` 1e-3 runs to convergence.
* ``solve`` -- ``Context.load_columns`` then ``Context.solve``: the whole two-stage solve of new columns.
* ``load`` -- ``Context.load_columns`` from device memory: validation, electron densities, LTE populations, rates.
* ``spectrum`` / ``stokes`` -- emergent intensities, and the Zeeman Stokes vector of H alpha, of given populations.
* ``train`` -- ``Context.surrogate_train``: one epoch of the learned start's network on converged columns.

Sizes follow the repository's own workloads: 82 heights (128 in the full run), the hydrogen-like 5-level + continuum
atom with 608 wavelengths and 5 angles, the reduced 3-level atom with 2 angles, Lyman alpha and beta in partial
redistribution at 64 or 200 points, 400 Stokes wavelengths, training batches of 512.

Results of the single-precision formal solution are kept as float32, as a program that stores cubes of populations or
spectra does; the all-FP64 path's stay float64.
"""
import math

import numpy as np
import torch

import paper_1411_1079_gb300 as rh
import rh_synth

LINE_HALPHA = 4        # index of the n = 2-3 line in the hydrogen-like atom's list (lines in order of n, n')


def listed():
    return [
        # the smallest call: a handful of shallow columns, a reduced atom, odd sizes -- launch and latency
        dict(name="iterate 37x13 small atom", kind="iterate", ncol=37, ndep=13, atom="small", precision=1, formal=0,
             maxiter=25, tol=0.0),
        # one column solved interactively: latency of a single column's iteration chain
        dict(name="iterate 1 column to 1e-3", kind="iterate", ncol=1, ndep=82, atom="h6", precision=1, formal=0,
             maxiter=500, tol=1e-3),
        # the ordinary workload: a slab of a cube, about the iterations a column takes from a good start
        dict(name="iterate 1000 columns", kind="iterate", ncol=1000, ndep=82, atom="h6", precision=1, formal=0,
             maxiter=12, tol=0.0),
        # the largest mixed-precision call: new columns loaded and solved from LTE with the re-run ladder
        dict(name="solve 2048 columns", kind="solve", ncol=2048, ndep=82, atom="h6", precision=1),
        # the all-FP64 path, used as the accuracy reference
        dict(name="iterate FP64 150 columns", kind="iterate", ncol=150, ndep=82, atom="h6", precision=0, formal=0,
             maxiter=3, tol=0.0),
        # the higher-order formal solver, used for steep atmospheres and as the rescue of PRD solves
        dict(name="iterate Bezier 300 columns", kind="iterate", ncol=300, ndep=82, atom="h6", precision=1, formal=1,
             maxiter=8, tol=0.0),
        # partial redistribution of the resonance lines in the static frame
        dict(name="iterate PRD 300 columns", kind="prd", ncol=300, ndep=82, npoint=64, hybrid=0, precision=1,
             maxiter=8),
        # the full run's configuration: 128 heights, 200 points per resonance line, frame of the moving gas
        dict(name="iterate hybrid PRD 128x200", kind="prd", ncol=160, ndep=128, npoint=200, hybrid=1, precision=1,
             maxiter=4),
        # spectra of a cube slab in the call's default precision, around Lyman alpha and H alpha and continua
        dict(name="spectrum 4096x201", kind="spectrum", ncol=4096, ndep=82, nlam=201, mu=1.0, precision=0),
        # the full run's last step: polarised H alpha spectra
        dict(name="Stokes 2048x400", kind="stokes", ncol=2048, ndep=128, nlam=400, precision=1),
        # the learned start: an epoch over a slab of converged columns
        dict(name="train 4096 columns", kind="train", ncol=4096, ndep=82, batch=512),
        # a whole cube handed over
        dict(name="load 65536 columns", kind="load", ncol=65536, ndep=82),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["iterate", "iterate", "iterate", "iterate64", "bezier", "prd", "prd", "solve", "spectrum",
                       "stokes", "train", "load"])
    ndep = rng.choice([13, 32, 41, 64, 82, 82, 100, 128])
    if what == "iterate":
        return dict(kind="iterate", ncol=_log(rng, 1, 1000), ndep=ndep, atom=rng.choice(["h6", "h6", "small"]),
                    precision=1, formal=0, maxiter=rng.randint(4, 14), tol=0.0)
    if what == "iterate64":
        return dict(kind="iterate", ncol=_log(rng, 1, 150), ndep=rng.choice([13, 32, 64, 82]),
                    atom=rng.choice(["h6", "small"]), precision=0, formal=0, maxiter=rng.randint(2, 3), tol=0.0)
    if what == "bezier":
        return dict(kind="iterate", ncol=_log(rng, 1, 300), ndep=ndep, atom="h6", precision=1, formal=1,
                    maxiter=rng.randint(4, 8), tol=0.0)
    if what == "prd":
        return dict(kind="prd", ncol=_log(rng, 4, 300), ndep=rng.choice([32, 64, 82]),
                    npoint=rng.choice([32, 50, 64, 97]), hybrid=rng.randint(0, 1), precision=1,
                    maxiter=rng.randint(3, 8))
    if what == "solve":
        return dict(kind="solve", ncol=_log(rng, 16, 1500), ndep=rng.choice([64, 82]), atom="h6", precision=1)
    if what == "spectrum":
        return dict(kind="spectrum", ncol=_log(rng, 1, 4096), ndep=ndep, nlam=_log(rng, 5, 200),
                    mu=rng.choice([1.0, 0.35]), precision=rng.randint(0, 1))
    if what == "stokes":
        p = rng.randint(0, 1)
        return dict(kind="stokes", ncol=_log(rng, 1, 2048 if p else 150), ndep=ndep, nlam=_log(rng, 9, 400),
                    precision=p)
    if what == "train":
        return dict(kind="train", ncol=_log(rng, 300, 4096), ndep=rng.choice([24, 82]),
                    batch=rng.choice([100, 256, 512]))
    return dict(kind="load", ncol=_log(rng, 1, 65536), ndep=rng.choice([13, 82]))


# ---- inputs ---------------------------------------------------------------------------------------------------------
def _atom(case):
    if case.get("atom") == "small":
        return rh_synth.small_atom()
    if case["kind"] == "prd":
        return rh_synth.hydrogen_like_atom(prd_lines=((1, 2), (1, 3)), prd_nlambda=case["npoint"])
    return rh_synth.hydrogen_like_atom()


def _columns(case, seed):
    return rh_synth.chromosphere_cube(nx=case["ncol"], ny=1, ndep=case["ndep"], seed=seed)


def _departures(case, nlev, seed):
    """Smooth departure coefficients growing towards the top, as a solved cube has: [ncol][nlev][ndep]."""
    rng = np.random.default_rng(seed + 77)
    top = np.linspace(1.0, 0.0, case["ndep"]) ** 2
    amp = rng.uniform(-1.0, 1.0, (case["ncol"], nlev, 1))
    amp[:, 0] = 0.0
    return np.exp(amp * top)


def _wavelengths(case):
    n = case["nlam"]
    if case["kind"] == "stokes":
        return 656.46e-9 + np.linspace(-0.15e-9, 0.15e-9, n)
    na = max(1, (2 * n) // 5)
    nb = max(1, (2 * n) // 5)
    nc = max(1, n - na - nb)
    return np.concatenate([np.linspace(121.4e-9, 121.8e-9, na), np.linspace(656.0e-9, 656.9e-9, nb),
                           np.linspace(80e-9, 4100e-9, nc)])[:n]


def _fields(case, seed):
    rng = np.random.default_rng(seed + 5)
    shape = (case["ncol"], case["ndep"])
    one = (case["ncol"], 1)
    B = np.broadcast_to(rng.uniform(0.0, 0.2, one), shape)
    th = np.broadcast_to(np.arccos(rng.uniform(-1.0, 1.0, one)), shape)
    az = np.broadcast_to(rng.uniform(0.0, 2.0 * np.pi, one), shape)
    return [np.ascontiguousarray(x) for x in (B, th, az)]


def _gpu(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def prepare(case, seed):
    atom, cols = _atom(case), _columns(case, seed)
    ctx = rh.Context(0)
    ctx.setup_atom(atom)
    dev = {k: _gpu(v) for k, v in cols.items()}
    torch.cuda.synchronize()
    s = dict(case=case, ctx=ctx, cols=dev)
    shape = (case["ncol"], atom["nlev"], case["ndep"])
    if case["kind"] in ("iterate", "prd", "solve", "load"):
        s["pops"] = torch.empty(shape, dtype=torch.float64, device="cuda")
        if case["kind"] in ("iterate", "prd"):
            ctx.load_columns(dev, on_device=True)
    else:
        ctx.load_columns(dev, on_device=True)
        n = _departures(case, atom["nlev"], seed) * ctx.lte()[0]
        if case["kind"] == "train":
            # the columns count as converged and carry these populations
            ctx.iterate(maxiter=1, tol=1e30, ng_order=0)
            ctx.set_populations(n)
            ctx.surrogate_init(hidden=512, nhidden=3, seed=seed)
            s["weights"] = ctx.surrogate_state()
        else:
            ctx.set_populations(n)
            s["lam"] = _wavelengths(case)
            out = (case["ncol"], case["nlam"]) + ((4,) if case["kind"] == "stokes" else ())
            s["out"] = torch.empty(out, dtype=torch.float64, device="cuda")
            if case["kind"] == "stokes":
                s["field"] = [_gpu(x) for x in _fields(case, seed)]
                torch.cuda.synchronize()
    return s


def _kept(x, case):
    return x.float() if case["precision"] == 1 else x


def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "iterate":
        ctx.iterate(maxiter=case["maxiter"], tol=case["tol"], precision=case["precision"], formal=case["formal"])
        n, iters, status, _ = ctx.populations(out=s["pops"])
        if case["tol"] > 0:
            return {"n": _kept(n, case), "status": status}
        return {"n": _kept(n, case), "iters": iters, "status": status}
    if kind == "prd":
        ctx.iterate(maxiter=case["maxiter"], tol=0.0, precision=case["precision"], prd_eps0=0.05,
                    prd_hybrid=case["hybrid"])
        n, iters, status, _ = ctx.populations(out=s["pops"])
        return {"n": _kept(n, case), "iters": iters, "status": status}
    if kind == "solve":
        ctx.load_columns(s["cols"], on_device=True)
        ctx.solve(precision=case["precision"])
        n, _, status, _ = ctx.populations(out=s["pops"])
        return {"n": _kept(n, case), "status": status}
    if kind == "load":
        ctx.load_columns(s["cols"], on_device=True)
        return {"n": ctx.populations(out=s["pops"])[0]}
    if kind == "spectrum":
        return {"I": _kept(ctx.emergent_spectrum(case["mu"], s["lam"], precision=case["precision"], out=s["out"]),
                           case)}
    if kind == "stokes":
        return {"IQUV": _kept(ctx.emergent_stokes(LINE_HALPHA, 1.5, *s["field"], s["lam"],
                                                  precision=case["precision"], out=s["out"]), case)}
    ctx.surrogate_set_state(s["weights"])
    st = ctx.surrogate_train(epochs=1, batch=case["batch"], seed=3)
    return {"state": ctx.surrogate_state(), "loss": st["loss_last_epoch"]}


# ---- work a pass cannot do without -----------------------------------------------------------------------------------
def work(case):
    atom, ncol, N = _atom(case), case["ncol"], case["ndep"]
    L, nline, ncont = atom["nlev"], len(atom["line_l"]), len(atom["cont_l"])
    nlam, nmu = int(sum(atom["line_nlambda"]) + sum(atom["cont_nlambda"])), atom["nmu"]
    pts = float(ncol) * N
    cols = 4 * 8 * pts                                   # z, T, n_H, v_z
    pops = 8 * L * pts
    # per point and iteration: opacity, source function, short-characteristics step and rate terms, both directions
    sweep = 2 * 30.0 * pts * nlam * nmu
    per_it = sweep + pts * (2.0 * L ** 3 / 3 + 2 * L * L)
    rates = 8 * 2 * (nline + ncont) * pts                # collisional rates
    if case["kind"] == "iterate":
        nit = case["maxiter"] if case["tol"] == 0 else 36
        return dict(bytes=cols + 2 * pops + rates, flops=nit * per_it)
    if case["kind"] == "solve":
        return dict(bytes=cols + pops, flops=36 * per_it)
    if case["kind"] == "prd":
        # per PRD line: the redistribution integral of every point over the line, each iteration, and its
        # kernel (half the pairs, a quadrature of some 100 operations each) once per column
        red = 2 * pts * case["npoint"] ** 2
        return dict(bytes=cols + 2 * pops + rates, flops=case["maxiter"] * (per_it + 2 * red) + 100 * red / 2)
    if case["kind"] == "load":
        return dict(bytes=2 * cols + 2 * 8 * pts + 2 * pops + rates, flops=pts * 60 * (nline + ncont))
    if case["kind"] == "spectrum":
        return dict(bytes=cols + 2 * pops + 8.0 * ncol * case["nlam"], flops=60.0 * pts * case["nlam"])
    if case["kind"] == "stokes":
        return dict(bytes=cols + 2 * pops + 3 * 8 * pts + 32.0 * ncol * case["nlam"],
                    flops=300.0 * pts * case["nlam"])
    nin, h, nout = 4 * N, 512, L * N
    w = nin * h + 2 * h * h + h * nout
    steps = ncol // case["batch"] if ncol >= case["batch"] else 1
    return dict(bytes=cols + 2 * pops + steps * 4.0 * 8 * w, flops=6.0 * w * steps * min(case["batch"], ncol))


# ---- the same results in 64 bits, by plain torch ---------------------------------------------------------------------
_H, _C, _K, _Q, _ME = 6.62607015e-34, 2.99792458e8, 1.380649e-23, 1.602176634e-19, 9.1093837015e-31
_EPS0, _AMU, _SIGT = 8.8541878128e-12, 1.66053906660e-27, 6.6524587321e-29


def _faddeeva(x, y):
    """w(x + iy), y > 0, by modified trapezoidal rules (Al Azah & Chandler-Wilde 2021), N = 11."""
    x, y = torch.broadcast_tensors(x, y)
    ax = x.abs()
    z = torch.complex(ax, y)
    z2 = z * z
    N = 11
    h = math.sqrt(math.pi / (N + 1))
    mid = torch.zeros_like(z)
    trap = torch.zeros_like(z)
    for k in range(N + 1):
        t = (k + 0.5) * h
        mid = mid + math.exp(-t * t) / (z2 - t * t)
        if k:
            tau = k * h
            trap = trap + math.exp(-tau * tau) / (z2 - tau * tau)
    mid = (2j * h / math.pi) * z * mid
    trap = (2j * h / math.pi) * z * trap + 1j * h / (math.pi * z)
    e = 2.0 * torch.exp(-z2)
    g = torch.exp(-2j * math.pi / h * z)
    frac = (ax / h) - torch.floor(ax / h)
    use_t = (frac >= 0.25) & (frac <= 0.75)
    # near a pole of one rule the other one is used
    w = torch.where(use_t, trap + e / (1.0 - g), mid + e / (1.0 + g))
    w = torch.where(y >= torch.clamp(ax, min=math.pi / h), mid, w)
    return torch.complex(w.real, torch.sign(x) * w.imag)


class _Model:
    """Grid, rates and LTE state of one atom and one set of columns, FP64."""

    def __init__(self, atom, cols):
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
        self.atom, self.L = atom, atom["nlev"]
        E, g = np.asarray(atom["E_J"]), np.asarray(atom["g"])
        ic = self.L - 1
        self.mass = atom["mass_amu"] * _AMU
        vD = math.sqrt(2 * _K * atom["T_ref"] / self.mass)
        self.tr = []
        nus = []
        for i, (l, u) in enumerate(zip(atom["line_l"], atom["line_u"])):
            nu0 = (E[u] - E[l]) / _H
            f = atom["line_f"][i]
            A = 2 * math.pi * _Q ** 2 * nu0 ** 2 / (_EPS0 * _ME * _C ** 3) * (g[l] / g[u]) * f
            Bul = A * _C ** 2 / (2 * _H * nu0 ** 3)
            d = nu0 / _C * vD
            q = atom["line_qwing"][i]
            s = -1.0 + 2.0 * np.arange(atom["line_nlambda"][i]) / (atom["line_nlambda"][i] - 1)
            nus.append(nu0 + q * np.sinh(5.0 * s) / math.sinh(5.0) * d)
            self.tr.append(dict(kind=0, l=int(l), u=int(u), nu0=nu0, A=A, Bul=Bul, Blu=Bul * g[u] / g[l], f=f,
                                lo=nu0 - q * d, hi=nu0 + q * d, la=(math.log(atom["line_a_top"][i]),
                                                                    math.log(atom["line_a_bot"][i]))))
        for i, l in enumerate(atom["cont_l"]):
            nu0 = (E[ic] - E[l]) / _H
            r = atom["cont_ratio"][i]
            nus.append(nu0 * r ** (np.arange(atom["cont_nlambda"][i]) / (atom["cont_nlambda"][i] - 1)))
            self.tr.append(dict(kind=1, l=int(l), u=ic, nu0=nu0, alpha0=atom["cont_alpha0"][i], lo=nu0, hi=nu0 * r))
        own = np.concatenate([np.full(len(x), i) for i, x in enumerate(nus)])
        self.nu = np.concatenate(nus)
        for i, tr in enumerate(self.tr):
            on = np.nonzero((own == i) | ((self.nu >= tr["lo"] * (1 - 1e-13)) & (self.nu <= tr["hi"] * (1 + 1e-13))))[0]
            o = np.argsort(self.nu[on], kind="stable")
            v = self.nu[on][o]
            w = np.zeros(len(on))
            w[o] = 0.5 * (np.append(v[1:], v[-1]) - np.append(v[:1], v[:-1]))
            tr["idx"], tr["w"] = torch.as_tensor(on, device="cuda"), t(w)
        x, w = np.polynomial.legendre.leggauss(atom["nmu"])
        self.mu, self.wmu = 0.5 * (x + 1), 0.5 * w
        self.z, self.T, self.nH, self.vz = (t(cols[k]) for k in ("z", "T", "nH", "vz"))
        self.N = self.T.shape[1]
        T, nH = self.T, self.nH
        kT = _K * T
        self.lam3 = (_H * _H / (2 * math.pi * _ME * kT)) ** 1.5
        phi = [g[i] / (2 * g[ic]) * self.lam3 * torch.exp((E[ic] - E[i]) / kT) for i in range(ic)]
        Phi = sum(phi)
        b = 1 + atom["metal_floor"] * nH * Phi
        self.ne = 2 * nH / (b + torch.sqrt(b * b + 4 * Phi * nH)) + atom["metal_floor"] * nH
        nc = nH / (1 + self.ne * Phi)
        self.ns = torch.stack([nc * self.ne * p for p in phi] + [nc], 1)          # [ncol][L][N]
        self.vth = torch.sqrt(2 * kT / self.mass)
        sk = torch.arange(self.N, dtype=torch.float64, device="cuda") / max(1, self.N - 1)
        for tr in self.tr:
            if tr["kind"] == 0:
                tr["a"] = torch.exp((1 - sk) * tr["la"][0] + sk * tr["la"][1])

    def collisions(self, T=None):
        T, ne = self.T, self.ne
        out = []
        Kc = _H * _H / ((2 * math.pi * _ME) ** 1.5 * math.sqrt(_K))
        for tr in self.tr:
            y = _H * tr["nu0"] / (_K * T)
            if tr["kind"] == 0:
                P = torch.clamp(0.276 * _exp_e1(y), min=0.2)
                Om = 8 * math.pi / math.sqrt(3.0) * (13.605693122994 * _Q / (_H * tr["nu0"])) * tr["f"] * P
                up = ne * Kc * Om / torch.sqrt(T) * torch.exp(-y)
            else:
                up = 1.55e11 * ne * tr["alpha0"] * 0.1 * torch.exp(-y) / (y * torch.sqrt(T))
            out.append((up, up * self.ns[:, tr["l"]] / self.ns[:, tr["u"]]))
        return out

    def background(self, nu):
        """Opacity and Planck function [ncol][N][nlam] at the frequencies nu."""
        nu = torch.as_tensor(nu, dtype=torch.float64, device="cuda")
        T, ne = self.T[..., None], self.ne[..., None]
        e2 = _Q * _Q / (4 * math.pi * _EPS0)
        Cff = e2 ** 3 * 4 / (3 * _ME * _H * _C) * math.sqrt(2 * math.pi / (3 * _K * _ME))
        lum = (_C / nu) * 1e6
        xx = torch.clamp(1 / lum - 1 / 1.6419, min=0.0)
        sx = torch.sqrt(xx)
        f = 152.519 + sx * (49.534 + sx * (-118.858 + sx * (92.536 + sx * (-34.194 + sx * 4.982))))
        hm = torch.where(lum < 1.6419, 1e-22 * lum ** 3 * xx * sx * f, torch.zeros_like(xx))
        nhm = 0.25 * self.ns[:, 0] * self.ne * self.lam3 * torch.exp(0.754 * _Q / (_K * self.T))
        x = _H * nu / (_K * T)
        om = -torch.expm1(-x)
        chi = (Cff * ne * self.ns[:, -1][..., None] / torch.sqrt(T) / nu ** 3 + nhm[..., None] * hm) * om + _SIGT * ne
        return chi, 2 * _H * nu ** 3 / _C ** 2 * torch.exp(-x) / om, torch.exp(-x)

    def profile(self, tr, nu, muz):
        v = (_C * ((nu - tr["nu0"]) / tr["nu0"]) - muz * self.vz[..., None]) / self.vth[..., None]
        H = _faddeeva(v, tr["a"][None, :, None]).real
        return H * _C / (math.sqrt(math.pi) * tr["nu0"]) / self.vth[..., None]


def _exp_e1(y):
    """e^y E1(y) for y > 0: the integral of e^-t / (t + y) over t by 200-point Gauss-Laguerre where y > 3, the series
    below."""
    s = torch.zeros_like(y)
    term = torch.ones_like(y)
    ys = torch.clamp(y, max=8.0)
    for n in range(1, 60):
        term = -term * ys / n
        s = s + term / n
    small = torch.exp(ys) * (-0.57721566490153286061 - torch.log(ys) - s)
    x, w = np.polynomial.laguerre.laggauss(60)
    big = torch.zeros_like(y)
    for a, b in zip(x, w):
        big = big + b / (a + y)
    return torch.where(y < 4.0, small, big)


def _sc(d):
    small = d < 0.2
    ds = torch.where(small, d, torch.zeros_like(d))
    s, t = torch.zeros_like(d), torch.ones_like(d)
    for n in range(2, 18):
        t = t / n if n == 2 else -t * ds / n
        s = s + t
    e0 = -torch.expm1(-d)
    dl = torch.where(small, torch.ones_like(d), d)
    wo = torch.where(small, ds * s, 1 - e0 / dl)
    omwo = torch.where(small, 1 - ds * s, e0 / dl)
    wu = torch.where(small, e0 - ds * s, e0 / dl - torch.exp(-d))
    return torch.exp(-d), wu, wo, omwo


def _bez(d):
    small = d < 1.0
    ds = torch.where(small, d, torch.ones_like(d))
    t = torch.ones_like(d)
    su, so, sc, sp = (torch.zeros_like(d) for _ in range(4))
    for n in range(22):
        if n:
            t = -t * ds / n
        su = su + t / (n + 3)
        so = so + t * 2 / ((n + 1) * (n + 2) * (n + 3))
        sc = sc + t * 2 / ((n + 2) * (n + 3))
        sp = sp + t * 2 / (n + 2)
    e = torch.exp(-d)
    dl = torch.where(small, torch.ones_like(d), d)
    wu = torch.where(small, d * su, (2 - e * (dl * dl + 2 * dl + 2)) / dl ** 2)
    wo = torch.where(small, d * so, (dl * dl - 2 * dl + 2 - 2 * e) / dl ** 2)
    wc = torch.where(small, d * sc, (2 * dl - 4 + (2 * dl + 4) * e) / dl ** 2)
    om = torch.where(small, sp, 2 * (1 - e * (1 + dl)) / dl ** 2)
    return e, wu, wo, wc, om


def _mali(atom, cols, maxiter, tol, formal):
    """Populations after the iteration of ``Context.iterate`` from LTE with order-2 Ng (delay 5, period 3)."""
    m = _Model(atom, cols)
    nc, N, L, nl = m.T.shape[0], m.N, m.L, len(m.nu)
    nu = torch.as_tensor(m.nu, device="cuda")
    chib, B, ex = m.background(m.nu)
    dz = m.z[:, :-1] - m.z[:, 1:]
    C = m.collisions()
    rays = [(mu, d) for mu in m.mu for d in (0, 1)]
    wr = [0.5 * w for w in m.wmu for _ in (0, 1)]
    phi = [[m.profile(tr, nu[tr["idx"]], mu if d else -mu) for mu, d in rays] if tr["kind"] == 0 else None
           for tr in m.tr]
    cst = []
    for tr in m.tr:
        v = nu[tr["idx"]]
        if tr["kind"] == 0:
            h4 = _H * v / (4 * math.pi)
            cst.append(dict(c=tr["w"] * tr["Blu"], V=h4 * tr["Blu"], U=h4 * tr["A"],
                            E=torch.full_like(v, 2 * _H * tr["nu0"] ** 3 / _C ** 2), R=tr["Bul"] / tr["Blu"]))
        else:
            al = tr["alpha0"] * (tr["nu0"] / v) ** 3
            tw = 2 * _H * v ** 3 / _C ** 2
            G = (m.ns[:, tr["l"]] / m.ns[:, tr["u"]])[..., None] * ex[:, :, tr["idx"]]
            cst.append(dict(c=4 * math.pi * tr["w"] * al / (_H * v), V=al, U=tw * al * G, E=tw, R=G))
    n = m.ns.clone()
    hist, live = [], torch.ones(nc, dtype=torch.bool, device="cuda")
    hcount = torch.zeros(nc, dtype=torch.long, device="cuda")
    for it in range(1, maxiter + 1):
        G = torch.zeros(nc, N, L, L, dtype=torch.float64, device="cuda")
        for (up, dn), tr in zip(C, m.tr):
            G[:, :, tr["u"], tr["l"]] += up
            G[:, :, tr["l"], tr["u"]] += dn
        X = [n[:, tr["l"]][..., None] - k["R"] * n[:, tr["u"]][..., None] for tr, k in zip(m.tr, cst)]
        for r, (mu, d) in enumerate(rays):
            chi, eta = chib.clone(), chib * B
            ch, U = [], []
            for j, (tr, k) in enumerate(zip(m.tr, cst)):
                p = phi[j][r] if phi[j] is not None else 1.0
                ch.append(k["V"] * p * X[j])
                U.append(k["U"] * p * torch.ones_like(X[j]))
                chi[:, :, tr["idx"]] += ch[j]
                eta[:, :, tr["idx"]] += n[:, tr["u"]][..., None] * U[j]
            S = eta / chi
            Ieff, psi, om = torch.empty_like(chi), torch.empty_like(chi), torch.empty_like(chi)
            order = list(range(N)) if d == 0 else list(range(N - 1, -1, -1))
            k0 = order[0]
            if d == 0:
                I = torch.zeros_like(chi[:, 0])
            else:
                I = B[:, -1] + mu * (B[:, -1] - B[:, -2]) / (0.5 * (chi[:, -1] + chi[:, -2]) * dz[:, -1:])
            Ieff[:, k0], psi[:, k0], om[:, k0] = I, 0.0, 1.0
            dt = 0.5 * (chi[:, 1:] + chi[:, :-1]) * dz[..., None] / mu           # between k and k + 1
            for s in range(1, N):
                k, kp = order[s], order[s - 1]
                du = dt[:, min(k, kp)]
                bg = chib[:, k] * B[:, k] / chi[:, k]
                if formal == 0:
                    e, wu, wo, omw = _sc(du)
                    base = I * e + wu * S[:, kp]
                else:
                    e, wu, wb, wc, omw = _bez(du)
                    if s + 1 < N:
                        kd = order[s + 1]
                        dd = dt[:, min(k, kd)]
                        a1, a2 = (S[:, k] - S[:, kp]) / du, (S[:, kd] - S[:, k]) / dd
                        al = (1 + dd / (du + dd)) / 3
                        den = al * a2 + (1 - al) * a1
                        ok = a1 * a2 > 0
                        der = torch.where(ok, a1 * a2 / torch.where(ok, den, torch.ones_like(den)),
                                          torch.zeros_like(du))
                        ctl = S[:, k] - 0.5 * du * der
                        ctl = torch.maximum(torch.minimum(ctl, torch.maximum(S[:, k], S[:, kp])),
                                            torch.minimum(S[:, k], S[:, kp]))
                    else:
                        ctl = 0.5 * (S[:, k] + S[:, kp])
                    base = I * e + wu * S[:, kp] + wc * (ctl - S[:, k])
                    wo = wb + wc
                I = base + wo * S[:, k]
                Ieff[:, k], psi[:, k], om[:, k] = base + wo * bg, wo / chi[:, k], omw
            for j, (tr, k) in enumerate(zip(m.tr, cst)):
                ix = tr["idx"]
                p = phi[j][r] if phi[j] is not None else 1.0
                cw = k["c"] * wr[r] * p
                Ij, pj = Ieff[:, :, ix], psi[:, :, ix]
                f = om[:, :, ix] + pj * (chi[:, :, ix] - ch[j])
                G[:, :, tr["u"], tr["l"]] += (cw * Ij).sum(-1)
                G[:, :, tr["l"], tr["u"]] += (cw * k["R"] * (k["E"] * f + Ij)).sum(-1)
                for j2, t2 in enumerate(m.tr):
                    if j2 == j:
                        continue
                    on = torch.isin(ix, t2["idx"])
                    if not bool(on.any()):
                        continue
                    at = torch.searchsorted(t2["idx"], ix[on])
                    x = (((cw * X[j]) * pj)[:, :, on] * U[j2][:, :, at]).sum(-1)
                    if tr["l"] != t2["u"]:
                        G[:, :, tr["l"], t2["u"]] -= x
                    if tr["u"] != t2["u"]:
                        G[:, :, tr["u"], t2["u"]] += x
        eye = torch.eye(L, dtype=torch.bool, device="cuda")
        G = torch.where(eye, torch.zeros_like(G), G)
        G = G - torch.diag_embed(G.sum(-2))
        sc = n.transpose(1, 2)                                                   # [nc][N][L]
        big = torch.nn.functional.one_hot(sc.argmax(-1), L).bool()
        G = torch.where(big[..., None], torch.ones_like(G), G) * sc[..., None, :]
        rhs = torch.where(big, m.nH[..., None], torch.zeros_like(sc))
        mx = G.abs().amax(-1, keepdim=True)
        new = (torch.linalg.solve(G / mx, rhs[..., None] / mx)[..., 0] * sc).transpose(1, 2)
        dmax = ((new - n).abs() / new).amax((1, 2))
        conv = dmax < tol
        hist.insert(0, new.clone())
        hist = hist[:4]
        hcount = torch.clamp(hcount + 1, max=4)
        if it >= 5 and len(hist) == 4 and (it - 5) % 3 == 0:
            x0, x1, x2, x3 = (h.reshape(nc, -1) for h in hist)
            d0, d1, d2 = x0 - x1, x1 - x2, x2 - x3
            p, q = d0 - d1, d0 - d2
            a11, a12, a22, b1, b2 = ((u * v).sum(-1) for u, v in ((p, p), (p, q), (q, q), (d0, p), (d0, q)))
            det = a11 * a22 - a12 * a12
            ca, cb = (b1 * a22 - b2 * a12) / det, (a11 * b2 - a12 * b1) / det
            acc = (1 - ca - cb)[:, None] * x0 + ca[:, None] * x1 + cb[:, None] * x2
            ok = ~conv & (hcount >= 4) & torch.isfinite(acc).all(-1) & (acc > 0).all(-1)
            new = torch.where(ok[:, None, None], acc.reshape(new.shape), new)
            hist[0] = new.clone()
            hcount = torch.where(ok, torch.ones_like(hcount), hcount)
        n = torch.where(live[:, None, None], new, n)
        live = live & ~conv
        if not bool(live.any()):
            break
    return n


def _spectrum(m, n, lam, mu, skip=-1):
    """chi, eta, B [ncol][N][nlam] of every transition but ``skip``, at direction cosine mu upward."""
    nu = torch.as_tensor(_C / lam, dtype=torch.float64, device="cuda")
    chi, B, ex = m.background(nu)
    eta = chi * B
    for i, tr in enumerate(m.tr):
        on = torch.nonzero((nu >= tr["lo"] * (1 - 1e-13)) & (nu <= tr["hi"] * (1 + 1e-13)))[:, 0]
        if i == skip or not len(on):
            continue
        v = nu[on]
        lo, up = n[:, tr["l"]][..., None], n[:, tr["u"]][..., None]
        if tr["kind"] == 0:
            p = m.profile(tr, v, mu) * (_H * v / (4 * math.pi))
            chi[:, :, on] += p * (lo * tr["Blu"] - up * tr["Bul"])
            eta[:, :, on] += up * tr["A"] * p
        else:
            al = tr["alpha0"] * (tr["nu0"] / v) ** 3
            G = (m.ns[:, tr["l"]] / m.ns[:, tr["u"]])[..., None] * ex[:, :, on]
            chi[:, :, on] += al * (lo - up * G)
            eta[:, :, on] += up * G * al * 2 * _H * v ** 3 / _C ** 2
    return nu, chi, eta, B


def _exact_spectrum(m, n, case):
    lam, mu = _wavelengths(case), case["mu"]
    _, chi, eta, B = _spectrum(m, n, lam, mu)
    S, dz, N = eta / chi, m.z[:, :-1] - m.z[:, 1:], m.N
    I = B[:, -1] + mu * (B[:, -1] - B[:, -2]) / (0.5 * (chi[:, -1] + chi[:, -2]) * dz[:, -1:])
    for k in range(N - 2, -1, -1):
        e, wu, wo, _ = _sc(0.5 * (chi[:, k] + chi[:, k + 1]) * dz[:, k:k + 1] / mu)
        I = I * e + wu * S[:, k + 1] + wo * S[:, k]
    return I


def _exact_stokes(m, n, case, field):
    lam = _wavelengths(case)
    nu, chi, eta, B = _spectrum(m, n, lam, 1.0, skip=LINE_HALPHA)
    tr = m.tr[LINE_HALPHA]
    Bf, th, az = (torch.as_tensor(x, device="cuda")[..., None] for x in field)
    dnu = tr["nu0"] * m.vth[..., None] / _C
    lo, up = n[:, tr["l"]][..., None], n[:, tr["u"]][..., None]
    net = lo * tr["Blu"] - up * tr["Bul"]
    kl, Sl = net * (_H * nu / (4 * math.pi)) / (math.sqrt(math.pi) * dnu), up * tr["A"] / net
    v = (_C * ((nu - tr["nu0"]) / tr["nu0"]) - m.vz[..., None]) / m.vth[..., None]
    vB = 1.5 * _Q / (4 * math.pi * _ME) * Bf / dnu
    a = tr["a"][None, :, None]
    b, p, r = _faddeeva(v - vB, a), _faddeeva(v, a), _faddeeva(v + vB, a)
    s2, ct, c2, n2 = torch.sin(th) ** 2, torch.cos(th), torch.cos(2 * az), torch.sin(2 * az)
    lI = 0.5 * kl * (p.real * s2 + 0.5 * (b.real + r.real) * (1 + ct * ct))
    lq = 0.5 * kl * (p.real - 0.5 * (b.real + r.real)) * s2
    rq = 0.5 * kl * (p.imag - 0.5 * (b.imag + r.imag)) * s2
    lV, rV = 0.5 * kl * (r.real - b.real) * ct, 0.5 * kl * (r.imag - b.imag) * ct
    eI = chi + lI
    eQ, eU, eV, rQ, rU, rV = (x / eI for x in (lq * c2, lq * n2, lV, rq * c2, rq * n2, rV))
    S = torch.stack([(eta + Sl * lI) / eI, Sl * eQ, Sl * eU, Sl * eV], -1)
    o = torch.zeros_like(eQ)
    Kp = torch.stack([torch.stack(x, -1) for x in ((o, eQ, eU, eV), (eQ, o, rV, -rU), (eU, -rV, o, rQ),
                                                   (eV, rU, -rQ, o))], -2)
    dz, N = m.z[:, :-1] - m.z[:, 1:], m.N
    I = torch.zeros_like(S[:, 0])
    I[..., 0] = B[:, -1] + (B[:, -1] - B[:, -2]) / (0.5 * (eI[:, -1] + eI[:, -2]) * dz[:, -1:])
    one = torch.eye(4, dtype=torch.float64, device="cuda")
    for k in range(N - 2, -1, -1):
        e, wu, wo, _ = (x[..., None] for x in _sc(0.5 * (eI[:, k] + eI[:, k + 1]) * dz[:, k:k + 1]))
        rhs = e * I + wu * (S[:, k + 1] - (Kp[:, k + 1] @ I[..., None])[..., 0]) + wo * S[:, k]
        I = torch.linalg.solve(one + wo[..., None] * Kp[:, k], rhs)
    return I


def _chunks(case, cols, size):
    for a in range(0, case["ncol"], size):
        yield slice(a, min(a + size, case["ncol"])), {k: v[a:a + size] for k, v in cols.items()}


def exact(case, seed):
    kind = case["kind"]
    # a redistribution solve, a whole convergent solve of many columns and a training run (steps of a normalised
    # gradient, from 16-bit activations) have no 64-bit result within the time or at all
    if kind in ("prd", "solve", "train"):
        return None
    atom, cols = _atom(case), _columns(case, seed)
    if kind == "load":
        return {"n": torch.cat([_Model(atom, c).ns for _, c in _chunks(case, cols, 16384)])}
    if kind == "iterate":
        n = torch.cat([_mali(atom, c, case["maxiter"], case["tol"], case["formal"])
                       for _, c in _chunks(case, cols, 125)])
        return {"n": n, "status": None} if case["tol"] > 0 else {"n": n, "iters": None, "status": None}
    dep = _departures(case, atom["nlev"], seed)
    field = _fields(case, seed) if kind == "stokes" else None
    out = []
    for at, c in _chunks(case, cols, 256 if kind == "spectrum" else 64):
        m = _Model(atom, c)
        n = m.ns * torch.as_tensor(dep[at], device="cuda")
        out.append(_exact_spectrum(m, n, case) if kind == "spectrum"
                   else _exact_stokes(m, n, case, [x[at] for x in field]))
    return {"I" if kind == "spectrum" else "IQUV": torch.cat(out)}
