"""The work that programs give this framework, as measured cases.

A lattice program builds a lattice, gives it initial fluctuations, evolves it in
stretches of some tens of steps and looks at t, a and a' between stretches; now
and then it takes the volume averages, the spectra and the energy density field.
Scans over couplings run many lattices as one ensemble, and fits take the
gradient of an observable with respect to the initial fluctuations. Each case is
one such call sequence through the Python classes:

* ``steps``: ``Lattice.evolve`` and the scalars (7 or 27 points, FP32 or FP64
  fields, phi stored whole or split, eq. scale, the L = 1/H form or static space);
* ``ensemble``: ``Ensemble.evolve`` and the members' states;
* ``gradient``: ``Lattice.adjoint`` from a given state;
* ``diagnostics``: energies, both spectra and the energy density field;
* ``init``: ``Lattice.init_fields``.

``prepare`` draws the state on the GPU: the inflaton near its homogeneous value
with Gaussian fluctuations, chi fluctuating about zero, a' from the Friedmann
equation. ``exact`` restates the scheme with torch in 64 bits.
"""
from __future__ import annotations

import math

import torch

from paper_0911_5692_gb300.lattice import Ensemble, Lattice
from paper_0911_5692_gb300.workloads import ensemble_64, lphi4, m2phi2

MODELS = {"lphi4": lphi4, "m2phi2": m2phi2}


def listed():
    return [
        # the FP64 reference run at 32^3 (1000 steps), looked at every 100 steps
        dict(name="steps_32_fp64", kind="steps", model="lphi4", n=32, precision=64, split=0, stencil=7, expansion=1,
             steps=100),
        # a quick look at a model on a small lattice whose side is no power of two
        dict(name="steps_100", kind="steps", model="m2phi2", n=100, precision=32, split=1, stencil=7, expansion=1,
             steps=50),
        # an accuracy run in FP64 at a medium side
        dict(name="steps_128_fp64", kind="steps", model="lphi4", n=128, precision=64, split=0, stencil=7, expansion=1,
             steps=40),
        # the chaotic-inflation run at 256^3, the configuration of the paper's timing
        dict(name="steps_256", kind="steps", model="m2phi2", n=256, precision=32, split=1, stencil=7, expansion=1,
             steps=64),
        # a production run between the two power-of-two sides
        dict(name="steps_384", kind="steps", model="lphi4", n=384, precision=32, split=1, stencil=7, expansion=1,
             steps=40),
        # the largest production run: the benchmark's lattice
        dict(name="steps_512", kind="steps", model="lphi4", n=512, precision=32, split=1, stencil=7, expansion=1,
             steps=40),
        # the paper's own Laplacian
        dict(name="steps_256_27", kind="steps", model="m2phi2", n=256, precision=32, split=1, stencil=27, expansion=1,
             steps=40),
        # DEFROST's scale-factor form
        dict(name="steps_256_lform", kind="steps", model="m2phi2", n=256, precision=32, split=1, stencil=7,
             expansion=2, steps=40),
        # a scan over couplings: 64 lattices of sides 32 to 96 in one launch
        dict(name="ensemble_64", kind="ensemble", members=64, side0=32, side1=48, side2=64, side3=96, steps=200),
        # the gradient of <chi^2> with respect to the initial fluctuations
        dict(name="gradient_128", kind="gradient", n=128, precision=32, steps=100),
        # what a run writes out every few hundred steps
        dict(name="diagnostics_256", kind="diagnostics", model="lphi4", n=256, precision=32, split=1, stencil=7,
             bins=128),
        # the start of every run: Gaussian vacuum fluctuations
        dict(name="init_256", kind="init", model="lphi4", n=256, precision=32, split=1, stencil=7),
    ]


def _side(rng, lo, hi):
    """A lattice side, a multiple of 4, spread over the logarithm of [lo, hi]."""
    return 4 * max(1, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 4))


def draw(rng):
    kind = rng.choice(["steps"] * 6 + ["ensemble", "gradient", "diagnostics", "init"])
    model = rng.choice(["lphi4", "m2phi2"])
    precision = 64 if rng.random() < 0.25 else 32
    split = 1 if precision == 32 and rng.random() < 0.7 else 0
    stencil = 27 if rng.random() < 0.25 else 7
    if kind == "steps":
        expansion = rng.choice([1, 1, 1, 1, 2, 0])
        if precision == 64:
            n = _side(rng, 16, 192)
        elif rng.random() < 0.3:
            n = rng.choice([32, 64, 128, 256, 512])
        else:
            n = _side(rng, 24, 512)
        # at most a fifth of the largest listed case's site updates, so that the slower forms cost no more than it
        most = int((0.02 if precision == 64 else 0.2) * 40 * 512 ** 3 / n ** 3)
        return dict(kind=kind, model=model, n=n, precision=precision, split=split, stencil=stencil,
                    expansion=expansion, steps=max(1, min(rng.randint(20, 100), most)))
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(4, 64), side0=_side(rng, 16, 96), side1=_side(rng, 16, 96),
                    side2=_side(rng, 16, 96), side3=_side(rng, 16, 96), steps=rng.randint(40, 100))
    if kind == "gradient":
        precision = 64 if rng.random() < 0.2 else 32
        return dict(kind=kind, n=_side(rng, 16, 64 if precision == 64 else 160), precision=precision,
                    steps=rng.randint(10, 60))
    if kind == "diagnostics":
        n = _side(rng, 32, 256)
        return dict(kind=kind, model=model, n=n, precision=precision, split=split, stencil=stencil,
                    bins=rng.choice([n // 2, n]))
    return dict(kind=kind, model=model, n=_side(rng, 32, 256), precision=precision, split=split, stencil=stencil)


# ---- inputs

def _params(case, seed=0):
    p = MODELS[case.get("model", "lphi4")](case["n"], precision=case["precision"], seed=seed,
                                           expansion=case.get("expansion", 1), split=case.get("split", 0))
    p["stencil"] = case.get("stencil", 7)
    return p


def _members(case, seed):
    sides = [case["side%d" % i] for i in range(4)]
    out = []
    for i, p in enumerate(ensemble_64(split=1)[:case["members"]]):
        n = sides[i % 4]
        out.append(dict(p, n=n, dt=p["L"] / n / 20.0, seed=seed + i))
    return out


def _program_units(p):
    """The rescaling of Sec. II.B and the program-unit potential's constants."""
    beta = 4 if p["model"] == 0 else 2
    cpl = p["lam"] if p["model"] == 0 else p["m"] ** 2
    phi0 = p["phi0"][0]
    A, B = 1.0 / phi0, math.sqrt(cpl) * abs(phi0) ** (beta / 2 - 1)
    r, s = 6.0 / (2 + beta), 3.0 * (2 - beta) / (2 + beta)
    dx = p["L"] / p["n"]
    return dict(beta=beta, cpl=cpl, A=A, B=B, r=r, s=s, dx=dx, dt=p["dt"], g8A2=p["eight_pi_G"] / A ** 2,
                cdom0=cpl * A ** (2 - beta) / B ** 2, pdom=2 * r - 2 * s - beta * r, kappa0=p["g2"] / (A * B) ** 2,
                pint=-2 * r - 2 * s, expansion=p.get("expansion", 1), stencil=p.get("stencil", 7))


def _homogeneous(p):
    """phi = 1 rolling, and a' from the Friedmann equation: (P, Pi, a')."""
    u = _program_units(p)
    v = -0.7 if p["model"] else -0.5
    ad = math.sqrt(u["g8A2"] / 3.0 * (0.5 * v * v + 1.0 / u["beta"])) if u["expansion"] else 0.0
    return 1.0, v + u["r"] * ad, ad


def _state(p, seed):
    """Stored arrays f_phi, f_chi, pi_phi, pi_chi (flat, in the lattice's type), and (P, Pi, a'): on a split lattice
    phi and its momentum are the fluctuations about P and Pi, else whole."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    P, Pi, ad = _homogeneous(p)
    dtype = torch.float32 if p["precision"] == 32 else torch.float64
    arrays = [torch.randn(p["n"] ** 3, generator=gen, device="cuda", dtype=dtype).mul_(1e-4) for _ in range(4)]
    if not p.get("split", 0):
        arrays[0] += P
        arrays[2] += Pi
    return arrays, (P, Pi, ad)


def _load(lat, p, seed):
    arrays, (P, Pi, ad) = _state(p, seed)
    torch.cuda.synchronize()
    lat.set_scalars(t=0.0, a=1.0, ad=ad, step=0)
    if p.get("split", 0):
        lat.set_background(P, Pi)
    lat.upload_state(*arrays)
    lat.sync()


_TUNED = set()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        members = _members(case, seed)
        ens = Ensemble(members)
        views = [ens.member(i) for i in range(len(ens))]
        for i, (lat, p) in enumerate(zip(views, members)):
            _load(lat, p, seed * 64 + i)
        key = tuple(sorted(p["n"] for p in members))
        if key not in _TUNED:   # a scan tunes its ensemble once; the library keeps the shape for the sides
            _TUNED.add(key)
            ens.tune()
        count = sum(p["n"] ** 3 for p in members)
        outs = [torch.empty(count, dtype=torch.float32, device="cuda") for _ in range(4)]
        cuts, at = [], 0
        for p in members:
            cuts.append([o[at:at + p["n"] ** 3] for o in outs])
            at += p["n"] ** 3
        torch.cuda.synchronize()
        return dict(kind=kind, case=case, ens=ens, views=views, outs=outs, cuts=cuts)
    p = _params(case, seed)
    lat = Lattice(p)
    state = dict(kind=kind, case=case, lat=lat)
    if kind == "gradient":
        state["start"], (_, _, state["ad"]) = _state(p, seed)
        torch.cuda.synchronize()
    elif kind != "init":
        _load(lat, p, seed)
    if kind == "diagnostics":
        shape = (p["n"],) * 3
        state["rho"] = torch.empty(shape, dtype=lat.dtype, device="cuda")
        state["p"] = torch.empty(shape, dtype=lat.dtype, device="cuda")
        torch.cuda.synchronize()
    return state


# ---- one pass

def _current(lat, scalars):
    """The state a program reads after a stretch of steps: the stored arrays of the current set, the scalars that are
    evolved in FP64, and the volume averages, which carry the precision of the lattice's own arithmetic."""
    par = scalars["step"] & 1
    out = dict(zip(("f_phi", "f_chi", "pi_phi", "pi_chi"), lat.buffers[4 * par:4 * par + 4]))
    out["time"] = [scalars["t"], scalars["a"], scalars["ad"]]
    out["averages"] = torch.tensor(scalars["S"], dtype=lat.dtype)
    out["step"] = scalars["step"]
    if lat.params.get("split", 0):
        out["mode"] = list(lat.background())
    if lat.params.get("expansion", 1) == 2:
        out["hubble_length"] = torch.tensor(lat.hubble_length(), dtype=lat.dtype)
    return out


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "steps":
        lat = state["lat"]
        lat.evolve(case["steps"])
        return _current(lat, lat.scalars())
    if kind == "ensemble":
        state["ens"].evolve(case["steps"])
        state["ens"].sync()
        scalars, modes = [], []
        for lat, cut in zip(state["views"], state["cuts"]):
            lat.download_state(*cut)
            s = lat.scalars()
            scalars.append([s["t"], s["a"], s["ad"]])
            modes.append(list(lat.background()))
        names = ("f_phi", "f_chi", "pi_phi", "pi_chi")
        return dict(zip(names, state["outs"]), time=torch.tensor(scalars, dtype=torch.float64),
                    mode=torch.tensor(modes, dtype=torch.float64))
    lat = state["lat"]
    if kind == "gradient":
        lat.set_scalars(t=0.0, a=1.0, ad=state["ad"], step=0)
        lat.upload_state(*state["start"])
        J, df, dpi, dg2 = lat.adjoint(case["steps"])
        # J and dJ/dg2 are sums over the lattice's own arithmetic: they have its precision
        return dict(J=torch.tensor(J, dtype=lat.dtype), df=df, dpi=dpi, dg2=torch.tensor(dg2 * 1e-9, dtype=lat.dtype))
    if kind == "diagnostics":
        energies = lat.energies()
        spectra = [lat.spectrum(field, case["bins"]) for field in (0, 1)]
        rho, p = lat.energy_field(state["rho"], state["p"])
        lat.sync()
        return dict(energies=energies, spectra=spectra, rho=rho, p=p)
    lat.init_fields()
    return _current(lat, lat.scalars())


# ---- what a pass cannot do without

def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        members = _members(case, 0)
        sites = sum(p["n"] ** 3 for p in members) * case["steps"]
        return dict(bytes=32 * sites, flops=60 * sites)
    n3, e = case["n"] ** 3, case["precision"] // 8
    if kind == "steps":   # read f and f' of both fields, write them
        per_site = 60 if case["stencil"] == 7 else 160
        return dict(bytes=8 * e * n3 * case["steps"], flops=per_site * n3 * case["steps"])
    if kind == "gradient":   # a step forward, and its reverse: f_k, f_{k-1} and the adjoints in, the adjoints out
        return dict(bytes=(8 + 12) * e * n3 * case["steps"], flops=180 * n3 * case["steps"])
    if kind == "diagnostics":   # the state in for the energies, a field in for each spectrum, the state in and rho, p out
        return dict(bytes=(4 + 2 + 6) * e * n3, flops=(200 + 10 * math.log2(n3)) * n3)
    # four arrays out; a forward and an inverse transform of each (2.5 N log2 N operations)
    return dict(bytes=4 * e * n3, flops=(4 * 2 * 2.5 * math.log2(n3) + 200) * n3)


# ---- the same in 64 bits

def _laplacian(f, u):
    """The configured Laplacian as a sum of neighbour differences (7 points) or of the weighted cube (27 points)."""
    inv = 1.0 / u["dx"] ** 2

    def pair(g, d):
        return torch.roll(g, 1, d) + torch.roll(g, -1, d)

    if u["stencil"] != 27:
        return (pair(f, 0) + pair(f, 1) + pair(f, 2) - 6.0 * f) * inv
    x = pair(f, 2)                       # the two x neighbours
    y, xy = pair(f, 1), pair(x, 1)       # and so on up to the corners
    faces, edges = x + y + pair(f, 0), xy + pair(x, 0) + pair(y, 0)
    return (14.0 * faces + 3.0 * edges + pair(xy, 0) - 128.0 * f) * (inv / 30.0)


def _averages(f, u, P):
    """<|grad f|^2> of both fields, <phi^beta / beta> and <phi^2 chi^2 / 2>; f[0] is measured from P."""
    grad = [-((g - g.mean()) * _laplacian(g - g.mean(), u)).mean() for g in f]
    phi = f[0] + P
    return grad + [(phi ** u["beta"]).mean() / u["beta"], (phi * f[1]).square().mean() / 2]


def _coefficients(u, a, ad, S):
    """a'(t + dt) and the field equation's coefficients cL, cF, cdom, kappa from the sums at the field time."""
    cdom, kappa = u["cdom0"] * a ** u["pdom"], u["kappa0"] * a ** u["pint"]
    if not u["expansion"]:
        return ad, ad, 1.0, 0.0, cdom, kappa
    r, s, dt = u["r"], u["s"], u["dt"]
    v = cdom * S[2] + kappa * S[3]
    c = u["g8A2"] * a ** (-2 * s - 2 * r - 1) * ((S[0] + S[1]) / 3 + a ** (2 * s + 2) * v)
    q = -(s + 2) / a
    alpha, gamma = dt * q / 4, 2 * ad + dt * c
    y = 2 * gamma / (1 + (1 - 4 * alpha * gamma) ** 0.5)
    half = y / 2
    cF = r * (s - r + 2) * (half / a) ** 2 + r * (q * half * half + c) / a
    return y - ad, half, a ** (-2 * s - 2), cF, cdom, kappa


def _force(u, f, phi, kappa, cdom):
    return cdom * phi ** (u["beta"] - 1) + kappa * phi * f[1] ** 2, kappa * phi ** 2 * f[1]


def _lform(u, a, ell, cF_before, f, pi, P, Pi):
    """The L = 1/H form's implicit midpoint equations: l(t + dt), cL, cF, cdom, kappa."""
    r, s, dt = u["r"], u["s"], u["dt"]
    cdom, kappa, cL = u["cdom0"] * a ** u["pdom"], u["kappa0"] * a ** u["pint"], a ** (-2 * s - 2)
    phi = f[0] + P
    force = _force(u, f, phi, kappa, cdom)
    w0 = dt / 2 * cF_before - r / ell
    whole = (phi, f[1])
    vel = [q + dt / 2 * (cL * _laplacian(g, u) - d) + w0 * h for q, g, d, h in zip((pi[0] + Pi, pi[1]), f, force, whole)]
    kin = float(sum(x.square().mean() for x in vel))
    cross = float(sum((x * h).mean() for x, h in zip(vel, whole)))
    square = float(sum(h.square().mean() for h in whole))
    V = float(cdom * (phi ** u["beta"]).mean() / u["beta"] + kappa * (phi * f[1]).square().mean() / 2)
    new, cF, g = ell, 0.0, u["g8A2"] / 3 * a ** (-2 * r)
    for _ in range(100):
        lam = (ell + new) / 2
        dw = dt / 2 * cF - r / lam - w0
        gam = g * (kin + 2 * dw * cross + dw * dw * square - V)
        cF, new = r * (2 - r) / lam ** 2 - r * gam, ell + dt * (s + 1 + gam * lam * lam)
    return new, cL, cF, cdom, kappa


def _evolve(p, f, pi, ad, steps, P=0.0, Pi=0.0):
    """`steps` leapfrog steps in 64 bits from t = 0, a = 1 of phi = P + f[0] and chi = f[1]: the fields, momenta,
    t, a, a', the homogeneous mode, the sums and l."""
    u = _program_units(p)
    dt = u["dt"]
    a, form = 1.0, u["expansion"] == 2
    ell = (a - dt / 2 * ad) / ad if form else 0.0
    cF = 0.0
    for k in range(steps):
        if form:
            ell_next, cL, cF, cdom, kappa = _lform(u, a, ell, cF, f, pi, P, Pi)
        else:
            S = [float(x) for x in _averages(f, u, P)]
            ad_next, _, cL, cF, cdom, kappa = _coefficients(u, a, ad, S)
        # the momenta's kick, measured from the mode's own
        lap = [_laplacian(g, u) for g in f]
        phi = f[0] + P
        inter = kappa * phi * f[1] ** 2
        d = f[0]
        dom = d * (phi * (phi + P) + P * P) if u["beta"] == 4 else d
        pi = [pi[0] + dt * (cL * lap[0] + cF * d - cdom * dom - inter),
              pi[1] + dt * (cL * lap[1] + cF * f[1] - kappa * phi ** 2 * f[1])]
        Pi = Pi + dt * (cF * P - cdom * P ** (u["beta"] - 1))
        f = [f[0] + dt * pi[0], f[1] + dt * pi[1]]
        P = P + dt * Pi
        if form:
            ell, ad = ell_next, a * math.expm1(dt / ell_next) / dt
            a = a + dt * ad
        elif u["expansion"]:
            ad = ad_next
            a = a + dt * ad
    return f, pi, steps * dt, a, ad, P, Pi, [float(x) for x in _averages(f, u, P)], ell


def _cube(arrays, n):
    return [x.double().view(n, n, n) for x in arrays]


def _exact_steps(p, seed, steps):
    arrays, (P, Pi, ad) = _state(p, seed)
    x = _cube(arrays, p["n"])
    del arrays
    if not p.get("split", 0):
        P = Pi = 0.0
    return _evolve(p, x[:2], x[2:], ad, steps, P, Pi)


def _whole_out(p, got):
    f, pi, t, a, ad, P, Pi, S, ell = got
    out = dict(zip(("f_phi", "f_chi", "pi_phi", "pi_chi"), [g.reshape(-1) for g in f + pi]))
    out["time"], out["averages"], out["step"] = [t, a, ad], torch.tensor(S, dtype=torch.float64), None
    if p.get("split", 0):
        out["mode"] = [P, Pi]
    if p.get("expansion", 1) == 2:
        out["hubble_length"] = torch.tensor(ell, dtype=torch.float64)
    return out


def _exact_gradient(p, seed, steps):
    from torch.utils.checkpoint import checkpoint
    u = _program_units(p)
    arrays, (_, _, ad) = _state(p, seed)
    x = [v.requires_grad_() for v in _cube(arrays, p["n"])]
    k0 = torch.tensor(u["kappa0"], dtype=torch.float64, device="cuda", requires_grad=True)
    dt = u["dt"]

    def step(f0, f1, p0, p1, a, ad, k0):
        w = dict(u, kappa0=k0)
        f = (f0, f1)
        lap = [_laplacian(g, w) for g in f]
        S = [-(g * l).mean() for g, l in zip(f, lap)]
        S += [(f0 ** u["beta"]).mean() / u["beta"], (f0 * f1).square().mean() / 2]
        ad, _, cL, cF, cdom, kappa = _coefficients(w, a, ad, S)
        force = _force(w, f, f0, kappa, cdom)
        p0 = p0 + dt * (cL * lap[0] + cF * f0 - force[0])
        p1 = p1 + dt * (cL * lap[1] + cF * f1 - force[1])
        return f0 + dt * p0, f1 + dt * p1, p0, p1, a + dt * ad, ad

    one = torch.ones((), dtype=torch.float64, device="cuda")
    now = (*x, one, one * ad)
    for _ in range(steps):
        now = checkpoint(step, *now, k0, use_reentrant=False)
    J = now[1].square().mean()
    g = torch.autograd.grad(J, x + [k0])
    return dict(J=J.detach(), df=torch.stack(g[:2]), dpi=torch.stack(g[2:4]), dg2=g[4] / (u["A"] * u["B"]) ** 2 * 1e-9)


def _shells(n):
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    return torch.sqrt(k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2)


def _exact_diagnostics(p, seed, bins):
    u, n = _program_units(p), p["n"]
    arrays, (P, Pi, ad) = _state(p, seed)
    x = _cube(arrays, n)
    f, pi = x[:2], x[2:]
    if not p.get("split", 0):
        P = Pi = 0.0
    dt, r, s, a = u["dt"], u["r"], u["s"], 1.0
    S = [float(v) for v in _averages(f, u, P)]
    _, half, cL, cF, cdom, kappa = _coefficients(u, a, ad, S)
    phi = f[0] + P
    force = _force(u, f, phi, kappa, cdom)
    h = half / a
    conv = u["B"] ** 2 / u["A"] ** 2 * a ** (2 * s - 2 * r)
    kin, grad = [], []
    for g, q, d, w in zip(f, (pi[0] + Pi, pi[1]), force, (phi, f[1])):
        kin.append((q + dt / 2 * (cL * _laplacian(g, u) + cF * w - d) - r * h * w) ** 2 / 2)
        # half the weighted squared differences to all the neighbours: L(g^2) - 2 g L(g)
        c = g - g.mean()
        grad.append(a ** (-2 * s - 2) / 4 * (_laplacian(c * c, u) - 2 * c * _laplacian(c, u)))
    pot = cdom * phi ** u["beta"] / u["beta"] + kappa * (phi * f[1]) ** 2 / 2
    rho = conv * (kin[0] + kin[1] + grad[0] + grad[1] + pot)
    pres = conv * (kin[0] + kin[1] - (grad[0] + grad[1]) / 3 - pot)
    H = u["B"] * a ** s * h
    mean = lambda v: float(v.mean())  # noqa: E731
    e = dict(t=dt / 2, a=a, ad=half, H=H, rho=mean(rho), p=mean(pres), pot=conv * mean(pot))
    e["w"], e["curv_resid"] = e["p"] / e["rho"], p["eight_pi_G"] * e["rho"] / (3 * H * H) - 1
    for i, w in enumerate((phi, f[1])):
        e["kin%d" % i], e["grad%d" % i], e["mean%d" % i] = conv * mean(kin[i]), conv * mean(grad[i]), mean(w)
        e["var%d" % i] = mean((w - w.mean()) ** 2)
    shell = _shells(n)
    b = torch.floor(shell + 0.5).long().reshape(-1)
    keep = b < bins
    count = torch.bincount(b[keep], minlength=bins).double()
    spectra = []
    for w in (phi, f[1]):
        power = torch.fft.fftn(w).abs().square().reshape(-1) / n ** 3
        total = [torch.zeros(bins, dtype=torch.float64, device="cuda").index_add_(0, b[keep], v[keep])
                 for v in (shell.reshape(-1) * (2 * math.pi / p["L"]), power)]
        spectra.append([t / count.clamp(min=1) for t in total] + [None])
    return dict(energies=e, spectra=spectra, rho=rho, p=pres)


def _philox(n, seed, field, quantity):
    """Two 32-bit words of Philox-4x32-10 for each site, as integers in [0, 2^32)."""
    m32 = 0xFFFFFFFF
    c = [torch.arange(n ** 3, dtype=torch.int64, device="cuda")]
    c += [torch.full_like(c[0], v) for v in (field, quantity, 0)]
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57   # the low 64 bits, which hold the whole product
        c = [((b >> 32) & m32) ^ c[1] ^ k0, b & m32, ((a >> 32) & m32) ^ c[3] ^ k1, a & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c[0], c[1]


def _exact_init(p, seed):
    u, n = _program_units(p), p["n"]
    phi0, dphi0 = p["phi0"], p["dphi0"]
    rho0 = dphi0[0] ** 2 / 2 + u["cpl"] / u["beta"] * phi0[0] ** u["beta"]
    ad = math.sqrt(p["eight_pi_G"] * rho0 / 3) / u["B"]
    fh = [u["A"] * v for v in phi0]
    ph = [u["A"] / u["B"] * v + u["r"] * ad * w for v, w in zip(dphi0, fh)]
    mass2 = [u["cdom0"] * (u["beta"] - 1) * fh[0] ** (u["beta"] - 2) + u["kappa0"] * fh[1] ** 2, u["kappa0"] * fh[0] ** 2]
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    sq = torch.sin(math.pi * k / n) ** 2
    s1, s2, s3 = sq[:, None, None], sq[None, :, None], sq[None, None, :]
    klat = 4 * (s1 + s2 + s3)
    if u["stencil"] == 27:
        klat = klat - 8 / 3 * (s1 * s2 + s1 * s3 + s2 * s3) + 32 / 15 * s1 * s2 * s3
    shell = _shells(n)
    inside = (shell > 0) & (shell <= n / 4.0)
    amp = u["A"] * u["B"] * u["dx"] ** -1.5 * p["fluct"]
    f, pi = [], []
    for i in range(2):
        w = torch.sqrt(klat / u["dx"] ** 2 + mass2[i])
        d = []
        for q in range(2):
            c0, c1 = _philox(n, seed, i, q)
            u1, u2 = (c0.double() + 0.5) / 2 ** 32, (c1.double() + 0.5) / 2 ** 32
            white = (torch.sqrt(-2 * torch.log(u1)) * torch.cos(2 * math.pi * u2)).view(n, n, n)
            scale = torch.where(inside, amp * (torch.rsqrt(2 * w) if q == 0 else torch.sqrt(w / 2)), 0.0)
            d.append(torch.fft.ifftn(torch.fft.fftn(white) * scale).real)
        bg = p.get("split", 0) and i == 0
        mom = (0.0 if bg else ph[i]) + d[1] + u["r"] * ad * d[0]
        pi.append(mom)
        f.append((0.0 if bg else fh[i]) + d[0] + u["dt"] / 2 * mom)
    P, Pi = (fh[0] + u["dt"] / 2 * ph[0], ph[0]) if p.get("split", 0) else (0.0, 0.0)
    return f, pi, 0.0, 1.0 + u["dt"] / 2 * ad, ad, P, Pi, [float(v) for v in _averages(f, u, P)], 0.0


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        got = [_exact_steps(p, seed * 64 + i, case["steps"]) for i, p in enumerate(_members(case, seed))]
        out = {name: torch.cat([g[j // 2][j % 2].reshape(-1) for g in got])
               for j, name in enumerate(("f_phi", "f_chi", "pi_phi", "pi_chi"))}
        out["time"] = torch.tensor([[g[2], g[3], g[4]] for g in got], dtype=torch.float64)
        out["mode"] = torch.tensor([[g[5], g[6]] for g in got], dtype=torch.float64)
        return out
    p = _params(case, seed)
    if kind == "steps":
        return _whole_out(p, _exact_steps(p, seed, case["steps"]))
    if kind == "gradient":
        return _exact_gradient(p, seed, case["steps"])
    if kind == "diagnostics":
        return _exact_diagnostics(p, seed, case["bins"])
    return _whole_out(p, _exact_init(p, seed))
