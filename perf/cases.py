"""The lattice stepper's work as its users have it done, one call sequence per case.

A case is one of four kinds:
  evolve   initial fields on the device -> set_initial, evolve(steps), energies, get_fields;
           model "expr_*" is a potential given as expressions (compiled at run time)
  linear   pycool_linear_evolve: the linearised evolution of lattice fields
  outputs  what a run writes at an output time: per-site energy density and pressure, the
           spectrum of every field and momentum, the energies
  serve    a batch of requests to the serving loop, submitted together and waited for

The lattice spacing and time step of a model are those of its workload in
paper_1201_5029_gb300.inputs at every lattice side n, so that any n is stable.
"""
import math
import random

import numpy as np
import torch

import paper_1201_5029_gb300 as P

STAGES = {2: 1, 4: 3, 6: 7, 8: 15}
# model: dx, dt, m_pl, parameters, background and momentum of the fields, noise
MODELS = {
    "chaotic2": dict(dx=10.0 / 128, dt=0.005, mpl=1.0, params=(1.0, 1.0e4), bg=(1.0, 0.0),
                     mom=(-0.5, 0.0), noise=1e-5),
    "oscillon": dict(dx=50.0 / 256, dt=0.02, mpl=100.0, params=(1.0, 1.0, 0.5), bg=(0.8,),
                     mom=(0.0,), noise=1e-4),
    "qball": dict(dx=200.0 / 256, dt=0.05, mpl=100.0, params=(1.0, -0.1, 1.0),
                  bg=(math.sqrt(2) * math.cos(0.3), math.sqrt(2) * math.sin(0.3)), mom=(0.0, 0.0),
                  noise=1e-6),
    "expr_phi4": dict(dx=20.0 / 64, dt=0.02, mpl=100.0, params=(1.0, 0.5), bg=(0.8,), mom=(0.0,),
                      noise=1e-4),
}
MODELS["expr_chaotic2"] = dict(MODELS["chaotic2"])
EXPRESSIONS = {
    "expr_chaotic2": ("0.5*p[0]*f0*f0 + 0.5*p[1]*f0*f0*f1*f1",
                      ("p[0]*f0 + p[1]*f0*f1*f1", "p[1]*f0*f0*f1")),
    "expr_phi4": ("0.5*p[0]*f0*f0 + 0.25*p[1]*f0*f0*f0*f0", ("p[0]*f0 + p[1]*f0*f0*f0",)),
}
_model_ids = {}   # a program compiles its potential once


def _evolve(name, n, model, order, steps, precision="fp64", stencil="7pt", time="conformal"):
    return dict(name=name, kind="evolve", n=n, model=model, order=order, steps=steps,
                precision=precision, stencil=stencil, time=time)


def listed():
    return [
        # the first small run of a model: 32^3 preheating, leapfrog, 100 steps
        _evolve("preheat32 fp64", 32, "chaotic2", 2, 100),
        # the paper's preheating runs: 128^3, fourth order, in both forms in use
        _evolve("preheat128 fp64", 128, "chaotic2", 4, 10),
        _evolve("preheat128 split", 128, "chaotic2", 4, 10, "split_fp32"),
        # oscillons, one field, 256^3, sixth order
        _evolve("oscillon256 fp64", 256, "oscillon", 6, 3),
        # the curvaton Q-ball, the largest workload: 256^3, two components, eighth order
        _evolve("qball256 fp64", 256, "qball", 8, 2),
        _evolve("qball256 split", 256, "qball", 8, 4, "split_fp32"),
        # a side chosen for the box, not for the hardware
        _evolve("preheat100 fp64", 100, "chaotic2", 4, 10),
        # the fourth-order stencil, for runs whose dispersion matters
        _evolve("preheat128 4th", 128, "chaotic2", 4, 10, "fp64", "4th"),
        # a model file's potential given as expressions
        _evolve("expr128", 128, "expr_chaotic2", 4, 10),
        # the linear stage before back-reaction, in one call
        dict(name="linear128", kind="linear", n=128, model="chaotic2", order=4, steps=100,
             stencil="7pt"),
        # an output time of the oscillon run
        dict(name="outputs256", kind="outputs", n=256, model="oscillon", precision="fp64",
             stencil="7pt"),
        # a batch of the serving mix's sizes up to 128^3
        dict(name="serve fp64", kind="serve", requests=12, mix=1, top=128, steps=40,
             precision="fp64"),
    ]


def _side(rng, lo, hi, by32):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi // 32 * 32, max(32, 32 * int(round(n / 32)))) if by32 else n


def draw(rng):
    kind = rng.choice(["evolve"] * 6 + ["expr", "linear", "outputs", "serve"])
    stencil = rng.choice(["7pt", "7pt", "7pt", "iso27", "4th"])
    by32 = rng.random() < 0.5
    order = rng.choice([2, 4, 6, 8])
    if kind in ("evolve", "expr"):
        expr = kind == "expr"
        n = _side(rng, 16, 160 if expr else 256, by32)
        model = rng.choice(["expr_phi4", "expr_chaotic2"] if expr
                           else ["chaotic2", "oscillon", "qball"])
        forms = ["fp64"] if expr else ["fp64", "fp64", "split_fp32"]
        precision = rng.choice(forms + (["split_dd"] if n % 32 == 0 and not expr else []))
        nf = len(MODELS[model]["bg"])
        most = 2.4e8 / (nf * n ** 3 * STAGES[order])   # well below the largest listed case
        steps = max(1, int(min(100.0, most) * rng.uniform(0.5, 1.0)))
        return dict(kind="evolve", n=n, model=model, order=order, steps=steps,
                    precision=precision, stencil=stencil,
                    time=rng.choice(["conformal", "conformal", "physical"]))
    if kind == "linear":
        return dict(kind="linear", n=_side(rng, 32, 160, by32),
                    model=rng.choice(["chaotic2", "oscillon", "qball"]),
                    order=rng.choice([2, 4]), steps=int(math.exp(rng.uniform(1.0, math.log(150)))),
                    stencil=stencil)
    if kind == "outputs":
        n = _side(rng, 32, 224, by32)
        return dict(kind="outputs", n=n, model=rng.choice(["chaotic2", "oscillon", "qball"]),
                    precision=rng.choice(["fp64", "split_fp32"] +
                                         (["split_dd"] if n % 32 == 0 else [])),
                    stencil=stencil)
    return dict(kind="serve", requests=rng.randint(4, 12), mix=rng.randint(2, 999),
                top=rng.choice([32, 64, 128]), steps=rng.randint(10, 40),
                precision=rng.choice(["fp64", "split_fp32"]))


# ---------------------------------------------------------------- the calls

def _config(model, n, order, precision, stencil, time="conformal"):
    m = MODELS[model]
    if model in EXPRESSIONS:
        if model not in _model_ids:
            _model_ids[model] = P.pycool_model_define(*EXPRESSIONS[model])
        model = _model_ids[model]
    return P.make_config(n, m["dx"] * n, model, m["params"], m["dt"], order=order,
                         precision=precision, stencil=stencil, mpl=m["mpl"], time_step=time)


def _fields(model, n, seed):
    """Homogeneous background plus white noise, phi and pi of shape (N_f, n, n, n)."""
    m = MODELS[model]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    out = []
    for base in (m["bg"], m["mom"]):
        b = torch.tensor(base, dtype=torch.float64, device="cuda").reshape(-1, 1, 1, 1)
        x = torch.randn((len(base), n, n, n), dtype=torch.float64, device="cuda", generator=g)
        out.append(b + m["noise"] * x)
    return out


def _requests(case):
    """The batch of a serve case: sides with the serving mix's weights up to `top`."""
    r = random.Random(case["mix"])
    sides, weights = zip(*[s for s in ((32, 0.4), (64, 0.3), (128, 0.15)) if s[0] <= case["top"]])
    out = []
    for i in range(case["requests"]):
        n = r.choices(sides, weights)[0] if i else sides[-1]
        order = r.choice([2, 4, 6, 8])
        most = max(1, int(6.0e7 / (n ** 3 * STAGES[order])))   # a few milliseconds of work each
        out.append(dict(n=n, model=r.choice(["chaotic2", "oscillon", "qball"]), order=order,
                        steps=min(most, r.randint(max(1, case["steps"] // 10), case["steps"]))))
    return out


class _Server:
    def __init__(self, budget, slots):
        self.handle = P.pycool_server_create(budget, slots)

    def __del__(self):
        P.pycool_server_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        reqs = _requests(case)
        jobs = []
        for i, q in enumerate(reqs):
            m = MODELS[q["model"]]
            jobs.append((_config(q["model"], q["n"], q["order"], case["precision"], "7pt"),
                         P.make_ic(m["bg"], m["mom"], m["noise"]), seed * 1000 + i, q["steps"],
                         len(m["bg"])))
        return dict(kind=kind, server=_Server(4 << 30, 64), jobs=jobs)
    phi, pi = _fields(case["model"], case["n"], seed)
    s = dict(kind=kind, phi=phi, pi=pi, steps=case.get("steps", 0))
    if kind == "linear":
        s["cfg"] = _config(case["model"], case["n"], case["order"], "fp64", case["stencil"])
        s["pa0"] = _root(case["model"], case["n"], phi.mean((1, 2, 3), keepdim=True),
                         pi.mean((1, 2, 3), keepdim=True), case["stencil"], case["n"] ** 3)
        s["out"] = torch.empty_like(phi), torch.empty_like(pi)
        return s
    s["sim"] = P.Simulation(_config(case["model"], case["n"], case.get("order", 2),
                                    case["precision"], case["stencil"],
                                    case.get("time", "conformal")))
    if kind == "evolve":
        s["out"] = torch.empty_like(phi), torch.empty_like(pi)
        return s
    s["sim"].set_initial(phi, pi, on_device=True)
    s["sim"].evolve(1)
    s["sim"].spectrum(0, 0)   # the plan a run makes at its first output
    s["out"] = torch.empty_like(phi[0]), torch.empty_like(phi[0])
    return s


def _summary(e, nf):
    """The energies whose value is not left over from cancelling terms: rho_grad of a field that
    sits on a background and the residual are rounding of that background."""
    return dict(a=float(e["a"]), pa=float(e["pa"]), eta=float(e["eta"]), rho=float(e["rho"]),
                P=float(e["P"]), rho_pot=float(e["rho_pot"]),
                mean=np.array([float(v) for v in list(e["mean"])[:nf]]))


def run(state):
    kind = state["kind"]
    if kind == "evolve":
        sim = state["sim"]
        sim.set_initial(state["phi"], state["pi"], on_device=True)
        sim.evolve(state["steps"])
        phi, pi = sim.get_fields(*state["out"], on_device=True)
        return dict(phi=phi, pi=pi, energies=_summary(sim.energies(), sim.nf))
    if kind == "linear":
        phi, pi = state["out"]
        a, pa, f0, p0 = P.pycool_linear_evolve(state["cfg"], 1.0, state["pa0"], state["phi"],
                                               state["pi"], state["steps"], phi, pi)
        return dict(phi=phi, pi=pi, a=float(a), pa=float(pa), phi0=f0, pi0=p0)
    if kind == "outputs":
        sim = state["sim"]
        rho, prs = sim.energy_fields(*state["out"], on_device=True)
        spectra = [sim.spectrum(which, f) for which in (0, 1) for f in range(sim.nf)]
        return dict(rho=rho, P=prs, power=[p for p, _ in spectra], count=spectra[0][1],
                    energies=_summary(sim.energies(), sim.nf))
    srv = state["server"].handle
    tickets = [P.pycool_server_submit(srv, cfg, ic, seed, steps)
               for cfg, ic, seed, steps, _ in state["jobs"]]
    out = []
    for t, job in zip(tickets, state["jobs"]):
        status, e = P.pycool_server_wait(srv, t)
        if status != P.OK:
            raise P.PycoolError(status, "pycool_server_wait")
        out.append(_summary(e.as_dict(), job[4]))
    keys = sorted(out[0])
    return {k: np.concatenate([np.atleast_1d(o[k]) for o in out]) for k in keys}


# ---------------------------------------------------------------- what a pass cannot do without

def _site_flops(model, stencil):
    nf = len(MODELS[model]["bg"])
    base = {"oscillon": 29, "expr_phi4": 26, "qball": 60}.get(model, 44)
    return base + nf * {"7pt": 0, "iso27": 30, "4th": 12}[stencil]


def work(case):
    kind = case["kind"]
    if kind == "serve":
        word = 8 if case["precision"] == "fp64" else 4
        b = f = 0.0
        for q in _requests(case):
            nf, k = len(MODELS[q["model"]]["bg"]), q["steps"] * STAGES[q["order"]]
            b += q["n"] ** 3 * nf * word * (4.0 * k + 3 + 2)
            f += q["n"] ** 3 * k * float(_site_flops(q["model"], "7pt"))
        return dict(bytes=b, flops=f)
    n, nf = case["n"], len(MODELS[case["model"]]["bg"])
    s = float(n ** 3)
    word = 4 if case.get("precision") == "split_fp32" else 8
    if kind == "evolve":   # a stage needs the lattice sums of the one before: fields in and out
        k = case["steps"] * STAGES[case["order"]]
        return dict(bytes=s * nf * (word * (4.0 * k + 3 + 4) + 32),
                    flops=s * k * _site_flops(case["model"], case["stencil"]))
    fft = 2.5 * s * math.log2(s)
    if kind == "linear":
        # distinct k_eff^2: about one mode in 48 (every sign and order of the axes)
        k = case["steps"] * STAGES[case["order"]]
        return dict(bytes=s * nf * 32.0, flops=4 * nf * fft + s / 48 * k * (2 * nf) ** 2 * 8.0)
    return dict(bytes=s * (2 * nf * word + 16) + s * nf * 2 * word,
                flops=2 * nf * fft + s * (22.0 * nf + 10))


# ---------------------------------------------------------------- the same in plain torch, 64 bits

_HALF = {6: (0.78451361047755726382, 0.23557321335935813368, -1.17767998417887100695),
         8: (0.74167036435061295345, -0.40910082580003159400, 0.19075471029623837995,
             -0.57386247111608226666, 0.29906418130365592384, 0.33462491824529818378,
             0.31529309239676659663)}


def _weights(order):
    if order == 2:
        return [1.0]
    if order == 4:
        c = 2.0 ** (1.0 / 3.0)
        return [1 / (2 - c), -c / (2 - c), 1 / (2 - c)]
    h = list(_HALF[order])
    return h + [1.0 - 2.0 * math.fsum(h)] + h[::-1]


def _potential(model, f):
    """V and dV/dphi_i (list) of the fields f (N_f, ...)."""
    p = MODELS[model]["params"]
    if model.endswith("chaotic2"):
        t = p[0] + p[1] * f[1] ** 2
        return 0.5 * f[0] ** 2 * t, [f[0] * t, p[1] * f[0] ** 2 * f[1]]
    if model == "oscillon":
        x = f[0] ** 2
        return (x * (p[0] / 2 - x * (p[1] / 4 - x * p[2] / 6)),
                [f[0] * (p[0] - x * (p[1] - x * p[2]))])
    if model == "expr_phi4":
        x = f[0] ** 2
        return x * (p[0] / 2 + x * p[1] / 4), [f[0] * (p[0] + x * p[1])]
    u = 0.5 * (f[0] ** 2 + f[1] ** 2)
    l = torch.log(u / p[2] ** 2)
    d = p[0] * (1 + p[1] + p[1] * l)
    return p[0] * u * (1 + p[1] * l), [d * f[0], d * f[1]]


def _neighbours(stencil):
    """(offset, weight) of every neighbour of the discrete Laplacian."""
    if stencil == "4th":
        axes = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
        return [(tuple(s * a for a in ax), w) for ax in axes
                for s, w in ((1, 16 / 12), (-1, 16 / 12), (2, -1 / 12), (-2, -1 / 12))]
    w = {"7pt": (0, 1.0, 0, 0), "iso27": (0, 14 / 30, 3 / 30, 1 / 30)}[stencil]
    offs = [(z, y, x) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    return [(o, w[sum(map(abs, o))]) for o in offs if any(o) and w[sum(map(abs, o))]]


def _laplacian(f, stencil):
    """Sum of weight (neighbour - centre), per field."""
    out = torch.zeros_like(f)
    for o, w in _neighbours(stencil):
        out += w * (torch.roll(f, o, (1, 2, 3)) - f)
    return out


def _root(model, n, phi, pi, stencil, sites=None, a=1.0):
    """p_a < 0 from H = 0; `sites` where one site stands for all."""
    m = MODELS[model]
    s = float(sites or n ** 3)
    grad = 0.0 if sites else float((phi * _laplacian(phi, stencil)).sum())
    each = s if sites else 1.0
    e = (each * float((pi * pi).sum()) / (2 * a * a) - 0.5 * a * a * grad / m["dx"] ** 2
         + a ** 4 * each * float(_potential(model, phi)[0].sum()))
    return -math.sqrt(12.0 * s * m["mpl"] ** 2 * e)


def _exact_evolve(model, n, order, steps, stencil, time, phi, pi):
    m = MODELS[model]
    S, dx2 = float(n ** 3), m["dx"] ** 2
    phi, pi = phi.clone(), pi.clone()
    a, eta = 1.0, 0.0
    pa = _root(model, n, phi, pi, stencil)
    c1 = 1.0 / (6.0 * S * m["mpl"] ** 2)
    for _ in range(steps):
        deta = m["dt"] / a if time == "physical" else m["dt"]
        for w in _weights(order):
            h = w * deta
            a -= 0.5 * h * c1 * pa
            kin = float((pi * pi).sum())
            pa += 0.5 * h * kin / a ** 3
            phi += (0.5 * h / a ** 2) * pi
            lap = _laplacian(phi, stencil)
            V, dV = _potential(model, phi)
            pa += h * a ** 3 * (float((phi * lap).sum()) / (a * a * dx2) - 4.0 * float(V.sum()))
            pi += (h * a * a / dx2) * lap
            for i, d in enumerate(dV):
                pi[i] -= (h * a ** 4) * d
            kin = float((pi * pi).sum())
            pa += 0.5 * h * kin / a ** 3
            phi += (0.5 * h / a ** 2) * pi
            a -= 0.5 * h * c1 * pa
            eta += h
    return phi, pi, a, pa, eta


def _exact_summary(model, n, stencil, phi, pi, a, pa, eta):
    m = MODELS[model]
    S = float(n ** 3)
    kin = float((pi * pi).sum()) / (2 * a ** 6 * S)
    grad = -float((phi * _laplacian(phi, stencil)).sum()) / (2 * a * a * m["dx"] ** 2 * S)
    pot = float(_potential(model, phi)[0].sum()) / S
    return dict(a=a, pa=pa, eta=eta, rho=kin + grad + pot, P=kin - grad / 3 - pot, rho_pot=pot,
                mean=phi.mean((1, 2, 3)).cpu().numpy())


def _exact_linear(case, seed):
    model, n, m = case["model"], case["n"], MODELS[case["model"]]
    phi, pi = _fields(model, n, seed)
    nf, p, S = phi.shape[0], m["params"], float(n ** 3)
    f0, p0 = phi.mean((1, 2, 3), keepdim=True), pi.mean((1, 2, 3), keepdim=True)
    a, pa = 1.0, _root(model, n, f0, p0, case["stencil"], n ** 3)
    F = torch.fft.rfftn(phi - f0, dim=(1, 2, 3))
    Q = torch.fft.rfftn(pi - p0, dim=(1, 2, 3))
    f0, p0 = f0.flatten().cpu(), p0.flatten().cpu()
    F[:, 0, 0, 0] = 0
    Q[:, 0, 0, 0] = 0
    t = [2 * math.pi / n * torch.arange(n, dtype=torch.float64, device="cuda").reshape(s)
         for s in ((-1, 1, 1), (1, -1, 1), (1, 1, -1))]
    t[2] = t[2][..., : n // 2 + 1]
    k2 = sum(w * (1 - torch.cos(o[0] * t[0] + o[1] * t[1] + o[2] * t[2]))
             for o, w in _neighbours(case["stencil"])) / m["dx"] ** 2
    c1 = 1.0 / (6.0 * S * m["mpl"] ** 2)
    for _ in range(case["steps"]):
        for w in _weights(case["order"]):
            h = w * m["dt"]
            for half in (0, 1):
                if half == 0:
                    a -= 0.5 * h * c1 * pa
                pa += 0.5 * h * S * float((p0 * p0).sum()) / a ** 3
                f0 = f0 + (0.5 * h / a ** 2) * p0
                F += (0.5 * h / a ** 2) * Q
                if half == 1:
                    a -= 0.5 * h * c1 * pa
                    continue
                V, dV = _potential(model, f0.reshape(nf, 1))
                x = [float(v) for v in f0]
                if model == "chaotic2":
                    M = [[p[0] + p[1] * x[1] ** 2, 2 * p[1] * x[0] * x[1]],
                         [2 * p[1] * x[0] * x[1], p[1] * x[0] ** 2]]
                elif model == "oscillon":
                    M = [[p[0] - 3 * p[1] * x[0] ** 2 + 5 * p[2] * x[0] ** 4]]
                else:
                    u = 0.5 * (x[0] ** 2 + x[1] ** 2)
                    d = p[0] * (1 + p[1] + p[1] * math.log(u / p[2] ** 2))
                    c = p[0] * p[1] / u
                    M = [[d + c * x[0] ** 2, c * x[0] * x[1]], [c * x[0] * x[1], d + c * x[1] ** 2]]
                for i in range(nf):
                    Q[i] -= (h * a * a) * k2 * F[i]
                    for j in range(nf):
                        Q[i] -= (h * a ** 4 * M[i][j]) * F[j]
                pa -= 4 * S * a ** 3 * float(V.sum()) * h
                p0 = p0 - (h * a ** 4) * torch.stack([d.sum() for d in dV])
    back = [torch.fft.irfftn(X, s=(n, n, n), dim=(1, 2, 3)) + x.cuda().reshape(-1, 1, 1, 1)
            for X, x in ((F, f0), (Q, p0))]
    return dict(phi=back[0], pi=back[1], a=a, pa=pa, phi0=f0.numpy(), pi0=p0.numpy())


def _exact_outputs(case, seed):
    model, n, stencil, m = case["model"], case["n"], case["stencil"], MODELS[case["model"]]
    phi, pi = _fields(model, n, seed)
    phi, pi, a, pa, eta = _exact_evolve(model, n, 2, 1, stencil, "conformal", phi, pi)
    grad = torch.zeros_like(phi[0])
    for o, w in _neighbours(stencil):
        grad += 0.5 * w * (torch.roll(phi, o, (1, 2, 3)) - phi).square().sum(0)
    grad /= (a * m["dx"]) ** 2
    kin = pi.square().sum(0) / (2 * a ** 6)
    V = _potential(model, phi)[0]
    k = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
    r = (k.reshape(-1, 1, 1) ** 2 + k.reshape(1, -1, 1) ** 2 + k.reshape(1, 1, -1) ** 2).sqrt()
    shell = torch.floor(r + 0.5).long().flatten()
    nb = int(math.floor(math.sqrt(3.0) * n / 2.0)) + 2
    power = []
    for x in (*phi, *pi):
        e = (torch.fft.fftn(x).abs() / float(n ** 3)).square().flatten()
        power.append(torch.bincount(shell, e, nb).cpu().numpy())
    return dict(rho=kin + 0.5 * grad + V, P=kin - grad / 6 - V, power=power, count=None,
                energies=_exact_summary(model, n, stencil, phi, pi, a, pa, eta))


def _philox_normals(seed, arr, count):
    """Normals of the serving loop's recipe: Philox4x32-10 counters (e // 4, arr, 0, 0), key the
    seed's two words, u = (x + 1/2) 2^-32, Box-Muller on the words (0, 1) and (2, 3)."""
    mask = 0xFFFFFFFF
    e = torch.arange(count, dtype=torch.int64, device="cuda")
    c = [e >> 2, torch.full_like(e, arr), torch.zeros_like(e), torch.zeros_like(e)]
    k = [seed & mask, seed >> 32]
    for r in range(10):
        if r:
            k = [(k[0] + 0x9E3779B9) & mask, (k[1] + 0xBB67AE85) & mask]
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & mask) ^ c[1] ^ k[0], p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k[1],
             p0 & mask]
    first = (e & 3) < 2
    u1 = (torch.where(first, c[0], c[2]).double() + 0.5) * 2.0 ** -32
    u2 = (torch.where(first, c[1], c[3]).double() + 0.5) * 2.0 ** -32
    t = 2 * math.pi * u2
    return torch.sqrt(-2.0 * torch.log(u1)) * torch.where((e & 1) == 1, torch.sin(t), torch.cos(t))


def _exact_serve(case, seed):
    out = []
    for i, q in enumerate(_requests(case)):
        m, n, S = MODELS[q["model"]], q["n"], q["n"] ** 3
        nf = len(m["bg"])
        z = [_philox_normals(seed * 1000 + i, j, S).reshape(n, n, n) * m["noise"]
             for j in range(2 * nf)]
        phi = torch.stack([b + x for b, x in zip(m["bg"], z[:nf])])
        pi = torch.stack([b + x for b, x in zip(m["mom"], z[nf:])])
        got = _exact_evolve(q["model"], n, q["order"], q["steps"], "7pt", "conformal", phi, pi)
        out.append(_exact_summary(q["model"], n, "7pt", *got))
    return {k: np.concatenate([np.atleast_1d(o[k]) for o in out]) for k in sorted(out[0])}


def exact(case, seed):
    if case["kind"] == "linear":
        return _exact_linear(case, seed)
    if case["kind"] == "outputs":
        return _exact_outputs(case, seed)
    if case["kind"] == "serve":
        return _exact_serve(case, seed)
    phi, pi = _fields(case["model"], case["n"], seed)
    phi, pi, a, pa, eta = _exact_evolve(case["model"], case["n"], case["order"], case["steps"],
                                        case["stencil"], case["time"], phi, pi)
    return dict(phi=phi, pi=pi,
                energies=_exact_summary(case["model"], case["n"], case["stencil"], phi, pi, a, pa,
                                        eta))
