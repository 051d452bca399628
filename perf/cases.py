"""The framework's standing workloads, each one pass through its public entry points, with a 64-bit reference.

A case is a dict of plain values; ``kind`` names the entry point:

* ``step``: ``QGSolver.set_state``, ``step(steps)``, ``get_state`` on device tensors, as a run between two outputs;
* ``ensemble``: the same for every member of a ``QGEnsemble``;
* ``vjp``: ``QGSolver.step_vjp``, one step of a gradient sweep;
* ``series``: ``qg_series_compare`` on two device series (the a posteriori lag table);
* ``apriori``: ``qg_sgs_apriori`` on host fields (the a priori closure test).

Inputs: an eddying vorticity field (spectrum k^4 exp(-(k/kp)^2) with kp = min(n / 16, 32), scaled so that eddy and
inflow speeds are alike), the island or cape coast smoothed over two cells, the sponge ramps at the x boundaries,
beta = 5, U = 0.5 past the island and beta = 10, U = 1 past the cape.  Runs past the cape use the Smagorinsky
closures: at its corners the Leith closures' explicit flux is at its stability limit, where rounding grows from step
to step in any precision; so does the paper's explicit scheme.
"""
import math

import numpy as np
import torch

import paper_2508_06678_gb300 as qg
from paper_2508_06678_gb300._lib import qg_closure, qg_params

L = 2 * math.pi
DT = 2e-3
NU = 1.0 / 200.0
RATE = 50.0
CLOSURES = {"none": qg.QG_NONE, "smag": qg.QG_SMAG, "leith": qg.QG_LEITH, "dsmag": qg.QG_DSMAG, "dleith": qg.QG_DLEITH}
CONST = {"smag": 0.17, "leith": 0.25}
# real two-dimensional transforms of one evaluation of the explicit terms: the fields in and the products out
TRANSFORMS = {"none": 5, "smag": 9, "leith": 7, "dsmag": 18, "dleith": 14}


def listed():
    return [
        # the plain FP64 LES past an island, the smallest configuration: launches and latency count
        {"name": "step-smag-128-f64", "kind": "step", "n": 128, "prec": "f64", "closure": "smag", "coast": "island",
         "scheme": "rk3", "steps": 20},
        # a member-sized FP32 run with the dynamic Smagorinsky closure
        {"name": "step-dsmag-256-f32", "kind": "step", "n": 256, "prec": "f32", "closure": "dsmag", "coast": "cape",
         "scheme": "rk3", "steps": 20},
        # a static closure at the LES grid of the paper
        {"name": "step-leith-512-f32", "kind": "step", "n": 512, "prec": "f32", "closure": "leith", "coast": "island",
         "scheme": "rk3", "steps": 10},
        # a grid that is neither 2^p nor 3 * 2^p: users pick the resolution, the library takes any 2^a 3^b
        {"name": "step-smag-1296-f32", "kind": "step", "n": 1296, "prec": "f32", "closure": "smag", "coast": "island",
         "scheme": "rk3", "steps": 5},
        # the production step past an island, the headline workload of bench.py
        {"name": "step-dleith-2048-f32", "kind": "step", "n": 2048, "prec": "f32", "closure": "dleith",
         "coast": "island", "scheme": "rk3", "steps": 10},
        # the same workload in the paper's own time scheme
        {"name": "step-dleith-2048-ab2cn-f32", "kind": "step", "n": 2048, "prec": "f32", "closure": "dleith",
         "coast": "island", "scheme": "ab2cn", "steps": 12},
        # the largest grid: open-ocean turbulence with a static closure
        {"name": "step-leith-4096-f32", "kind": "step", "n": 4096, "prec": "f32", "closure": "leith", "coast": "none",
         "scheme": "rk3", "steps": 12},
        # a fully resolved FP64 run (no closure), the reference an LES is compared with
        {"name": "step-none-1024-f64", "kind": "step", "n": 1024, "prec": "f64", "closure": "none", "coast": "island",
         "scheme": "rk3", "steps": 4},
        # one backward step of the gradient through a dynamic Smagorinsky LES
        {"name": "vjp-dsmag-256-f64", "kind": "vjp", "n": 256, "prec": "f64", "closure": "dsmag", "coast": "cape"},
        # sixteen LES of four grids and four closures side by side
        {"name": "ensemble-16-f32", "kind": "ensemble", "members": 16, "n": 256, "prec": "f32", "steps": 10},
        # lag table of two 96-snapshot series on the paper's LES grid
        {"name": "series-512-f32", "kind": "series", "n": 512, "prec": "f32", "snaps": 96, "lag": 32},
        # a priori test of a closure: a 1024^2 field filtered to 256^2
        {"name": "apriori-dsmag-1024-f64", "kind": "apriori", "n": 1024, "nles": 256, "closure": "dsmag",
         "coast": "island"},
    ]


def _grids(lo, hi):
    return sorted(2 ** a * 3 ** b for a in range(1, 13) for b in range(0, 8) if lo <= 2 ** a * 3 ** b <= hi)


def _regular(n):
    m = n // 3 if n % 3 == 0 else n
    return m & (m - 1) == 0


def _pick(rng, lo, hi):
    """A valid grid size, spread over the logarithm of the range; half of them 2^p or 3 * 2^p."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    grids = _grids(lo, hi)
    if rng.random() < 0.5:
        grids = [n for n in grids if _regular(n)]
    return min(grids, key=lambda n: abs(math.log(n / want)))


def _coast_for(closure, scheme, coast):
    return "island" if coast == "cape" and (closure.endswith("leith") or scheme == "ab2cn") else coast


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["vjp", "ensemble", "series", "apriori"])
    closure = rng.choice(sorted(CLOSURES))
    coast = rng.choice(["island", "cape", "none"])
    if kind == "step":
        prec = rng.choice(["f32", "f32", "f64"])
        scheme = rng.choice(["rk3", "rk3", "ab2cn"])
        case = {"kind": kind, "n": _pick(rng, 64, 1024 if prec == "f64" else 4096), "prec": prec, "closure": closure,
                "coast": _coast_for(closure, scheme, coast), "scheme": scheme, "steps": 1}
        # at most the operations of the listed cases of that kind of grid, and of that precision
        most = 4.5e9 if prec == "f64" else 2.5e11 if _regular(case["n"]) else 5.5e10
        return {**case, "steps": max(1, min(rng.randint(4, 12), int(most / _step_work(case)["flops"])))}
    if kind == "vjp":
        return {"kind": kind, "n": _pick(rng, 64, 512), "prec": rng.choice(["f32", "f64"]), "closure": closure,
                "coast": _coast_for(closure, "rk3", coast)}
    if kind == "ensemble":
        return {"kind": kind, "members": rng.randint(2, 16), "n": rng.choice([64, 96, 128, 192, 256, 384]),
                "prec": "f32", "steps": rng.randint(4, 10)}
    if kind == "series":
        return {"kind": kind, "n": _pick(rng, 64, 512), "prec": rng.choice(["f32", "f64"]),
                "snaps": rng.randint(8, 96 if rng.random() < 0.5 else 48), "lag": rng.randint(2, 24)}
    n = _pick(rng, 256, 1536)
    return {"kind": kind, "n": n, "nles": max(m for m in _grids(32, n // 2) if m <= n / rng.choice([2, 3, 4])),
            "closure": rng.choice(["smag", "leith", "dsmag", "dleith"]), "coast": coast}


# ---- inputs


def _dtype(case):
    return torch.float32 if case.get("prec", "f64") == "f32" else torch.float64


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _field(n, gen, speed):
    """A random vorticity field in the 2/3 band, zero mean, eddies of about ``speed`` (FP64, on the GPU)."""
    spec = torch.fft.rfft2(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=gen))
    o = _Ops(n)
    kp = min(n / 16.0, 32.0)
    m2 = o.mx ** 2 + o.my ** 2
    w = torch.fft.irfft2(spec * o.T * m2 * torch.exp(-0.5 * m2 / kp ** 2), s=(n, n))
    return w * (0.5 * kp * speed / w.square().mean().sqrt())


def _coast(n, kind):
    """chi_obs (None without a coast), smoothed over two cells, and chi_sponge."""
    d = L / n
    x = torch.arange(n, dtype=torch.float64, device="cuda") * d
    y = x[:, None]
    x = x[None, :]
    sponge = torch.clamp(1.0 - torch.minimum(x, L - x) / (0.1 * L), min=0.0).expand(n, n).contiguous()
    if kind == "none":
        return None, sponge
    if kind == "island":
        s = torch.sqrt((x - math.pi / 2) ** 2 + (y - math.pi) ** 2) - 0.4
    else:  # a coastal strip y < 0.3 L and a cape of half the box's width that reaches to 0.45 L
        top = torch.where((x - L / 2).abs() <= 0.25 * L, 0.45 * L, 0.3 * L)
        s = torch.minimum(y - top, L - y)
        s = torch.where(y >= top, s, torch.maximum(y - top, -y))
    return 0.5 * (1.0 - torch.tanh(s / (2.0 * d))), sponge


def _host(a):
    return None if a is None else a.cpu().numpy()


def _physics(coast):
    return {"beta": 10.0, "U": 1.0} if coast == "cape" else {"beta": 5.0, "U": 0.5}


def _flow(case, gen):
    return _field(case["n"], gen, _physics(case["coast"])["U"])


def _spec(case, coast):
    """QGSolver's keyword arguments."""
    ab2 = case.get("scheme") == "ab2cn"
    return dict(n=case["n"], L=L, precision=qg.QG_FP32 if case["prec"] == "f32" else qg.QG_FP64, mask=_host(coast[0]),
                sponge=_host(coast[1]), kind=CLOSURES[case["closure"]], c=CONST.get(case["closure"], 0.0), dt=DT, nu=NU,
                eta=1.025 * DT if ab2 else 1e-3, sponge_rate=RATE,
                scheme=qg.QG_SCHEME_AB2CN if ab2 else qg.QG_SCHEME_RK3_EXACT, **_physics(case["coast"]))


def _members(case):
    """The members of an ensemble: four sizes from n to 3 n, the four closures, island and cape."""
    n = case["n"]
    sizes = [n, n * 3 // 2, n * 2, n * 3]
    kinds = ["smag", "leith", "dsmag", "dleith"]
    return [{"n": sizes[i % 4], "prec": case["prec"], "closure": kinds[(i // 4) % 4],
             "coast": _coast_for(kinds[(i // 4) % 4], "rk3", ["island", "cape"][(i // 2) % 2]), "scheme": "rk3",
             "steps": case["steps"]} for i in range(case["members"])]


def _series(case, seed):
    """Two series of a translating pattern, the second two snapshots ahead, each with its own noise."""
    n, snaps = case["n"], case["snaps"]
    gen = _gen(seed)
    base = _field(n, gen, 0.1)
    out = []
    for ahead in (0, 2):
        s = torch.stack([torch.roll(base, shifts=((t + ahead) // 2, t + ahead), dims=(0, 1)) for t in range(snaps)])
        out.append((s + 0.2 * torch.randn(s.shape, dtype=torch.float64, device="cuda", generator=gen)).to(_dtype(case)))
    return out


def prepare(case, seed):
    kind = case["kind"]
    gen = _gen(seed)
    if kind == "series":
        les, ff = _series(case, seed)
        return {"case": case, "les": les, "ff": ff}
    if kind == "apriori":
        coast = _coast(case["n"], case["coast"])
        return {"case": case, "w": _host(_flow(case, gen)), "mask": _host(coast[0]), "sponge": _host(coast[1])}
    if kind == "ensemble":
        members = _members(case)
        coasts = {(m["n"], m["coast"]): _coast(m["n"], m["coast"]) for m in members}
        ens = qg.QGEnsemble([_spec(m, coasts[m["n"], m["coast"]]) for m in members])
        w = [_flow(m, gen).to(_dtype(case)) for m in members]
        return {"case": case, "solver": ens, "w": w, "out": [torch.empty_like(x) for x in w]}
    stream = torch.cuda.Stream()  # a stream of its own: steps are replayed as graphs there
    solver = qg.QGSolver(stream=stream, **_spec(case, _coast(case["n"], case["coast"])))
    w = _flow(case, gen).to(_dtype(case))
    state = {"case": case, "solver": solver, "stream": stream, "w": w, "out": torch.empty_like(w)}
    if kind == "vjp":
        state["lam"] = _field(case["n"], gen, 0.1).to(_dtype(case))
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        s = state["solver"]
        s.set_state(state["w"])
        s.step(case["steps"])
        return s.get_state(out=state["out"])
    if kind == "ensemble":
        ens = state["solver"]
        for s, w in zip(ens.members, state["w"]):
            s.set_state(w)
        ens.step(case["steps"])
        return [s.get_state(out=o) for s, o in zip(ens.members, state["out"])]
    if kind == "vjp":
        lam, grads = state["solver"].step_vjp(state["w"], state["lam"], state["out"])
        return {"lam": lam, **{k: np.array([v]) for k, v in grads.items()}}
    if kind == "series":
        return qg.qg_series_compare(state["les"], state["ff"], -case["lag"], case["lag"],
                                    stream=torch.cuda.current_stream())
    closure = qg_closure(CLOSURES[case["closure"]], 0, CONST.get(case["closure"], 0.0), 2.0)
    params = qg_params(DT, NU, 0.0, 1e-3, RATE, 0, 0)
    pi, model, parts, pcc = qg.qg_sgs_apriori(state["w"], case["nles"], L, state["mask"], state["sponge"], closure,
                                              params, **_physics(case["coast"]))
    return {"pi": pi, "model": model, "parts": parts, "pcc": np.array([pcc])}


def _step_work(case):
    n, b = case["n"], 4 if case["prec"] == "f32" else 8
    per = TRANSFORMS[case["closure"]] * (1 if case["scheme"] == "ab2cn" else 3)
    per += (4 if case["coast"] != "none" else 0) + 2
    # transforms at 2.5 n^2 log2(n^2) each; bytes: the field in and out, chi_obs and chi_sponge
    return {"bytes": float(n * n * b * (4 if case["coast"] != "none" else 3)),
            "flops": 2.5 * n * n * math.log2(n * n) * per * case["steps"]}


def work(case):
    kind = case["kind"]
    if kind == "step":
        return _step_work(case)
    if kind == "ensemble":
        w = [_step_work(m) for m in _members(case)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    n = case["n"]
    if kind == "vjp":  # the step and, for each of its transforms and products, the transposed one
        w = _step_work({**case, "scheme": "rk3", "steps": 1})
        b = 4 if case["prec"] == "f32" else 8
        return {"bytes": w["bytes"] + n * n * b, "flops": 3 * w["flops"]}
    if kind == "series":
        pairs = sum(1 for t in range(case["snaps"]) for p in range(-case["lag"], case["lag"] + 1)
                    if 0 <= t - p < case["snaps"])
        b = 4 if case["prec"] == "f32" else 8
        return {"bytes": float(2 * case["snaps"] * n * n * b + 16 * case["snaps"] * (2 * case["lag"] + 1)),
                "flops": float(5 * pairs * n * n)}
    fine, coarse = 5 + (4 if case["coast"] != "none" else 0) + 3, 10 + TRANSFORMS[case["closure"]]
    m = case["nles"]
    return {"bytes": float(8 * (n * n * (3 if case["coast"] != "none" else 2) + 5 * m * m)),
            "flops": 2.5 * (n * n * math.log2(n * n) * fine + m * m * math.log2(m * m) * coarse)}


# ---- the same results in plain 64-bit torch


class _Ops:
    """Wavenumbers of an n x n grid (rfft2 layout) and the 2/3 rule."""

    def __init__(self, n):
        self.n = n
        self.mx = torch.arange(n // 2 + 1, dtype=torch.float64, device="cuda")[None, :]
        self.my = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")[:, None]
        self.kx, self.ky = self.mx * (2 * math.pi / L), self.my * (2 * math.pi / L)
        self.k2 = self.kx ** 2 + self.ky ** 2
        self.ik2 = torch.where(self.k2 > 0, 1.0 / self.k2.clamp(min=1e-30), torch.zeros_like(self.k2))
        K = (n - 1) // 3
        self.T = ((self.mx <= K) & (self.my.abs() <= K)).to(torch.float64)
        self.G = ((self.mx ** 2 + self.my ** 2) * 16.0 <= float(n) ** 2).to(torch.float64)  # test filter, ratio 2
        self.delta = L / n

    def fwd(self, f):
        return torch.fft.rfft2(f)

    def inv(self, f):
        return torch.fft.irfft2(f, s=(self.n, self.n))

    def project(self, w):
        wh = self.T * self.fwd(w)
        keep = torch.ones_like(self.T)
        keep[0, 0] = 0.0
        return wh * keep


def _velocity(o, wh, U):
    psi = -wh * o.ik2
    return o.inv(-1j * o.ky * psi) + U, o.inv(1j * o.kx * psi)


def _jacobian(o, wh, U):
    u, v = _velocity(o, wh, U)
    return o.T * o.fwd(u * o.inv(1j * o.kx * wh) + v * o.inv(1j * o.ky * wh))


def _flux_divergence(o, wh, closure):
    """T F[div(g grad w)], g = |S| or |grad w|."""
    wx, wy = o.inv(1j * o.kx * wh), o.inv(1j * o.ky * wh)
    if closure.endswith("smag"):
        psi = -wh * o.ik2
        pxy, pd = o.inv(-(o.kx * o.ky) * psi), o.inv(-(o.kx ** 2 - o.ky ** 2) * psi)
        g = torch.sqrt(4.0 * pxy ** 2 + pd ** 2)
    else:
        g = torch.sqrt(wx ** 2 + wy ** 2)
    return o.T * (1j * o.kx * o.fwd(g * wx) + 1j * o.ky * o.fwd(g * wy))


def _coefficient(o, wh, closure, U, J, D):
    p = 2 if closure.endswith("smag") else 3
    if closure in CONST:
        return torch.tensor((CONST[closure] * o.delta) ** p, dtype=torch.float64, device="cuda")
    wt = o.G * wh
    H = o.inv(_jacobian(o, wt, U) - o.G * J)
    M = o.inv(2.0 ** p * _flux_divergence(o, wt, closure) - o.G * D)
    return torch.clamp((H * M).mean() / (M * M).mean(), min=0.0)


def _explicit(o, wh, closure, U, extra=None):
    """-J + C div(g grad w); ``extra`` is added to the coefficient."""
    J = _jacobian(o, wh, U)
    if closure == "none":
        return -J
    D = _flux_divergence(o, wh, closure)
    C = _coefficient(o, wh, closure, U, J, D)
    return (C if extra is None else C + extra) * D - J


def _curl(o, u, v):
    return o.T * (1j * o.kx * o.fwd(v) - 1j * o.ky * o.fwd(u))


def _rk3(o, w0, case, coast, beta, U, extra=None, rate=RATE):
    ws = w0
    for a, b in ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)):
        rhs = _explicit(o, ws, case["closure"], U, extra) + beta * 1j * o.kx * (ws * o.ik2)
        ws = a * w0 + b * (ws + DT * rhs)
    ws = torch.exp(-NU * o.k2 * DT) * ws
    if coast[0] is not None:
        f = torch.exp(-coast[0] * DT / 1e-3)
        u, v = _velocity(o, ws, U)
        ws = _curl(o, f * u, f * v)
    return o.project(torch.exp(-rate * coast[1] * DT) * o.inv(ws))


def _ab2cn(o, wh, case, coast, beta, U, steps):
    lin = -NU * o.k2 + 1j * beta * o.kx * o.ik2
    prev = star_prev = None
    for _ in range(steps):
        E = _explicit(o, wh, case["closure"], U)
        if coast[0] is not None:
            u, v = _velocity(o, wh, U)
            E = E - _curl(o, coast[0] * u, coast[0] * v) / (1.025 * DT)
        prev = E if prev is None else prev
        star = ((1.0 + 0.5 * DT * lin) * wh + DT * (1.5 * E - 0.5 * prev)) / (1.0 - 0.5 * DT * lin)
        star_prev = star if star_prev is None else star_prev
        damp = o.fwd(DT * RATE * coast[1] * o.inv(1.5 * star - 0.5 * star_prev))
        wh = o.project(o.inv(star - o.T * damp))
        prev, star_prev = E, star
    return wh


def _exact_step(case, w):
    o = _Ops(case["n"])
    coast = _coast(case["n"], case["coast"])
    p = _physics(case["coast"])
    wh = o.project(w.to(torch.float64))
    if case["scheme"] == "ab2cn":
        return o.inv(_ab2cn(o, wh, case, coast, p["beta"], p["U"], case["steps"]))
    for _ in range(case["steps"]):
        wh = _rk3(o, wh, case, coast, p["beta"], p["U"])
    return o.inv(wh)


def _exact_vjp(case, w, lam):
    o = _Ops(case["n"])
    coast = _coast(case["n"], case["coast"])
    p = _physics(case["coast"])
    w = w.to(torch.float64).requires_grad_(True)
    extra = torch.zeros((), dtype=torch.float64, device="cuda", requires_grad=True)
    rate = torch.tensor(RATE, dtype=torch.float64, device="cuda", requires_grad=True)
    out = o.inv(_rk3(o, o.project(w), case, coast, p["beta"], p["U"], extra, rate))
    wrt = [w, rate] + ([extra] if case["closure"] != "none" else [])
    g = torch.autograd.grad((out * lam.to(torch.float64)).sum(), wrt)
    dC = float(g[2]) if case["closure"] != "none" else 0.0
    q = 2 if case["closure"].endswith("smag") else 3
    c = CONST.get(case["closure"])
    dc = dC * q * c ** (q - 1) * o.delta ** q if c else 0.0
    return {"lam": g[0], "C": np.array([dC]), "c": np.array([dc]), "sponge_rate": np.array([float(g[1])])}


def _exact_series(case, les, ff):
    snaps, lag = case["snaps"], case["lag"]
    a, b = (x.to(torch.float64).reshape(snaps, -1) for x in (les, ff))
    ca, cb = a - a.mean(1, keepdim=True), b - b.mean(1, keepdim=True)
    na, nb = ca.norm(dim=1), cb.norm(dim=1)
    dist = torch.full((snaps, 2 * lag + 1), math.nan, dtype=torch.float64, device="cuda")
    pcc = dist.clone()
    for j, phi in enumerate(range(-lag, lag + 1)):
        t0, t1 = max(0, phi), min(snaps, snaps + phi)
        if t0 < t1:
            dist[t0:t1, j] = (a[t0 - phi:t1 - phi] - b[t0:t1]).square().sum(1)
            pcc[t0:t1, j] = (ca[t0 - phi:t1 - phi] * cb[t0:t1]).sum(1) / (na[t0 - phi:t1 - phi] * nb[t0:t1])
    mean = dist.nanmean(0)
    best = min((float(m), abs(j - lag), j - lag) for j, m in enumerate(mean.tolist()) if not math.isnan(m))
    return {"dist": dist, "pcc": pcc, "mean_dist": mean, "phase": best[2]}


def _exact_apriori(case, w, coast):
    n, m = case["n"], case["nles"]
    U, closure = _physics(case["coast"])["U"], case["closure"]
    of, oc = _Ops(n), _Ops(m)

    def filt(fh, band=True):
        """Gaussian times the sharp cut-off, the kept modes copied to the coarse grid without its Nyquist lines."""
        m2 = of.mx ** 2 + of.my ** 2
        fh = fh * torch.exp(-of.k2 * oc.delta ** 2 / 6.0) * (4.0 * m2 <= float(m) ** 2)
        out = torch.zeros(m, m // 2 + 1, dtype=torch.complex128, device="cuda")
        h = m // 2
        out[:h, :h] = fh[:h, :h]
        out[m - h + 1:, :h] = fh[n - h + 1:, :h]
        return out * (m / n) ** 2 * (oc.T if band else 1.0)

    wh = of.project(w)
    wb = filt(wh)
    parts = [oc.inv(_jacobian(oc, wb, U) - filt(_jacobian(of, wh, U)))]
    if coast[0] is None:
        parts.append(torch.zeros_like(parts[0]))
    else:
        u, v = _velocity(of, wh, U)
        ub, vb = _velocity(oc, wb, U)
        chi = oc.inv(filt(of.fwd(coast[0]), band=False))
        parts.append(oc.inv(_curl(oc, chi * ub, chi * vb) - filt(_curl(of, coast[0] * u, coast[0] * v))) / 1e-3)
    chi = oc.inv(filt(of.fwd(coast[1]), band=False))
    parts.append(RATE * oc.inv(oc.T * oc.fwd(chi * oc.inv(wb)) - filt(of.T * of.fwd(coast[1] * of.inv(wh)))))
    pi = parts[0] + parts[1] + parts[2]
    D = _flux_divergence(oc, wb, closure)
    model = oc.inv(_coefficient(oc, wb, closure, U, _jacobian(oc, wb, U), D) * D)
    x, y = pi - pi.mean(), model - model.mean()
    pcc = float((x * y).mean() / ((x * x).mean().sqrt() * (y * y).mean().sqrt()))
    return {"pi": pi, "model": model, "parts": torch.stack(parts), "pcc": np.array([pcc])}


def exact(case, seed):
    kind = case["kind"]
    gen = _gen(seed)
    if kind == "series":
        return _exact_series(case, *_series(case, seed))
    if kind == "apriori":
        return _exact_apriori(case, _flow(case, gen), _coast(case["n"], case["coast"]))
    if kind == "ensemble":
        return [_exact_step(m, _flow(m, gen).to(_dtype(case))) for m in _members(case)]
    w = _flow(case, gen).to(_dtype(case))
    if kind == "vjp":
        return _exact_vjp(case, w, _field(case["n"], gen, 0.1).to(_dtype(case)))
    return _exact_step(case, w)
