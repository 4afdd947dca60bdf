"""The work that users of this library have it do, as cases that can be timed
and checked one by one: whole passes through the public entry points, from a
few hundred short orbits to a million, in both precisions.

A case is a dict of plain values.  ``prepare`` makes a program's inputs and
the context it keeps, ``run`` is one pass, ``exact`` the same result in plain
64-bit torch (its own Philox, Box-Muller, step schemes and adjoint).
"""
import math

import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300.autograd import integrate_final, order_parameter
from paper_1908_03869_gb300.integrator import BatchIntegrator, Integrator
from paper_1908_03869_gb300.swarm import SwarmSearch

TWO_PI = 2.0 * math.pi
DTYPES = {"fp32": torch.float32, "fp64": torch.float64}


def _forward(name, model, n, orbits, dt, steps, stride, precision, read, scheme="em"):
    case = dict(kind="forward", model=model, n=n, orbits=orbits, dt=dt, steps=steps, stride=stride,
                precision=precision, read=read, scheme=scheme)
    return dict(case, name=name) if name else case


def _adjoint(name, n, orbits, dt, steps, precision):
    case = dict(kind="adjoint", n=n, orbits=orbits, dt=dt, steps=steps, ckpt_every=100, precision=precision)
    return dict(case, name=name) if name else case


def _batch(name, instances, orbits, n_low, n_high, k_low, k_high, horizon, precision):
    case = dict(kind="batch", instances=instances, orbits=orbits, n_low=n_low, n_high=n_high, k_low=k_low,
                k_high=k_high, horizon=horizon, precision=precision)
    return dict(case, name=name) if name else case


def _swarm(name, particles, realisations, n, dt, steps, precision):
    case = dict(kind="swarm", particles=particles, realisations=realisations, n=n, dt=dt, steps=steps,
                precision=precision)
    return dict(case, name=name) if name else case


def listed():
    return [
        # a first try or a unit test: so few and so short that launches and copies count
        _forward("small_fp32_n8", "kuramoto", 8, 256, 0.01, 200, 20, "fp32", "frames"),
        # the plain workload: 1024 orbits of four phases in double, read every ten steps
        _forward("plain_fp64_n4", "kuramoto", 4, 1024, 0.01, 1000, 10, "fp64", "frames"),
        # the three ensembles of the throughput workload (a shorter horizon): one lane, some
        # lanes and half a warp per orbit; the middle one is read as ensemble statistics
        _forward("ensemble_fp32_n8", "kuramoto", 8, 1 << 20, 0.005, 1000, 100, "fp32", "frames"),
        _forward("ensemble_fp32_n32_moments", "kuramoto", 32, 1 << 18, 0.005, 1000, 50, "fp32", "moments"),
        _forward("ensemble_fp32_n128", "kuramoto", 128, 1 << 16, 0.005, 1000, 100, "fp32", "frames"),
        # the same in double, where the arithmetic is the scarce thing
        _forward("ensemble_fp64_n32", "kuramoto", 32, 1 << 16, 0.005, 200, 50, "fp64", "frames"),
        # the published speed protocol: 15 oscillators (an odd size), noise of its own for each, 163840 orbits
        _forward("paper_speed_fp64_n15", "kuramoto_paper", 15, 163840, 0.05, 200, 100, "fp64", "frames"),
        # the published accuracy protocol: 64 realisations of 100 oscillators, read as the order
        # parameter's statistics; far too few orbits to fill the GPU
        _forward("paper_accuracy_fp64_n100", "kuramoto_paper", 100, 64, 0.2, 1000, 50, "fp64", "moments"),
        # multiplicative noise and two components per unit: the FitzHugh-Nagumo network
        _forward("fhn_fp32_64units", "fhn_net", 128, 1 << 17, 0.01, 400, 100, "fp32", "frames"),
        # a training step: the loss over all orbits and its gradients (over a horizon at which single
        # precision still resolves the gradient of every orbit)
        _adjoint("adjoint_fp32_n32", 32, 16384, 0.002, 1000, "fp32"),
        # a sweep over models of many sizes and step counts, 64 realisations each, in one launch
        _batch("batch_fp32", 48, 64, 2, 256, 1000, 100000, 5.0, "fp32"),
        # a generation of the parameter search: 256 particles of 64 realisations
        _swarm("swarm_fp32_n32", 256, 64, 32, 0.005, 1000, "fp32"),
    ]


def _log_int(rng, low, high):
    return int(min(high, max(low, round(math.exp(rng.uniform(math.log(low), math.log(high)))))))


def draw(rng):
    kind = rng.choice(["kuramoto", "kuramoto", "kuramoto", "paper", "fhn", "ode", "adjoint", "batch", "swarm"])
    precision = rng.choice(["fp32", "fp64"])
    most = (1 << 32) if precision == "fp32" else (1 << 28)  # unit-steps
    if kind in ("kuramoto", "paper", "ode"):
        n = _log_int(rng, 2, 256)
        orbits = max(1, _log_int(rng, 1 << 11, 1 << 23) // n)
        most //= 1 if kind != "ode" else 8
        steps = max(20, min(_log_int(rng, 100, 2000), most // (n * orbits)))
        dt = 5.0 / steps if steps > 500 else 0.01
        stride = rng.choice([10, 25, 50, 100]) if n * orbits < (1 << 20) else 50
        return _forward("", "kuramoto_paper" if kind == "paper" else "kuramoto", n, orbits, dt, steps, stride, precision,
                        rng.choice(["frames", "moments"]),
                        rng.choice(["rk4", "euler", "midpoint"]) if kind == "ode" else "em")
    if kind == "fhn":
        units = _log_int(rng, 2, 128)
        orbits = max(1, _log_int(rng, 1 << 12, 1 << 22) // units)
        steps = max(20, min(_log_int(rng, 100, 1000), most // (units * orbits)))
        return _forward("", "fhn_net", 2 * units, orbits, 0.01, steps, 50, precision, "frames",
                        rng.choice(["em", "milstein"]))
    if kind == "adjoint":
        n = _log_int(rng, 3, 128)
        orbits = max(1, _log_int(rng, 1 << 13, 1 << 19) // n)
        steps = rng.randint(150, 1000) if precision == "fp32" else rng.randint(50, 200)
        return _adjoint("", n, orbits, 2.0 / steps, steps, precision)
    if kind == "batch":
        return _batch("", rng.randint(8, 48), _log_int(rng, 1, 64), 2, 256, 200,
                      _log_int(rng, 1000, 50000) if precision == "fp32" else 1000, 5.0, precision)
    return _swarm("", _log_int(rng, 16, 256), rng.randint(8, 64), _log_int(rng, 4, 100), 0.005,
                  rng.randint(100, 800) if precision == "fp32" else rng.randint(50, 100), precision)


# ---- inputs ------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, shape, low, high, dtype=torch.float64):
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype) * (high - low) + low


def _inputs(model, n, orbits, seed, dtype, shared=False):
    """(params, x0) of the library's configured distributions, in the context's type."""
    g = _generator(seed)
    rows = 1 if shared else orbits
    u = lambda cols, low, high, r=rows: _uniform(g, (r, cols), low, high)  # noqa: E731
    if model == "kuramoto":
        omega = torch.randn((rows, n), generator=g, device="cuda", dtype=torch.float64)
        p = torch.cat([u(1, 0.0, 4.0), u(1, 0.1, 0.5), omega], 1)
        x0 = u(n, 0.0, TWO_PI, orbits)
    elif model == "kuramoto_paper":
        p = torch.cat([u(1, 0.2, 1.0), u(n, 0.01, 0.4), u(n, 0.001, 0.03)], 1)
        x0 = u(n, -math.pi, math.pi, orbits)
    else:
        p = torch.cat([u(1, 0.6, 0.8), u(1, 0.7, 0.9), u(1, 0.05, 0.1), u(1, 0.3, 0.6), u(1, 0.0, 0.5),
                       u(1, 0.01, 0.1)], 1)
        x0 = torch.cat([u(n // 2, -2.0, 2.0, orbits), u(n // 2, -0.5, 1.5, orbits)], 1)
    return (p[0] if shared else p).to(dtype).contiguous(), x0.to(dtype).contiguous()


def _batch_sizes(case):
    """[(n, steps, dt)] of a batch's instances: sizes spread evenly, step counts over their logarithm, one horizon."""
    got = []
    for i in range(case["instances"]):
        a, b = (i + 0.5) / case["instances"], math.fmod((i + 1) * 0.6180339887498949, 1.0)
        n = case["n_low"] + int(a * (case["n_high"] - case["n_low"] + 1))
        steps = int(round(case["k_low"] * (case["k_high"] / case["k_low"]) ** b))
        got.append((n, steps, case["horizon"] / steps))
    return got


def _swarm_start(case, seed):
    g = _generator(seed + 1)
    box = torch.tensor([4.0, 0.5], device="cuda", dtype=torch.float64)
    x = _uniform(g, (case["particles"], 2), 0.0, 1.0) * box
    v = _uniform(g, (case["particles"], 2), -0.1, 0.1) * box
    return x, v


def _swarm_inputs(case, seed):
    p, x0 = _inputs("kuramoto", case["n"], case["realisations"], seed, DTYPES[case["precision"]])
    return p[0].contiguous(), x0


# ---- a program's passes --------------------------------------------------------

def prepare(case, seed):
    dtype = DTYPES[case["precision"]]
    if case["kind"] == "forward":
        params, x0 = _inputs(case["model"], case["n"], case["orbits"], seed, dtype)
        scheme = case["scheme"]
        pb = sdeb.Problem.make(case["model"], case["n"], case["orbits"], case["dt"], case["steps"], case["stride"],
                               seed, case["precision"], milstein=scheme == "milstein", rk4=scheme == "rk4",
                               implicit=scheme if scheme in ("euler", "midpoint") else None)
        return dict(case=case, it=Integrator(pb), params=params, x0=x0)
    if case["kind"] == "adjoint":
        params, x0 = _inputs("kuramoto", case["n"], case["orbits"], seed, dtype, shared=True)
        pb = sdeb.Problem.make("kuramoto", case["n"], case["orbits"], case["dt"], case["steps"], case["steps"], seed,
                               case["precision"], ckpt_every=case["ckpt_every"], shared_params=True, no_frames=True)
        return dict(case=case, it=Integrator(pb), params=params.requires_grad_(), x0=x0.requires_grad_())
    if case["kind"] == "batch":
        sizes = _batch_sizes(case)
        pbs = [sdeb.Problem.make("kuramoto", n, case["orbits"], dt, steps, max(1, steps // 20), seed,
                                 case["precision"]) for n, steps, dt in sizes]
        inputs = [_inputs("kuramoto", n, case["orbits"], seed + i, dtype) for i, (n, _, _) in enumerate(sizes)]
        return dict(case=case, it=BatchIntegrator(pbs), params=[p for p, _ in inputs], x0=[x for _, x in inputs])
    base, x0 = _swarm_inputs(case, seed)
    pb = sdeb.Problem.make("kuramoto", case["n"], case["realisations"], case["dt"], case["steps"], case["steps"], seed,
                           case["precision"])
    search = SwarmSearch(pb, base, x0, [0, 1], [0.0, 0.0], [4.0, 0.5], case["particles"], r_target=0.8,
                         swarm_seed=seed)
    x, v = _swarm_start(case, seed)
    return dict(case=case, search=search, x=x, v=v)


def run(state):
    case = state["case"]
    if case["kind"] == "forward":
        it = state["it"]
        it.set_params(state["params"], state["x0"])
        it.integrate()
        if case["read"] == "frames":
            return {"frames": it.frames()}
        mom, rmom = it.moments(state=True, order_param=True)
        # 64-bit accumulators over frames of the context's type: no better than those
        return {"final": it.final(), "moments": mom.to(it.dtype), "order": rmom.to(it.dtype)}
    if case["kind"] == "adjoint":
        theta = integrate_final(state["it"], state["params"], state["x0"])
        loss = order_parameter(theta).mean()
        dp, dx0 = torch.autograd.grad(loss, (state["params"], state["x0"]))
        return {"final": theta, "loss": loss, "d_params": dp, "d_x0": dx0}
    if case["kind"] == "batch":
        it = state["it"]
        it.set_params(state["params"], state["x0"])
        it.integrate()
        return {"final": [it.final(i) for i in range(case["instances"])]}
    s = state["search"]
    s.reset(state["x"], state["v"])
    s.step()
    return {"final": s.final, "x": s.x, "v": s.v, "best": s.pbest, "best_at": s.gbest,
            "best_fitness": s.pbest_fit.to(s.final.dtype)}


def _unit_steps(case):
    """(orbits, states of all orbits, unit-steps) of a case."""
    if case["kind"] == "batch":
        sizes = _batch_sizes(case)
        orbits = case["orbits"] * len(sizes)
        return orbits, case["orbits"] * sum(n for n, _, _ in sizes), case["orbits"] * sum(n * k for n, k, _ in sizes)
    orbits = case["particles"] * case["realisations"] if case["kind"] == "swarm" else case["orbits"]
    states = orbits * case["n"]
    return orbits, states, states * case["steps"] // (2 if case.get("model") == "fhn_net" else 1)


def work(case):
    """Floating-point operations (a sine, a logarithm, a root or a division is one) and bytes in and out."""
    orbits, states, unit_steps = _unit_steps(case)
    elem = 8 if case["precision"] == "fp64" else 4
    noise = 6.0  # a pair of normals: two uniforms, logarithm, root, sine, cosine, scalings
    phase_drift = 9.0  # sine, cosine, two sums, two products and sums, frequency
    per_unit = phase_drift + noise + 3.0
    state, params = states * elem, (states + 2 * orbits) * elem
    out = state
    if case["kind"] == "forward":
        frames = case["steps"] // case["stride"] + 1
        scheme = case["scheme"]
        if case["model"] == "fhn_net":
            per_unit = 22.0 + noise + (4.0 if scheme == "milstein" else 0.0)
            params = orbits * 6 * elem
        elif case["model"] == "kuramoto_paper":
            params = (2 * states + orbits) * elem
        if scheme == "rk4":
            per_unit = 4 * (phase_drift + 4.0)
        elif scheme in ("euler", "midpoint"):
            per_unit = 4 * (phase_drift + 20.0)
        out = frames * state
        if case["read"] == "moments":
            out = state + frames * (case["n"] + 1) * 2 * elem
            per_unit += 16.0 / case["stride"]
    elif case["kind"] == "adjoint":
        params = (case["n"] + 2) * elem
        per_unit += 16.0  # the reverse sweep: two sums, the transposed drift, the parameter gradients
        out = 2 * state + params
    elif case["kind"] == "swarm":
        params = params + case["realisations"] * case["n"] * elem - state  # the realisations' states are shared
    return {"bytes": float(params + state + out), "flops": float(unit_steps * per_unit)}


# ---- the same results in 64 bits -------------------------------------------------

MASK = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    k0, k1 = seed & MASK, (seed >> 32) & MASK
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & MASK) ^ c1 ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c3 ^ k1, p0 & MASK
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return c0, c1, c2, c3


def _normals(k, orbit_ids, m, seed):
    """[..., m] normals of step k for the orbits in orbit_ids [...]."""
    blocks = torch.arange((m + 3) // 4, device="cuda")
    o = orbit_ids.unsqueeze(-1)
    zero = torch.zeros_like(o + blocks)
    w = _philox(zero + k, zero + blocks, zero + o, zero, int(seed))
    u = [(t.double() + 0.5) * 2.0 ** -32 for t in w]
    z = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = torch.sqrt(-2.0 * torch.log(a))
        z += [r * torch.cos(TWO_PI * b), r * torch.sin(TWO_PI * b)]
    return torch.stack(z, -1).reshape(*orbit_ids.shape, -1)[..., :m]


class _Phases:
    """Kuramoto drift, diffusion and Newton solve over the last axis; live: 0 for padding."""

    def __init__(self, K, g, omega, live=None):
        self.live = torch.ones_like(omega) if live is None else live
        self.K, self.g, self.omega, self.n = K, g, omega, self.live.sum(-1, keepdim=True)

    def sums(self, x):
        s, c = torch.sin(x), torch.cos(x)
        return s, c, (s * self.live).sum(-1, keepdim=True), (c * self.live).sum(-1, keepdim=True)

    def drift(self, x):
        s, c, S, C = self.sums(x)
        return self.omega + self.K / self.n * (S * c - C * s)

    def diffusion(self, x):
        return self.g

    def newton(self, z, r, h):
        """(I - h J(z))^-1 r: a diagonal plus [c s] [c s]^T."""
        s, c, S, C = self.sums(z)
        b = h * self.K / self.n
        d = 1.0 / (1.0 + b * (C * c + S * s))
        w = d * r
        total = lambda t: t.sum(-1, keepdim=True)  # noqa: E731
        e11, e12, e22 = 1.0 - b * total(c * c * d), -b * total(c * s * d), 1.0 - b * total(s * s * d)
        q1, q2 = total(c * w), total(s * w)
        det = e11 * e22 - e12 * e12
        return w + b * d * (c * (e22 * q1 - e12 * q2) + s * (e11 * q2 - e12 * q1)) / det


class _Fhn:
    def __init__(self, p):
        self.a, self.b, self.eps, self.I, self.c, self.sigma = (p[:, i:i + 1] for i in range(6))

    def drift(self, x):
        v, w = x.chunk(2, -1)
        fv = v - v ** 3 / 3.0 - w + self.I + self.c * (v.mean(-1, keepdim=True) - v)
        return torch.cat([fv, self.eps * (v + self.a - self.b * w)], -1)


def _step(model, x, k, dt, ids, m, seed, scheme):
    if scheme == "rk4":
        k1 = model.drift(x)
        k2 = model.drift(x + 0.5 * dt * k1)
        k3 = model.drift(x + 0.5 * dt * k2)
        return x + dt / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + model.drift(x + dt * k3))
    if scheme in ("euler", "midpoint"):
        theta, d = (1.0 if scheme == "euler" else 0.5), torch.zeros_like(x)
        for _ in range(4):
            z = x + theta * d
            d = d + model.newton(z, dt * model.drift(z) - d, theta * dt)
        return x + d
    dw = _normals(k, ids, m, seed) * dt ** 0.5
    if isinstance(model, _Fhn):
        v = x[:, :m]
        noise = model.sigma * v * dw
        if scheme == "milstein":
            noise = noise + 0.5 * model.sigma ** 2 * v * (dw * dw - dt)
        return x + dt * model.drift(x) + torch.cat([noise, torch.zeros_like(noise)], -1)
    return x + dt * model.drift(x) + model.diffusion(x) * dw


def _model(name, p, n):
    if name == "kuramoto":
        return _Phases(p[..., :1], p[..., 1:2], p[..., 2:])
    if name == "kuramoto_paper":
        return _Phases(p[..., :1], p[..., 1 + n:], p[..., 1:1 + n])
    return _Fhn(p)


def _order(x):
    return torch.sqrt(torch.cos(x).mean(-1) ** 2 + torch.sin(x).mean(-1) ** 2)


def _exact_forward(case, seed):
    n, orbits, steps, stride = case["n"], case["orbits"], case["steps"], case["stride"]
    p, x = (t.double() for t in _inputs(case["model"], n, orbits, seed, DTYPES[case["precision"]]))
    model, m = _model(case["model"], p, n), n // 2 if case["model"] == "fhn_net" else n
    ids = torch.arange(orbits, device="cuda")
    frames, mom, order = [], [], []

    def keep():
        if case["read"] == "frames":
            frames.append(x)
        else:
            r = _order(x)
            mom.append(torch.stack([x.mean(0), x.var(0, unbiased=False)], -1))
            order.append(torch.stack([r.mean(), r.var(unbiased=False)]))

    keep()
    for k in range(steps):
        x = _step(model, x, k, case["dt"], ids, m, seed, case["scheme"])
        if (k + 1) % stride == 0:
            keep()
    if case["read"] == "frames":
        return {"frames": torch.stack(frames)}
    return {"final": x, "moments": torch.stack(mom), "order": torch.stack(order)}


def _exact_adjoint(case, seed):
    n, orbits, dt = case["n"], case["orbits"], case["dt"]
    p, x = (t.double() for t in _inputs("kuramoto", n, orbits, seed, DTYPES[case["precision"]], shared=True))
    ids = torch.arange(orbits, device="cuda")
    xs = []
    model = _model("kuramoto", p, n)
    for k in range(case["steps"]):
        xs.append(x)
        x = _step(model, x, k, dt, ids, n, seed, "em")
    c, s = torch.cos(x), torch.sin(x)
    C, S = c.mean(-1, keepdim=True), s.mean(-1, keepdim=True)
    r = torch.sqrt(C * C + S * S)
    lam = (S * c - C * s) / (n * r) / orbits
    gK, gs, gw = torch.zeros((), device="cuda", dtype=torch.float64), 0.0, torch.zeros_like(p[2:])
    for k in range(case["steps"] - 1, -1, -1):
        c, s = torch.cos(xs[k]), torch.sin(xs[k])
        C, S = c.sum(-1, keepdim=True), s.sum(-1, keepdim=True)
        gK = gK + dt / n * (lam * (S * c - C * s)).sum()
        gs = gs + math.sqrt(dt) * (lam * _normals(k, ids, n, seed)).sum()
        gw = gw + dt * lam.sum(0)
        A, B = (lam * c).sum(-1, keepdim=True), (lam * s).sum(-1, keepdim=True)
        lam = lam + p[0] * dt / n * (c * A + s * B - lam * (c * C + s * S))
    return {"final": x, "loss": r.mean(), "d_params": torch.cat([gK.reshape(1), gs.reshape(1), gw]), "d_x0": lam}


def _exact_batch(case, seed, most_steps=4000):
    """The instances of few steps, side by side; nothing for the others."""
    sizes = _batch_sizes(case)
    some = [i for i, (_, steps, _) in enumerate(sizes) if steps <= most_steps]
    final = [None] * len(sizes)
    if not some:
        return None
    top, orbits = max(sizes[i][0] for i in some), case["orbits"]
    pad = lambda t: torch.nn.functional.pad(t.double(), (0, top - t.shape[-1]))  # noqa: E731
    inputs = [_inputs("kuramoto", sizes[i][0], orbits, seed + i, DTYPES[case["precision"]]) for i in some]
    x = torch.stack([pad(x0) for _, x0 in inputs])
    live = torch.stack([pad(torch.ones_like(x0)) for _, x0 in inputs])
    model = _Phases(torch.stack([p[:, :1].double() for p, _ in inputs]),
                    torch.stack([p[:, 1:2].double() for p, _ in inputs]), torch.stack([pad(p[:, 2:]) for p, _ in inputs]),
                    live)
    dt = torch.tensor([sizes[i][2] for i in some], device="cuda", dtype=torch.float64).reshape(-1, 1, 1)
    ends = [sizes[i][1] for i in some]
    ids = torch.arange(orbits, device="cuda").expand(len(some), orbits)
    for k in range(max(ends)):
        x = x + dt * model.drift(x) + model.g * _normals(k, ids, top, seed) * torch.sqrt(dt)
        for j, i in enumerate(some):
            if ends[j] == k + 1:
                final[i] = x[j, :, :sizes[i][0]].clone()
    return {"final": final}


def _exact_swarm(case, seed):
    P, R, n = case["particles"], case["realisations"], case["n"]
    dtype = DTYPES[case["precision"]]
    base, x0 = _swarm_inputs(case, seed)
    x, v = _swarm_start(case, seed)
    p = base.repeat(P, 1)
    p[:, :2] = x.to(dtype)
    p = p.double().repeat_interleave(R, 0)
    theta, ids = x0.double().repeat(P, 1), torch.arange(P * R, device="cuda")
    model = _model("kuramoto", p, n)
    for k in range(case["steps"]):
        theta = _step(model, theta, k, case["dt"], ids, n, seed, "em")
    fit = (_order(theta).reshape(P, R).mean(-1) - 0.8) ** 2
    b = torch.argmin(fit)
    i, j = torch.arange(P, device="cuda").unsqueeze(1), torch.arange(2, device="cuda").unsqueeze(0)
    zero = torch.zeros_like(i + j)
    w = _philox(zero, zero + j, zero + i, zero + 2, int(seed))
    u2 = (w[1].double() + 0.5) * 2.0 ** -32
    lim = torch.tensor([4.0, 0.5], device="cuda", dtype=torch.float64)
    vn = 0.7298 * v + 1.49618 * u2 * (x[b] - x)  # a first generation: every particle is at its own best
    vn = torch.minimum(torch.maximum(vn, -lim), lim)
    xn = torch.minimum(torch.clamp(x + vn, min=0.0), lim)
    return {"final": theta, "x": xn, "v": vn, "best": x, "best_at": None, "best_fitness": fit}


def exact(case, seed):
    with torch.no_grad():
        kind = case["kind"]
        if kind == "forward":
            return _exact_forward(case, seed)
        if kind == "adjoint":
            return _exact_adjoint(case, seed)
        return _exact_batch(case, seed) if kind == "batch" else _exact_swarm(case, seed)
