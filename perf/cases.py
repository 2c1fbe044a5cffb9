"""The work a user of the solver has it do, as timed cases: imaginary-time steps
of one lattice (every arithmetic, 16^3 to 1024^3), lockstep batches, the
finite-difference kinetic term, energies with observables, and a small solve.

Each case drives the public entry points of paper_2006_16935_gb300.qfd.  States
of complex64 plans (and their energies) come back as complex64 (float32): what
such a plan holds.  exact() restates the method (arXiv:2006.16935, Sec. 2.1 to
2.4) in complex128 with torch's own transforms.
"""
import math

import numpy as np
import torch

from paper_2006_16935_gb300 import qfd

SIZES = (8, 16, 32, 64, 96, 128, 192, 256, 512)
PRECS = ("c128", "c64", "df64")


def listed():
    def case(name, kind, n, prec, **kw):
        d = dict(name=name, kind=kind, n=n, prec=prec, kinetic=2, steps=10, ortho=10, states=1, parity=0, potential="cornell",
                 centre="grid", start="random", count=1, energy=False, tune=False)
        d.update(kw)
        return d

    return [
        # the smallest call: the 16^3 lattice of a quick check, default arithmetic
        case("step_16_c128", "step", 16, "c128", kinetic=3, ortho=5, parity=1),
        # a short request of the serving mix: 64^3 complex64, relativistic kinetic term
        case("step_64_c64", "step", 64, "c64", kinetic=3, steps=20, parity=1),
        # a whole ground + first excited state solve at the oscillator's 32^3
        case("solve_32_c128", "solve", 32, "c128", kinetic=2, steps=200, states=2, parity=1, potential="ho"),
        # 32 lattices of 64^3 in lockstep (the batched workload)
        case("batch_64_c64", "batch", 64, "c64", count=32),
        # the radix-3 lattice of the batched workload, potential from an array
        case("step_96_df64", "step", 96, "df64", kinetic=1, steps=13, ortho=5, potential="array"),
        # the second excited state of the 256^3 Cornell workload (Gram-Schmidt against two)
        case("excited_256_c64", "step", 256, "c64", states=3, parity=1, start="settled"),
        # energy and observables of a stored 256^3 state
        case("measure_256_c128", "measure", 256, "c128", kinetic=3, steps=0, start="settled"),
        # H_K(0), the finite-difference term of the original code
        case("fdtd_256_c128", "step", 256, "c128", kinetic=0, centre="offgrid", parity=1, energy=True),
        # the benchmark's 512^3 ground-state period in each arithmetic
        case("ground_512_c64", "step", 512, "c64", parity=1, potential="softcoul", energy=True, tune=True),
        case("ground_512_df64", "step", 512, "df64", parity=1, potential="softcoul", start="settled", energy=True, tune=True),
        case("ground_512_c128", "step", 512, "c128", parity=1, potential="softcoul", energy=True, tune=True),
        # the largest lattice, started from the library's own seeded noise
        case("ground_1024_c64", "step", 1024, "c64", steps=3, ortho=3, parity=1, potential="softcoul", start="fill", tune=True),
    ]


def draw(rng):
    kind = rng.choice(("step", "step", "step", "batch", "measure", "solve"))
    d = dict(kind=kind, n=rng.choice(SIZES), prec=rng.choice(PRECS), kinetic=rng.randint(1, 3), steps=rng.randint(3, 25),
             ortho=rng.randint(2, 12), states=rng.randint(1, 3), parity=rng.choice((0, 1, -1)),
             potential=rng.choice(("cornell", "ho", "softcoul", "array")), centre=rng.choice(("grid", "offgrid")),
             start=rng.choice(("random", "settled")), count=1, energy=rng.random() < 0.3, tune=rng.random() < 0.3)
    if kind == "step" and rng.random() < 0.2:
        d.update(kinetic=0, centre="offgrid")
    if d["n"] == 512:
        d.update(steps=min(d["steps"], 7), states=1)
    if kind == "batch":
        d.update(n=rng.choice((16, 32, 64, 96, 128)), states=1, parity=0, centre="grid", energy=False, tune=False)
        d["count"] = rng.randint(2, 32 if d["n"] <= 64 else 9)
    if kind == "measure":
        d.update(steps=0, states=1)
    if kind == "solve":
        d.update(n=rng.choice((16, 32, 64)), ortho=10, steps=10 * rng.randint(6, 20), tune=False)
    return d


# ------------------------------------------------------------ shared inputs
def _spacing(case):
    return 0.05 if case["n"] >= 256 else 0.1


def _physics(case, i=0):
    """(a, mass, kinetic, dtau) of lattice i: dtau at half the stability limit."""
    a, m = _spacing(case), 1.0 + 0.37 * (i % 11)
    kin = case["kinetic"] if case["kind"] != "batch" else 1 + i % 3
    if kin == 1:
        tmax = 3.0 * math.pi ** 2 / (2.0 * a * a * m)
    elif kin == 3:
        tmax = math.sqrt(12.0 / (a * a) + m * m) - m
    else:
        tmax = 12.0 / (2.0 * a * a * m)
    return a, m, kin, 1.0 / tmax


def _axis(case):
    """Signed distance from the potential's centre along one axis, in lattice units."""
    n = case["n"]
    return torch.arange(n, dtype=torch.float64, device="cuda") - (0.5 * (n - 1) if case["centre"] == "offgrid" else n // 2)


def _r2(case):
    d = _axis(case) ** 2
    return d[:, None, None] + d[None, :, None] + d[None, None, :]


def _array_potential(case, seed):
    """A smooth anisotropic potential, as a user's own array."""
    g = torch.Generator(device="cuda").manual_seed(7000 + seed)
    c = torch.rand(3, generator=g, dtype=torch.float64, device="cuda")
    d = _axis(case) * _spacing(case)
    w = 2.0 * math.pi / (case["n"] * _spacing(case))
    f = [0.4 * (0.5 + c[k]) * d * d + 0.05 * torch.cos(3 * w * d + 6.0 * c[k]) for k in range(3)]
    return (f[0][:, None, None] + f[1][None, :, None] + f[2][None, None, :]).contiguous()


def _coeffs(case, i=0):
    return {"cornell": (0.3 + 0.01 * i, 0.2), "ho": (1.0,), "softcoul": (0.01,)}.get(case["potential"], ())


def _potential(case, seed, i=0):
    """V of lattice i in 64 bits, by the definitions of include/qfd.h."""
    if case["potential"] == "array":
        return _array_potential(case, seed)
    a = _spacing(case)
    r, c = a * torch.sqrt(_r2(case)), _coeffs(case, i)
    if case["potential"] == "ho":
        return 0.5 * c[0] * r * r
    if case["potential"] == "cornell":
        r = r.clamp(min=0.5 * a)
        return -c[0] / r + c[1] * r
    return -1.0 / torch.sqrt(r * r + c[0])


def _states(case, seed, i=0):
    """The states a program holds: seeded noise, or a settled state (a smooth
    decaying envelope with some noise left); the lower ones orthonormal."""
    g = torch.Generator(device="cuda").manual_seed(100003 * (i + 1) + seed)
    n, out = case["n"], []
    env = torch.exp(-torch.sqrt(_r2(case) + 1.0) * (6.0 / n)) if case["start"] == "settled" else None
    for s in range(case["states"]):
        p = torch.view_as_complex(torch.rand(n, n, n, 2, generator=g, dtype=torch.float64, device="cuda") * 2 - 1)
        if env is not None:
            p = env * (1.0 + 0.02 * p)
            if s == 1:
                p = p * _axis(case)[:, None, None]
            if s == 2:
                p = p * (_axis(case)[None, :, None] ** 2 - 0.02 * n * n)
        if s < case["states"] - 1 and case["kind"] != "solve":
            p = p / math.sqrt(float((p.abs() ** 2).sum()))
            for q in out:
                p = p - q * torch.vdot(q.reshape(-1), p.reshape(-1))
            p = p / math.sqrt(float((p.abs() ** 2).sum()))
        out.append(p.contiguous())
    return out


def prepare(case, seed):
    stream = torch.cuda.Stream()
    st = {"case": case, "stream": stream, "seed": seed, "plans": [], "psi": [], "out": []}
    n = case["n"]
    for i in range(case["count"]):
        a, m, kin, dt = _physics(case, i)
        p = qfd.Plan(n, a, m, dt, kin, nstates=case["states"], precision=case["prec"], ortho_every=case["ortho"],
                     check_every=case["steps"] // 2 if case["kind"] == "solve" and case["steps"] % 20 == 0 else max(1, case["steps"]),
                     centre=case["centre"], max_steps=case["steps"], tol=-1.0, stream=stream.cuda_stream)
        if case["potential"] == "array":
            V = _array_potential(case, seed)
            torch.cuda.synchronize()
            p.set_potential(V)
        else:
            p.fill_potential(case["potential"], _coeffs(case, i))
        top = case["states"] - 1
        if case["kind"] != "solve":
            p.set_parity(top, case["parity"])
        if case["tune"]:
            p.autotune()
        psi = [] if case["start"] == "fill" else _states(case, seed, i)
        torch.cuda.synchronize()
        if case["kind"] != "solve":
            for s in range(top):  # the converged lower states
                p.set_psi(s, psi[s])
            if case["kind"] == "measure":
                p.set_psi(top, psi[top])
        outs = [] if case["kind"] == "measure" else [torch.empty(n, n, n, dtype=torch.complex128, device="cuda")
                                                     for _ in range(case["states"] if case["kind"] == "solve" else 1)]
        p.sync()
        st["plans"].append(p)
        st["psi"].append(psi if case["kind"] == "solve" else psi[-1:])
        st["out"].append(outs)
    torch.cuda.synchronize()
    return st


def _parities(case):
    """Parity sector per state of a solve: the given one, alternating upwards."""
    return [case["parity"] * (-1) ** s for s in range(case["states"])]


def _held(case, x):
    """A state or a number as the plan's arithmetic holds it."""
    if case["prec"] != "c64":
        return x
    return x.to(torch.complex64) if isinstance(x, torch.Tensor) else np.float32(x)


def run(state):
    case, plans = state["case"], state["plans"]
    p = plans[0]
    with torch.cuda.stream(state["stream"]):
        if case["kind"] == "measure":
            e, n2 = p.energy(0)
            return [_held(case, v) for v in (e, n2)] + [_held(case, v) for v in p.observables(0).values()]
        if case["kind"] == "solve":
            for s, psi in enumerate(state["psi"][0]):
                p.set_psi(s, psi)
            es, _, _ = p.solve_states(case["states"], _parities(case))
            return [_held(case, v) for v in es] + [_held(case, p.get_psi(s, o)) for s, o in enumerate(state["out"][0])]
        top = case["states"] - 1
        for q, psi in zip(plans, state["psi"]):
            if case["start"] == "fill":
                q.fill_psi_uniform(top, state["seed"])
            else:
                q.set_psi(top, psi[-1])
        if case["kind"] == "batch":
            qfd.step_batch(plans, top, case["steps"])
        else:
            p.step(top, case["steps"])
        res = [_held(case, v) for v in p.energy(top)] if case["energy"] else []
        return res + [_held(case, q.get_psi(top, o[0])) for q, o in zip(plans, state["out"])]


def work(case):
    """One pass: psi in and out of the caller's buffers, and per step psi read
    and written and V read once; 5 log2 n flops a site for each of the six
    line transforms of a step (H_K(0): 16 flops a site)."""
    n3 = float(case["n"]) ** 3 * case["count"]
    site, v = (8.0, 4.0) if case["prec"] == "c64" else (16.0, 8.0)
    fft = 16.0 if case["kinetic"] == 0 else 30.0 * math.log2(case["n"])
    if case["kind"] == "measure":
        return {"bytes": n3 * (2 * site + v), "flops": n3 * (0.5 * fft + 40.0)}
    ns = case["states"] if case["kind"] == "solve" else 1
    steps = case["steps"] * ns
    return {"bytes": n3 * (32.0 * ns + steps * (2 * site + v)), "flops": n3 * steps * (fft + 8.0)}


# -------------------------------------------------- the method in 64 bits
def _reflect(case, x):
    y = torch.flip(x, (0, 1, 2))
    return y if case["centre"] == "offgrid" else torch.roll(y, (1, 1, 1), (0, 1, 2))


class _Exact:
    def __init__(self, case, seed, i=0):
        self.case = case
        self.a, self.m, self.kin, self.dt = _physics(case, i)
        self.V = _potential(case, seed, i)
        h = 0.5 * self.dt * self.V
        self.B = 1.0 / (1.0 + h)
        self.A = (1.0 - h) * self.B
        n, a, m = case["n"], self.a, self.m
        if self.kin:
            k = 2.0 * math.pi * torch.fft.fftfreq(n, dtype=torch.float64, device="cuda")
            t = k * k if self.kin == 1 else 4.0 * torch.sin(0.5 * k) ** 2
            s = t[:, None, None] + t[None, :, None] + t[None, None, :]
            self.T = torch.sqrt(s / (a * a) + m * m) - m if self.kin == 3 else s / (2.0 * a * a * m)

    def hk(self, p):
        if self.kin:
            return torch.fft.ifftn(self.T * torch.fft.fftn(p))
        f = 6.0 * p
        for ax in range(3):
            q = p.movedim(ax, 0)
            g = f.movedim(ax, 0)  # a view: updates f
            g[1:] -= q[:-1]
            g[:-1] -= q[1:]
        return f / (2.0 * self.m * self.a * self.a)

    def cadence(self, p, parity, lower):
        if parity:
            p = 0.5 * (p + parity * _reflect(self.case, p))
        c = [torch.vdot(q.reshape(-1), p.reshape(-1)) for q in lower]
        for q, x in zip(lower, c):
            p = p - x * q
        return p / torch.sqrt((p.abs() ** 2).sum())

    def steps(self, p, count, parity, lower):
        for t in range(1, count + 1):
            p = self.A * p - self.dt * self.B * self.hk(p)
            if t % self.case["ortho"] == 0:
                p = self.cadence(p, parity, lower)
        return p

    def energy(self, p):
        n2 = (p.abs() ** 2).sum()
        return float((torch.vdot(p.reshape(-1), self.hk(p).reshape(-1)).real + (self.V * p.abs() ** 2).sum()) / n2), float(n2)

    def observables(self, p, edge=0.3):
        d, n = _axis(self.case), self.case["n"]
        w, r2 = p.abs() ** 2, _r2(self.case)
        inb = (d.abs() <= (1.0 - edge) * n / 2.0).double()
        box = inb[:, None, None] * inb[None, :, None] * inb[None, None, :]
        n2, nb = w.sum(), (w * box).sum()

        def flip(x, axes):
            y = torch.flip(x, axes)
            return y if self.case["centre"] == "offgrid" else torch.roll(y, (1,) * len(axes), axes)

        r = flip(p, (0, 1, 2))
        out = [n2, nb, (torch.sqrt(r2) * w * box).sum() / nb, (r2 * w).sum() / n2]
        out += [(d.reshape([-1 if j == ax else 1 for j in range(3)]) * w).sum() / n2 for ax in range(3)]
        out += [((0.5 * (p + s * r)).abs() ** 2 * box).sum() / nb for s in (1, -1)]
        for ax in range(3):
            oth = tuple(j for j in range(3) if j != ax)
            out.append(((0.25 * (p + flip(p, oth) - flip(p, (ax,)) - r)).abs() ** 2 * box).sum() / nb)
        return [float(v) for v in out]


def exact(case, seed):
    if case["start"] == "fill":  # the library's own noise, and a lattice of 17 GB
        return None
    if case["kind"] == "measure":
        x, p = _Exact(case, seed), _states(case, seed)[0]
        obs = x.observables(p)
        # the centroid and the weights of the other sectors are differences of nearly equal sums
        return list(x.energy(p)) + obs[:4] + [None] * 8 if case["start"] == "settled" else list(x.energy(p)) + obs[:4] + [None] * 3 + obs[7:]
    if case["kind"] == "solve":
        x, done, es = _Exact(case, seed), [], []
        for s, p in enumerate(_states(case, seed)):
            par = _parities(case)[s]
            p = x.steps(x.cadence(p, par, done), case["steps"], par, done)
            p = p / torch.sqrt((p.abs() ** 2).sum())
            done.append(p)
            es.append(x.energy(p)[0])
        return es + done
    out = []
    for i in range(case["count"]):
        x, psi = _Exact(case, seed, i), _states(case, seed, i)
        p = x.steps(psi[-1], case["steps"], case["parity"], psi[:-1])
        out += (list(x.energy(p)) if case["energy"] else []) + [p]
    return out
