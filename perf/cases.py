"""Performance cases: what a user of the FDM library has it do, through its public entry points.

A case is one whole pass: the initial field goes from (pinned) host memory to the device, the
library does its work, the results come back to (pinned) host memory.  Kinds of pass:

* ``run``      a simulation: set U13, take `steps` time steps in one call, read fields;
* ``monitor``  the same with one call per step, reading the step's scalars each time;
* ``batch``    many uneven instances stepped together, each with its own step budget;
* ``readout``  a Nye field in (curl inverse), the static problem, all six fields out;
* ``hetero``   the heterogeneous static problem, a fixed number of iterations.

FP64 and double-word results are taken as float64, the mixed path's as float32: its transforms
and transport compute in 32 bits and its stated accuracy is theirs (1e-5).
"""
import math

import numpy as np
import torch

from paper_1911_03225_gb300 import FDM, Batch, Params
from paper_1911_03225_gb300 import binding as B

PRECISION = {"fp64": B.FP64, "mixed": B.MIXED, "df64": B.DF64}


def listed():
    return [
        # one small interactive study: the script reads time, dt and the Burgers vector after every step
        dict(name="monitor_64_fp64", kind="monitor", field="random", n1=64, n2=64, precision="fp64", steps=20,
             theta=1.0, cfl=0.4, stress=True),
        # annihilation of two walls at the benchmark's own size: launches and small-grid latency
        dict(name="annihilation_128_fp64", kind="run", field="walls", n1=128, n2=128, precision="fp64", steps=200,
             theta=1.0, cfl=0.5, stress=False),
        # impenetrable precipitates in a rectangular cell with lattice friction
        dict(name="orowan_512x256_fp64", kind="run", field="random", n1=512, n2=256, precision="fp64", steps=60,
             theta=1.0, cfl=0.4, stress=True, mobility=True, friction=True),
        # expanding loop, both precisions the benchmark names: with the MC limiter in FP64, with minmod in the long
        # mixed run (the MC limiter amplifies 32-bit rounding without bound there: 60 steps would compare noise)
        dict(name="ring_1024_fp64", kind="run", field="ring", n1=1024, n2=1024, precision="fp64", steps=10,
             theta=2.0, cfl=0.4, stress=False),
        dict(name="ring_1024_mixed", kind="run", field="ring", n1=1024, n2=1024, precision="mixed", steps=60,
             theta=1.0, cfl=0.4, stress=False),
        # the headline workload: coupled random field under a strain ramp, in every precision
        dict(name="coupled_2048_fp64", kind="run", field="random", n1=2048, n2=2048, precision="fp64", steps=30,
             theta=1.0, cfl=0.4, stress=True),
        dict(name="coupled_2048_df64", kind="run", field="random", n1=2048, n2=2048, precision="df64", steps=40,
             theta=1.0, cfl=0.4, stress=True),
        dict(name="coupled_2048_mixed", kind="run", field="random", n1=2048, n2=2048, precision="mixed", steps=150,
             theta=1.0, cfl=0.4, stress=True),
        # the largest grid the library takes
        dict(name="coupled_4096_mixed", kind="run", field="random", n1=4096, n2=4096, precision="mixed", steps=80,
             theta=1.0, cfl=0.4, stress=True),
        # batched parameter study: sides 64 to 512 mixed, uneven run lengths
        dict(name="batch_64_mixed", kind="batch", field="random", count=64, lo=64, hi=512, precision="mixed",
             steps=150, theta=1.0, cfl=0.4, stress=True),
        # start from a measured density, look at every field
        dict(name="readout_1024_fp64", kind="readout", field="random", n1=1024, n2=1024, precision="fp64", steps=0,
             theta=1.0, cfl=0.4, stress=True),
        # static problem in a medium of varying shear modulus
        dict(name="hetero_1024_fp64", kind="hetero", field="random", n1=1024, n2=1024, precision="fp64", steps=25,
             theta=1.0, cfl=0.4, stress=True),
    ]


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "monitor", "batch", "readout", "hetero"])
    precision = rng.choice(["fp64", "df64", "mixed"])
    n1, n2 = _pow2(rng, 64, 2048), _pow2(rng, 64, 2048)
    c = dict(kind=kind, field="random", n1=n1, n2=n2, precision=precision, steps=rng.randint(20, 80), theta=1.0,
             cfl=rng.choice([0.25, 0.4, 0.5]), stress=True)
    if kind == "monitor":
        c.update(n1=_pow2(rng, 64, 512), n2=_pow2(rng, 64, 512), steps=rng.randint(10, 40))
    elif kind == "batch":
        del c["n1"], c["n2"]
        c.update(precision="mixed", count=rng.randint(8, 64), lo=64, hi=rng.choice([128, 256, 512]))
    elif kind in ("readout", "hetero"):
        if kind == "hetero":
            c.update(steps=rng.randint(8, 30))
        c.update(precision="fp64")
    elif rng.random() < 0.3:   # a loop or walls at a prescribed celerity
        c.update(field=rng.choice(["ring", "walls"]), stress=False)
        if c["field"] == "ring":
            c.update(n1=max(n1, 256), n2=max(n2, 256))
        if rng.random() < 0.5:   # the MC limiter amplifies rounding in long runs: short ones, in FP64
            c.update(theta=2.0, precision="fp64", steps=rng.randint(6, 10))
    elif rng.random() < 0.3 and precision == "fp64":
        c.update(mobility=True, friction=rng.random() < 0.5)
    return c


# ------------------------------------------------------------------ inputs (from the seed alone)
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _grid(n1, n2, dev="cuda"):
    x = torch.arange(n1, dtype=torch.float64, device=dev)
    y = torch.arange(n2, dtype=torch.float64, device=dev)
    return x[None, :], y[:, None]


def _freq(n1, n2, dev="cuda"):
    k1 = torch.fft.fftfreq(n1, dtype=torch.float64, device=dev) * 2 * math.pi
    k2 = torch.fft.fftfreq(n2, dtype=torch.float64, device=dev) * 2 * math.pi
    return k1[None, :], k2[:, None]


def _smooth(n1, n2, g, ell):
    k1, k2 = _freq(n1, n2)
    z = torch.randn((n2, n1), generator=g, device="cuda", dtype=torch.float64)
    zh = torch.fft.fft2(z) * torch.exp(-(k1 ** 2 + k2 ** 2) * ell ** 2 / 4)
    zh[0, 0] = 0
    return torch.fft.ifft2(zh).real


def _field(case, n1, n2, seed):
    """U13 of the case, float64 on the device."""
    g = _gen(seed)
    if case["field"] == "random":   # smoothed Gaussian random field, RMS |grad U13| = 0.1
        u = _smooth(n1, n2, g, min(16.0, min(n1, n2) / 8.0))
        d1, d2 = torch.roll(u, -1, 1) - u, torch.roll(u, -1, 0) - u
        return u * (0.1 / torch.sqrt((d1 ** 2 + d2 ** 2).mean()))
    x, y = _grid(n1, n2)
    a, b = (torch.rand(2, generator=g, device="cuda", dtype=torch.float64) - 0.5).tolist()
    if case["field"] == "walls":    # two edge walls of opposite sign with Gaussian sections
        s, sep = 3.0 * (1 + 0.2 * a), n1 / 4.0 * (1 + 0.1 * b)
        c1, c2 = n1 / 2 - sep / 2, n1 / 2 + sep / 2
        f = s * math.sqrt(math.pi / 2) * (torch.erf((x - c1) / (s * math.sqrt(2))) - torch.erf((x - c2) / (s * math.sqrt(2))))
        return f.expand(n2, n1).contiguous()
    r0 = 0.1 * min(n1, n2) * (1 + 0.1 * a)   # a circular loop
    r = torch.hypot(x - n1 / 2 - b, y - n2 / 2 - a)
    return 2.0 * math.sqrt(math.pi / 2) * torch.erfc((r - r0) / (2.0 * math.sqrt(2)))


def _nye(u):
    """alpha11 = -dU/dx2 and alpha12 = dU/dx1 by spectral differentiation (odd symbols zero at Nyquist)."""
    n2, n1 = u.shape
    k1, k2 = (k.clone() for k in _freq(n1, n2, u.device))
    k1[0, n1 // 2] = 0
    k2[n2 // 2, 0] = 0
    uh = torch.fft.fft2(u)
    return torch.fft.ifft2(-1j * k2 * uh).real, torch.fft.ifft2(1j * k1 * uh).real


def _pinned(t):
    h = torch.empty(t.shape, dtype=torch.float64, pin_memory=True)
    h.copy_(t)
    return h.numpy()


def _out(n1, n2):
    return torch.empty((n2, n1), dtype=torch.float64, pin_memory=True).numpy()


def _mobility(n1, n2, seed):
    """Mobility factor: impenetrable discs (0) in a matrix with softer zones."""
    g = _gen(seed + 100003)
    m = torch.where(_smooth(n1, n2, g, 8.0) > 0, 1.0, 0.5).to(torch.float64)
    x, y = _grid(n1, n2)
    for cx, cy in torch.rand((6, 2), generator=g, device="cuda", dtype=torch.float64).tolist():
        m[torch.hypot(x - cx * n1, y - cy * n2) < 0.04 * min(n1, n2)] = 0.0
    return m


def _modulus(n1, n2, seed):
    f = _smooth(n1, n2, _gen(seed + 200003), 24.0)
    return 0.25 + 0.75 * (f - f.min()) / (f.max() - f.min())


def _params(case, n1, n2):
    p = Params(n1=n1, n2=n2, theta=case["theta"], cfl=case["cfl"], precision=PRECISION[case["precision"]])
    if case["stress"]:
        p.velocity_mode, p.loading_mode, p.eps_bar13_rate = B.V_STRESS, B.LOAD_STRAIN_RAMP, 1e-4
    else:
        p.v0 = -1.0 if case["field"] == "ring" else 1.0
    if case.get("friction"):
        p.tau_y, p.beta = 0.02, 0.5
    if case["kind"] == "hetero":
        p.nz = p.nh = 64
        p.loading_mode, p.sigma_bar13 = B.LOAD_STRESS, 0.01
    return p


def _members(case, seed):
    """Sides and step budgets of a batch: the mix is the case's own, the fields the seed's."""
    r = np.random.RandomState(case["count"])
    sides = [s for s in (64, 128, 256, 512) if case["lo"] <= s <= case["hi"]]
    return [(int(r.choice(sides)), int(r.randint(case["steps"] // 2, case["steps"] + 1))) for _ in range(case["count"])]


# ------------------------------------------------------------------ the pass
def prepare(case, seed):
    if case["kind"] == "batch":
        members = _members(case, seed)
        b = Batch([_params(case, n, n) for n, _ in members])
        return dict(case=case, batch=b, budgets=[k for _, k in members],
                    u=[_pinned(_field(case, n, n, seed * 1000 + i)) for i, (n, _) in enumerate(members)])
    n1, n2 = case["n1"], case["n2"]
    sim = FDM(_params(case, n1, n2))
    u = _field(case, n1, n2, seed)
    s = dict(case=case, sim=sim)
    names = ["up13", "tau13"]
    if case["kind"] == "readout":
        a11, a12 = _nye(u)
        s.update(a11=_pinned(a11), a12=_pinned(a12))
        names = ["up13", "alpha11", "alpha12", "tau13", "v1", "v2"]
    else:
        s["u"] = _pinned(u)
    if case.get("mobility"):
        sim.set_mobility_field(_mobility(n1, n2, seed).cpu().numpy())
    if case["kind"] == "hetero":
        s["mu"] = _pinned(_modulus(n1, n2, seed))
        sim.set_plastic_distortion(s["u"])
    s["out"] = {nm: _out(n1, n2) for nm in names}
    return s


def _typed(case, fields):
    if case["precision"] == "mixed":
        return {k: torch.from_numpy(v).to(torch.float32) for k, v in fields.items()}
    return fields


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        for i, u in enumerate(state["u"]):
            b.set_plastic_distortion(i, u)
            b.set_budget(i, state["budgets"][i])
        b.enqueue_steps(max(state["budgets"]))
        b.sync()
        return torch.cat([torch.from_numpy(b.read_fields(i, "up13")["up13"]).to(torch.float32).reshape(-1)
                          for i in range(b.count)])
    sim, out = state["sim"], state["out"]
    if case["kind"] == "hetero":
        s13, s23, _, _ = sim.static_solve_heterogeneous(state["mu"], tol=0.0, max_iter=case["steps"])
        return {"sigma13": s13, "sigma23": s23}
    if case["kind"] == "readout":
        sim.set_density(state["a11"], state["a12"], 0.0)
        sim.static_solve()
        return sim.read_fields(*out, out=out)
    sim.set_plastic_distortion(state["u"])
    if case["kind"] == "monitor":
        log = []
        for _ in range(case["steps"]):
            i = sim.step(1)
            log.append((i.t, i.dt, i.max_abs_v0, i.sigma_bar13, i.sum_abs_alpha))
        return _typed(case, dict(sim.read_fields(*out, out=out), log=np.array(log)))
    sim.step(case["steps"])
    return _typed(case, sim.read_fields(*out, out=out))


def work(case):
    """Each step reads and writes the state once and writes the stress; each iteration of the heterogeneous problem
    reads and writes its two-component iterate and reads the modulus; host fields cross once."""
    e = {"fp64": 8, "df64": 8, "mixed": 4}[case["precision"]]
    state = 8 if case["precision"] == "mixed" else e   # the mixed path keeps U13 as a pair of words
    if case["kind"] == "batch":
        cells = [(n * n, k, math.log2(n)) for n, k in _members(case, 0)]
        return {"bytes": float(sum(c * (k * (2 * state + e) + 16) for c, k, _ in cells)),
                "flops": float(sum(c * k * (250 + 10 * lg) for c, k, lg in cells))}
    cells, lg = case["n1"] * case["n2"], math.log2(case["n1"] * case["n2"])
    if case["kind"] == "hetero":
        return {"bytes": float(cells * (case["steps"] * 5 * e + 24)), "flops": float(cells * case["steps"] * (20 + 10 * lg))}
    if case["kind"] == "readout":
        return {"bytes": float(cells * 8 * 8), "flops": float(cells * (40 + 2.5 * 7 * lg))}
    return {"bytes": float(cells * (case["steps"] * (2 * state + e) + 24)),
            "flops": float(cells * case["steps"] * (250 + 5 * lg))}


# ------------------------------------------------------------------ the same in 64 bits, plain torch
def _kernel(p):
    """Layer Green kernel on the full grid: (1/(nz nh)) sum_k3 m(xi) |chi-hat(k3)|^2 (even in every index)."""
    nz = p.nz or p.n1
    x1 = torch.arange(p.n1 // 2 + 1, dtype=torch.float64, device="cuda")[None, :] / p.n1
    x2 = torch.arange(p.n2 // 2 + 1, dtype=torch.float64, device="cuda")[:, None] / p.n2
    mu = p.E / (2 * (1 + p.nu))
    s1, s2 = x1 * x1, x2 * x2
    s12 = s1 + s2
    acc = torch.zeros_like(s12)
    for k3 in range(nz // 2 + 1):
        if k3 == 0:
            w = float(p.nh) ** 2
        else:
            w = (math.sin(math.pi * k3 * p.nh / nz) / math.sin(math.pi * k3 / nz)) ** 2
        if k3 != 0 and 2 * k3 != nz:
            w *= 2
        x3 = (k3 / nz) ** 2
        q = s12 + x3
        if k3 == 0:
            q[0, 0] = 1.0
        m = -mu * (s2 / q + 2 * s1 * x3 / (q * q) / (1 - p.nu))
        if k3 == 0:
            m[0, 0] = 0.0
        acc += w * m
    acc /= nz * p.nh
    full = torch.cat([acc, acc[1:p.n2 // 2].flip(0)], 0)
    return full   # kx in [0, n1/2], every ky: for rfft2


def _loading(p, step, t, mean):
    mu, frac = p.E / (2 * (1 + p.nu)), p.nh / (p.nz or p.n1)
    if p.loading_mode == B.LOAD_STRESS:
        return torch.full_like(mean, p.sigma_bar13)
    return 2 * mu * (p.eps_bar13_0 + p.eps_bar13_rate * step) - mu * frac * mean


def _tau(p, K, u, step):
    uh = torch.fft.rfft2(u) * K
    n = u.shape[-1] * u.shape[-2]
    uh[..., 0, 0] = _loading(p, step, 0.0, u.mean((-1, -2))) * n
    return torch.fft.irfft2(uh, s=u.shape[-2:])


def _minmod3(a, b, c):
    lo, hi = torch.minimum(torch.minimum(a, b), c), torch.maximum(torch.maximum(a, b), c)
    return torch.where(lo > 0, lo, torch.where(hi < 0, hi, torch.zeros_like(a)))


def _knp(u, v0, r, th):
    """One Kurganov-Noelle-Petrova update in cell units (r = dt / h), midpoint time level."""
    def f(i, j):
        return torch.roll(u, (-j, -i), (-2, -1))

    def sides(m2, m1, p1, p2):
        a, b, c, d = m1 - m2, u - m1, p1 - u, p2 - p1
        mid = th * (c - b)
        return (c, _minmod3(th * (d - c), 0.5 * (d - b), mid)), (b, _minmod3(mid, 0.5 * (c - a), th * (b - a)))

    xs = sides(f(-2, 0), f(-1, 0), f(1, 0), f(2, 0))
    ys = sides(f(0, -2), f(0, -1), f(0, 1), f(0, 2))
    px = (xs[0][0] - 0.5 * xs[0][1], xs[1][0] + 0.5 * xs[1][1])
    qy = (ys[0][0] - 0.5 * ys[0][1], ys[1][0] + 0.5 * ys[1][1])
    z = torch.zeros_like(u)
    ap, am, bp, bm = z, z, z, z
    for p in px:
        for q in qy:
            r2 = p * p + q * q
            iv = torch.where(r2 > 0, v0 * torch.rsqrt(torch.where(r2 > 0, r2, torch.ones_like(r2))), z)
            ap, am = torch.maximum(ap, iv * p), torch.minimum(am, iv * p)
            bp, bm = torch.maximum(bp, iv * q), torch.minimum(bm, iv * q)

    def weights(a, b):
        w = a - b
        ok = w > 0
        s = torch.where(ok, w, torch.ones_like(w))
        h = torch.full_like(w, 0.5)
        return torch.where(ok, -b / s, h), torch.where(ok, a / s, h)

    wx, wy = weights(ap, am), weights(bp, bm)
    inc = z
    for s, (cx, a, (Dx, Sx)) in enumerate(((1, ap, xs[0]), (-1, am, xs[1]))):
        for t, (cy, b, (Dy, Sy)) in enumerate(((1, bp, ys[0]), (-1, bm, ys[1]))):
            ex, ey = a * r, b * r
            cross = (f(cx, cy) - f(0, cy) - f(cx, 0) + u) * (cx * cy)
            val = ex * (Dx + 0.5 * Sx * (ex - cx)) + ey * (Dy + 0.5 * Sy * (ey - cy)) + cross * ex * ey
            p = Dx + Sx * (ex - 0.5 * cx) + cross * ey
            q = Dy + Sy * (ey - 0.5 * cy) + cross * ex
            r2 = p * p + q * q
            w = torch.where(r2 > 0, 0.5 * v0 * r * torch.rsqrt(torch.where(r2 > 0, r2, torch.ones_like(r2))), z)
            p, q = p - w * (Sx * p + cross * q), q - w * (cross * p + Sy * q)
            inc = inc + wx[s] * wy[t] * (val - v0 * r * torch.sqrt(p * p + q * q))
    return u + inc


def _simulate(p, u, budgets, mfac=None):
    """`budgets` steps of each field of the stack u; (U13, tau13 of the last step, log per step)."""
    K = _kernel(p)
    left = torch.tensor(budgets, device="cuda")
    tau, log, t = torch.zeros_like(u), [], torch.zeros(u.shape[0], dtype=torch.float64, device="cuda")
    mu, frac = p.E / (2 * (1 + p.nu)), p.nh / (p.nz or p.n1)
    for k in range(max(budgets)):
        tn = _tau(p, K, u, k)
        if p.velocity_mode == B.V_STRESS:
            fr = p.tau_y * torch.cos(u / p.beta) if p.tau_y else 0.0
            v0 = p.mobility * (fr - tn)
        else:
            v0 = torch.full_like(u, p.v0)
        if mfac is not None:
            v0 = v0 * mfac
        vm = v0.abs().amax((-1, -2))
        dt = p.cfl * p.dx / vm
        go = (left > k)[:, None, None]
        u = torch.where(go, _knp(u, v0, (dt / p.dx)[:, None, None], p.theta), u)
        tau = torch.where(go, tn, tau)
        t = t + dt
        if u.shape[0] == 1 and u[0].numel() <= 1 << 18:
            d1, d2 = torch.roll(u, -1, 2) - u, torch.roll(u, -1, 1) - u
            sig = _loading(p, k + 1, 0.0, u.mean((-1, -2)))
            log.append((float(t), float(dt), float(vm), float(sig), float(torch.hypot(d1, d2).sum()) / p.dx))
    return u, tau, np.array(log)


def exact(case, seed):
    if case["kind"] == "batch":
        members = _members(case, seed)
        got = [None] * len(members)
        for n in sorted({n for n, _ in members}):
            at = [i for i, (m, _) in enumerate(members) if m == n]
            u = torch.stack([_field(case, n, n, seed * 1000 + i) for i in at])
            u, _, _ = _simulate(_params(case, n, n), u, [members[i][1] for i in at])
            for j, i in enumerate(at):
                got[i] = u[j].reshape(-1)
        return torch.cat(got)
    n1, n2 = case["n1"], case["n2"]
    p, u = _params(case, n1, n2), _field(case, n1, n2, seed)
    if case["kind"] == "hetero":
        mu = p.E / (2 * (1 + p.nu)) * _modulus(n1, n2, seed)
        mu0 = 0.5 * (mu.min() + mu.max())
        k1, k2 = _freq(n1, n2)
        o1, o2 = k1.clone(), k2.clone()
        o1[0, n1 // 2] = 0
        o2[n2 // 2, 0] = 0
        q = k1 ** 2 + k2 ** 2
        q[0, 0] = 1.0
        g1 = g2 = torch.zeros_like(u)
        for _ in range(case["steps"]):
            a = torch.fft.fft2((mu - mu0) * g1 - mu * u)
            b = torch.fft.fft2((mu - mu0) * g2)
            ga, gb = -(k1 ** 2 * a + o1 * o2 * b) / q / mu0, -(o1 * o2 * a + k2 ** 2 * b) / q / mu0
            ga[0, 0] = (p.sigma_bar13 * n1 * n2 - a[0, 0]) / mu0
            gb[0, 0] = -b[0, 0] / mu0
            g1, g2 = torch.fft.ifft2(ga).real, torch.fft.ifft2(gb).real
        return {"sigma13": mu * (g1 - u), "sigma23": mu * g2}
    if case["kind"] == "readout":
        a11, a12 = _nye(u)
        k1, k2 = _freq(n1, n2)
        o1, o2 = k1.clone(), k2.clone()
        o1[0, n1 // 2] = 0
        o2[n2 // 2, 0] = 0
        q = k1 ** 2 + k2 ** 2
        q[0, 0] = 1.0
        uh = 1j * (torch.fft.fft2(a11) * o2 - torch.fft.fft2(a12) * o1) / q
        uh[0, 0] = 0
        u = torch.fft.ifft2(uh).real
        a11, a12 = _nye(u)
        tau = _tau(p, _kernel(p), u, 0)
        v, m = -p.mobility * tau, torch.hypot(a11, a12)
        return {"up13": u, "alpha11": a11, "alpha12": a12, "tau13": tau, "v1": v * a12 / m, "v2": -v * a11 / m}
    mfac = _mobility(n1, n2, seed) if case.get("mobility") else None
    u, tau, log = _simulate(p, u[None], [case["steps"]], mfac)
    out = {"up13": u[0], "tau13": tau[0]}
    if case["kind"] == "monitor":
        out["log"] = log
    return out
