"""The work that a user of this package has it do, as cases that can be timed.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (lattice objects with their state, or recorded series),
``run`` is one call through the package's public entry points and returns its
outputs whole, ``work`` is what the call cannot do without, and ``exact`` is
the same result from plain torch in 64 bits, without this package.

Kinds:
  step       Lattice.step on a batch of lattices (static criticality,
             relaxation, finite-size scaling, schedules of field and
             couplings), with the state continued from pass to pass;
  quench     set_schedule for every configuration and one Lattice.step over
             the longest ramp: a Kibble-Zurek quench of uneven lengths;
  adjoint    Lattice.adjoint: objective and gradients of a trajectory;
  labels     Lattice.label_domains on quenched states;
  structure  Lattice.structure_factor (correlation lengths, App. C);
  tau        sampling.autocorr_time over recorded series (App. B).

Records, gradients and structure factors come back from the package in
doubles but are sums of FP32 site terms, whose grouping (and so the digits
past FP32) depends on the kernel and strip height that the package's
autotuner picks on the machine at hand; ``run`` hands them on in FP32, the
precision they carry.
"""
import math

import numpy as np
import torch

from paper_2409_06412_gb300 import XY_INIT_ORDERED, XY_INIT_USER, Config, Lattice, PAPER_PARAMS
from paper_2409_06412_gb300.sampling import autocorr_time

T_C = 1.969  # the paper's critical temperature for its couplings and field
FOREVER = 10 ** 12


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # one sampling interval (ds = 100 steps) of the plain-method lattice, a
        # single 64 x 64 from a random start: the smallest call, all latency
        dict(name="interval-64", kind="step", shapes="64x64", temps=1, replicas=1, steps=100, every=100,
             start="random"),
        # finite-size scaling on small lattices, sampled often: many lattices
        # that each fit one SM or a cluster
        dict(name="scaling-small", kind="step", shapes="32x32,64x64,128x128", temps=16, replicas=8, steps=100,
             every=10, start="ordered"),
        # static criticality: the benchmark's four sizes, temperatures around
        # T_c, one sampling interval; half its temperatures and an eighth of
        # its replicas (state 0.36 GB, larger than L2)
        dict(name="static-mix", kind="step", shapes="128x128,256x256,512x512,1024x1024", temps=16, replicas=2,
             steps=100, every=100, start="ordered"),
        # dynamic exponent z: relaxation of the ordered state at T_c, sizes up
        # to 2048, M and E every 10 steps
        dict(name="relax-z", kind="step", shapes="256x256,512x512,1024x1024,2048x2048", temps=1, replicas=6,
             steps=100, every=10, start="ordered"),
        # one mid-sized lattice alone under an orthogonal and anisotropic quench:
        # field schedule and coupling profiles, followed closely
        dict(name="schedules-512", kind="step", shapes="512x512", temps=1, replicas=1, steps=200, every=50,
             start="ordered", schedules=True),
        # lattices whose sides are no multiples of the tile sizes (lattices
        # matched to a terrace, periodic cells of an experiment's image)
        dict(name="ragged", kind="step", shapes="100x60,200x150,500x333,1000x1000", temps=2, replicas=4, steps=100,
             every=50, start="ordered"),
        # Kibble-Zurek quench: 1024 x 1024, ramps from 1.5 T_c to 0 of uneven
        # length over damping and field settings
        dict(name="quench-1024", kind="quench", shapes="1024x1024", taus="100,200,400", etas="0.1,1,10", fields="1,2",
             replicas=1),
        # the differentiation workload (64 replicas of 256 x 256 at T_c,
        # checkpoint every 100), a quarter of its 2000 steps
        dict(name="adjoint-256", kind="adjoint", shapes="256x256", replicas=64, steps=500, checkpoint=100, w_E=1.0,
             w_M=1.0),
        # a gradient step on small lattices, as in a fit of the couplings
        dict(name="adjoint-small", kind="adjoint", shapes="64x64", replicas=4, steps=100, checkpoint=20, w_E=1.0,
             w_M=0.5),
        # frozen domains of 64 quenched lattices
        dict(name="labels-1024", kind="labels", shapes="1024x1024", replicas=64),
        # structure factors near k = 0 of one temperature's replicas
        dict(name="structure-1024", kind="structure", shapes="1024x1024", replicas=16, K=16),
        # autocorrelation time of M^2 over the records of 256 replicas (10^5
        # steps, one record per 10)
        dict(name="tau-256", kind="tau", series=256, records=10000, tau=60, transform="f2", window=6.0),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def shape(lo=16, hi=1400):
        if rng.random() < 0.5:
            return (2 ** rng.randint(4, 11), 2 ** rng.randint(4, 11))
        return (4 * max(2, log_int(lo, hi) // 4), log_int(lo, hi))

    def some(n, budget, hi=1400):
        """n shapes and a replica count that keep the sites near `budget`."""
        got = [shape(hi=hi) for _ in range(n)]
        while sum(x * y for x, y in got) > budget and max(x * y for x, y in got) > 4096:
            k = max(range(n), key=lambda i: got[i][0] * got[i][1])
            got[k] = (max(16, got[k][0] // 8 * 4), max(8, got[k][1] // 2))
        reps = max(1, min(256, budget // sum(x * y for x, y in got)))
        return ",".join("%dx%d" % s for s in got), reps

    kind = rng.choice(["step", "step", "step", "quench", "adjoint", "labels", "structure", "tau"])
    if kind == "step":
        temps = rng.choice([1, 2, 3, 8])
        sites = log_int(2e4, 2e7)
        shapes, reps = some(rng.randint(1, 3), max(4096, sites // temps))
        steps = max(10, min(log_int(20, 400), int(1.5e9 / max(1, sites))))
        return dict(kind="step", shapes=shapes, temps=temps, replicas=reps, steps=steps,
                    every=rng.choice([0, 1, 7, 10, 50, 100]), start=rng.choice(["ordered", "random"]),
                    schedules=rng.random() < 0.2)
    if kind == "quench":
        shapes, reps = some(1, log_int(1e4, 5e5))
        taus = sorted({log_int(30, 400) for _ in range(rng.randint(2, 4))})
        etas, fields = rng.choice([("1", "1"), ("0.1,1,10", "1"), ("1", "0.5,1,2")])
        return dict(kind="quench", shapes=shapes, taus=",".join(map(str, taus)), etas=etas, fields=fields,
                    replicas=min(reps, 4))
    if kind == "adjoint":
        sites = log_int(4e3, 4e6)
        shapes, reps = some(1, sites, hi=600)
        return dict(kind="adjoint", shapes=shapes, replicas=reps, steps=max(8, min(log_int(20, 500), int(8e8 / sites))),
                    checkpoint=rng.choice([10, 20, 50, 100]), w_E=1.0, w_M=rng.choice([0.0, 0.5, 1.0]))
    if kind == "labels":
        shapes, reps = some(1, log_int(4e4, 6e7))
        return dict(kind="labels", shapes=shapes, replicas=reps)
    if kind == "structure":
        shapes, reps = some(1, log_int(4e4, 1.6e7))
        return dict(kind="structure", shapes=shapes, replicas=reps, K=min([rng.choice([4, 8, 16, 24])] +
                                                                          [int(v) for v in shapes.split("x")]))
    return dict(kind="tau", series=log_int(16, 512), records=log_int(300, 10000), tau=rng.choice([3, 20, 60]),
                transform=rng.choice(["f", "f2", "f4", "abs"]), window=6.0)


def _shapes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split(",")]


def _nums(text):
    return [float(v) for v in text.split(",")]


# the field goes through zero and back, the couplings part and meet again, over
# many passes
_FIELD = ((0, 4000, 8000), (1.0, 0.2, 1.0))
_COUPLINGS = ((0, 6000, 12000), (1.0, 0.7, 1.0), (1.0, 2.0, 1.0))


def _configs(case):
    """[(Lx, Ly, replicas, params, T knots)] in the order of the state."""
    out = []
    for Lx, Ly in _shapes(case):
        if case["kind"] == "step":
            n = case["temps"]
            for i in range(n):
                T = T_C * (1.0 if n == 1 else 0.9 + 0.2 * i / (n - 1))
                out.append((Lx, Ly, case["replicas"], {}, ((0,), (T,)), FOREVER))
        elif case["kind"] == "quench":
            for tau in _nums(case["taus"]):
                ramp = int(round(1.5 * tau))
                for eta in _nums(case["etas"]):
                    for f in _nums(case["fields"]):
                        out.append((Lx, Ly, case["replicas"], dict(eta=eta, h=f * PAPER_PARAMS["h"]),
                                    ((0, ramp), (1.5 * T_C, 0.0)), ramp))
        else:
            out.append((Lx, Ly, case["replicas"], {}, ((0,), (T_C,)), FOREVER))
    return out


def _random_angles(case, seed):
    n = sum(Lx * Ly * r for Lx, Ly, r, _, _, _ in _configs(case))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.rand(n, generator=gen, device="cuda") - 0.5) * 3.14159


def _domains(case, seed):
    """Angles after a quench: domains around +-2 pi / 5, longer along the dimer
    rows, with thermal spread and a few sites the other way up."""
    (Lx, Ly), = _shapes(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kx = torch.fft.rfftfreq(Lx, device="cuda")
    ky = torch.fft.fftfreq(Ly, device="cuda")
    damp = torch.exp(-0.5 * ((2 * math.pi * 6.0 * kx[None, :]) ** 2 + (2 * math.pi * 2.0 * ky[:, None]) ** 2))
    out = torch.empty((case["replicas"], Ly, Lx), device="cuda")
    for r in range(case["replicas"]):
        noise = torch.randn((Ly, Lx), generator=gen, device="cuda")
        smooth = torch.fft.irfft2(torch.fft.rfft2(noise) * damp, s=(Ly, Lx))
        up = torch.where(smooth >= 0, 1.0, -1.0)
        up = torch.where(torch.rand((Ly, Lx), generator=gen, device="cuda") < 0.01, -up, up)
        out[r] = up * (1.2566370614 + 0.1 * torch.randn((Ly, Lx), generator=gen, device="cuda")).clamp(0.02, 1.55)
    return out.reshape(-1)


def _series(case, seed):
    """Recorded (M, E) with exponentially decaying correlations."""
    B, R = case["series"], case["records"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn((B, 2, R), generator=gen, device="cuda", dtype=torch.float64)
    t = torch.arange(R, device="cuda", dtype=torch.float64)
    kern = torch.exp(-t / case["tau"])
    n = 2 * R
    f = torch.fft.irfft(torch.fft.rfft(z, n=n) * torch.fft.rfft(kern, n=n), n=n)[..., :R]
    f = f / f.std()
    rec = torch.stack([0.3 + 0.1 * f[:, 0], -9.0 + 0.05 * f[:, 1]], dim=-1)
    return rec.contiguous()


def prepare(case, seed):
    if case["kind"] == "tau":
        return dict(case=case, rec=_series(case, seed))
    specs = _configs(case)
    theta = omega = None
    mode = XY_INIT_ORDERED
    if case["kind"] in ("labels", "structure"):
        theta = _domains(case, seed)
    elif case["kind"] == "quench" or case.get("start") == "random":
        theta = _random_angles(case, seed)
    if theta is not None:
        mode, omega = XY_INIT_USER, torch.zeros_like(theta)
    sched = dict(field=_FIELD, couplings=_COUPLINGS) if case.get("schedules") else {}
    lat = Lattice([Config(Lx=Lx, Ly=Ly, n_replicas=r, seed=seed, init_mode=mode, params=prm, knots=knots,
                          n_total=n_total, **sched) for Lx, Ly, r, prm, knots, n_total in specs],
                  theta=theta, omega=omega)
    state = dict(case=case, lat=lat)
    if case["kind"] == "step" and case["every"]:
        state["rec"] = torch.zeros((lat.n_lattices, case["steps"] // case["every"] + 1, 2), dtype=torch.float64,
                                   device="cuda")
    if case["kind"] == "quench":
        state["ramps"] = [s[4][0][1] for s in specs]
        state["k"] = [0] * len(specs)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "tau":
        return [autocorr_time(state["rec"], "M", case["transform"], c_window=case["window"]).float()]
    lat = state["lat"]
    if kind == "step":
        if not case["every"]:
            lat.step(case["steps"])
            return [lat.theta, lat.omega]
        rec = lat.step(case["steps"], case["every"], rec=state["rec"])
        return [lat.theta, lat.omega, rec.float()]
    if kind == "quench":
        for c, (k, ramp) in enumerate(zip(state["k"], state["ramps"])):
            lat.set_schedule(c, (k, k + ramp), (1.5 * T_C, 0.0), k + ramp)
        lat.step(max(state["ramps"]))
        state["k"] = [k + ramp for k, ramp in zip(state["k"], state["ramps"])]
        return [lat.theta, lat.omega]
    if kind == "adjoint":
        obj, grads = lat.adjoint(case["steps"], case["checkpoint"], case["w_E"], case["w_M"])
        return [np.float32(obj), grads.astype(np.float32), lat.theta, lat.omega]
    if kind == "labels":
        return list(lat.label_domains(hist_cap=8192))
    S_par, S_perp = lat.structure_factor(K=case["K"])
    return [S_par.float(), S_perp.float()]


# ------------------------------------------------------------------ the work

# Arithmetic of one site-update: the force from four neighbours (sin and cos
# of q theta, sin of p theta, 18 products and sums), the merged update (10) and
# a Gaussian (half a Box-Muller pair: 12), transcendentals counted as one each.
STEP_FLOPS = 45
# Reverse of one site-update: the site-local adjoint, the Hessian of four
# bonds and of the field, and the four parameter sums.
ADJOINT_FLOPS = 75


def _site_steps(case):
    n = 0
    for Lx, Ly, r, _, _, n_total in _configs(case):
        n += Lx * Ly * r * min(case.get("steps", FOREVER), n_total)
    return n


def work(case):
    if case["kind"] == "tau":
        B, R = case["series"], case["records"]
        lags = min(R // 2, 6 * case["tau"])
        return {"bytes": 8 * B * R + 16 * B, "flops": 2.0 * B * R * lags}
    sites = sum(Lx * Ly * r for Lx, Ly, r, _, _, _ in _configs(case))
    B = sum(c[2] for c in _configs(case))
    if case["kind"] == "labels":
        return {"bytes": 8 * sites + 16 * 8192 * B, "flops": 0}
    if case["kind"] == "structure":
        # transforms along both directions of two real components, of which K
        # wavenumbers are kept: 2.5 N log2 N per component and direction at most
        n = sum(Lx * Ly * r * (math.log2(Lx) + math.log2(Ly)) for Lx, Ly, r, _, _, _ in _configs(case))
        direct = 8.0 * 2 * case["K"] * sites
        return {"bytes": 4 * sites + 16 * case["K"] * B, "flops": min(5.0 * n, direct)}
    # theta and omega in and out
    flops = STEP_FLOPS * _site_steps(case)
    if case["kind"] == "adjoint":
        flops += ADJOINT_FLOPS * _site_steps(case)
    return {"bytes": 16 * sites, "flops": flops}


# ------------------------------------------------------------------ in 64 bits

_EXACT_SITE_STEPS = 7e9   # a forward trajectory above this would take over 20 s
# From a random start FP32 and 64 bits part over some hundred steps (unstable
# bonds, and sites that cross the cut at +-pi/2): beyond this a 64-bit
# trajectory says nothing about an FP32 one.
_EXACT_RANDOM_STEPS = 120
_EXACT_TAPE = 4e6         # site-steps of a gradient by automatic differentiation
_MASK = 0xFFFFFFFF


def _mul(a, x):
    """High and low words of the 64-bit product of a constant and words x (in int64)."""
    p0, p1 = a * (x & 0xFFFF), a * (x >> 16)
    t = p0 + ((p1 & 0xFFFF) << 16)
    return (p1 >> 16) + (t >> 32), t & _MASK


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 words."""
    k0, k1 = key & _MASK, key >> 32
    for _ in range(10):
        h0, l0 = _mul(0xD2511F53, c0)
        h1, l1 = _mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return c0, c1, c2, c3


def _gauss(ids, Lx, Ly, k, seed):
    """Unit Gaussians of step k of lattices `ids` ((config << 16) | replica): (B, Ly, Lx)."""
    quad = torch.arange(Lx * Ly // 4, device=ids.device, dtype=torch.int64)[None, :]
    zero = torch.zeros_like(quad)
    w = _philox(quad, ids[:, None], zero + (k & _MASK), zero + (k >> 32), seed)
    u = [((x >> 9).double() + 0.5) * 2.0 ** -23 for x in w]
    g = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = torch.sqrt(-2.0 * torch.log(a))
        g += [r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)]
    return torch.stack(g, dim=-1).reshape(ids.numel(), Ly, Lx)


def _profile(k, knots, col):
    return float(np.interp(k, knots[0], knots[col]))


class _Model:
    """Lattices of one shape, each with its own constants, in 64 bits."""

    def __init__(self, Lx, Ly, ids, par, knots, seed, sched):
        self.Lx, self.Ly, self.seed, self.sched = Lx, Ly, seed, sched
        self.ids, self.par, self.knots = ids, par, knots
        self.q, self.p, self.dt = PAPER_PARAMS["q"], PAPER_PARAMS["p"], PAPER_PARAMS["dt"]

    def couplings(self, k):
        Jx, Jy, h, _ = self.par
        if self.sched:
            return (Jx * _profile(k, _COUPLINGS, 1), Jy * _profile(k, _COUPLINGS, 2), h * _profile(k, _FIELD, 1))
        return Jx, Jy, h

    def kick(self, theta, k):
        """g_k = dt/2 F(theta_k) + c_k n_k"""
        Jx, Jy, h = self.couplings(k)
        q, p = self.q, self.p
        T = torch.tensor([float(np.interp(k, kn[0], kn[1])) for kn in self.knots], dtype=torch.float64,
                         device=theta.device)[:, None, None]
        d = lambda n, ax: torch.sin(q * (theta - torch.roll(theta, n, ax)))  # noqa: E731
        F = -q * Jx * (d(1, 2) + d(-1, 2)) - q * Jy * (d(1, 1) + d(-1, 1)) + h * p * torch.sin(p * theta)
        c = 0.5 * torch.sqrt(2.0 * self.par[3] * T * self.dt)
        return 0.5 * self.dt * F + c * _gauss(self.ids, self.Lx, self.Ly, k, self.seed)

    def omega(self, v, g):
        return (v + g) / (1.0 + 0.5 * self.par[3] * self.dt)

    def advance(self, theta, om, g):
        v = (1.0 - 0.5 * self.par[3] * self.dt) * om + g
        t = theta + self.dt * v
        return t - math.pi * torch.floor(t.detach() / math.pi + 0.5), v

    def observe(self, theta, om, k):
        """M, E per lattice"""
        Jx, Jy, h = self.couplings(k)
        q = self.q
        M = torch.sin(q * theta).mean(dim=(1, 2))
        E = (0.5 * om * om - Jx * torch.cos(q * (theta - torch.roll(theta, -1, 2)))
             - Jy * torch.cos(q * (theta - torch.roll(theta, -1, 1))) + h * torch.cos(self.p * theta))
        return M, E.mean(dim=(1, 2))


def _start(case, seed):
    """theta_0 per configuration, in 64 bits"""
    specs = _configs(case)
    if case["kind"] == "quench" or case.get("start") == "random":
        flat = _random_angles(case, seed).double()
    else:
        n = sum(Lx * Ly * r for Lx, Ly, r, _, _, _ in specs)
        flat = torch.full((n,), float(np.float32(2 * math.pi / 5)), dtype=torch.float64, device="cuda")
    out, at = [], 0
    for Lx, Ly, r, _, _, _ in specs:
        out.append(flat[at:at + Lx * Ly * r].reshape(r, Ly, Lx))
        at += Lx * Ly * r
    return out


def _groups(case, seed, grad=False):
    """(model, theta_0, config indices, steps) of the configurations that share shape and length."""
    specs, start = _configs(case), _start(case, seed)
    keys = {}
    for c, s in enumerate(specs):
        keys.setdefault((s[0], s[1], min(case.get("steps", FOREVER), s[5])), []).append(c)
    for (Lx, Ly, n), cs in keys.items():
        reps = [specs[c][2] for c in cs]
        ids = torch.tensor([(c << 16) | r for c, m in zip(cs, reps) for r in range(m)], device="cuda")
        per_cfg, par = [], []
        for name in ("J_par", "J_perp", "h", "eta"):
            v = torch.tensor([float({**PAPER_PARAMS, **specs[c][3]}[name]) for c in cs], dtype=torch.float64,
                             device="cuda", requires_grad=grad)
            per_cfg.append(v)
            par.append(torch.cat([v[i:i + 1].expand(m) for i, m in enumerate(reps)])[:, None, None])
        knots = [specs[c][4] for c, m in zip(cs, reps) for _ in range(m)]
        yield _Model(Lx, Ly, ids, par, knots, seed, bool(case.get("schedules"))), torch.cat(
            [start[c] for c in cs]), cs, reps, n, per_cfg


def _exact_forward(case, seed):
    specs = _configs(case)
    every = case.get("every", 0)
    R = case["steps"] // every + 1 if every else 0
    th_out, v_out, rec_out = [None] * len(specs), [None] * len(specs), [None] * len(specs)
    for m, theta, cs, reps, n, _ in _groups(case, seed):
        v = None
        rec = torch.zeros((theta.shape[0], R, 2), dtype=torch.float64, device="cuda")
        for k in range(n):
            g = m.kick(theta, k)
            # the full-step velocity at step 0 is zero
            om = torch.zeros_like(theta) if v is None else m.omega(v, g)
            if every and k % every == 0:
                M, E = m.observe(theta, om, k)
                rec[:, k // every, 0], rec[:, k // every, 1] = M, E
            theta, v = m.advance(theta, om, g)
            theta = torch.where(theta >= 0.5 * math.pi, theta - math.pi, theta)
        at = 0
        for c, r in zip(cs, reps):
            th_out[c], v_out[c], rec_out[c] = (x[at:at + r] for x in (theta, v, rec))
            at += r
    flat = [torch.cat([x.reshape(-1) for x in o]) for o in (th_out, v_out)]
    return flat + ([torch.cat(rec_out)] if every else [])


def _exact_adjoint(case, seed):
    (m, theta, _, _, n, par), = _groups(case, seed, grad=True)
    total = torch.zeros((), dtype=torch.float64, device="cuda")
    v = None
    for k in range(n + 1):
        g = m.kick(theta, k)
        om = torch.zeros_like(theta) if v is None else m.omega(v, g)
        if k > 0:
            M, E = m.observe(theta, om, k)
            total = total + (case["w_E"] * E + case["w_M"] * M.abs()).sum()
        if k < n:
            theta, v = m.advance(theta, om, g)
    obj = total / (theta.shape[0] * n)
    grads = torch.autograd.grad(obj, par)
    return [float(obj), torch.stack(grads, dim=1).detach(), theta.detach().reshape(-1), v.detach().reshape(-1)]


def _exact_structure(case, seed):
    (Lx, Ly), = _shapes(case)
    th = _domains(case, seed).double().reshape(-1, Ly, Lx)
    out = [[], []]
    for t in th:
        z = [torch.cos(t), torch.sin(t)]
        for i, ax in enumerate((1, 0)):
            S = sum((torch.fft.fft(s, dim=ax).abs() ** 2).sum(dim=1 - ax) for s in z)
            out[i].append(S[:case["K"]] / (Lx * Ly))
    return [torch.stack(o) for o in out]


def _exact_tau(case, seed):
    f = _series(case, seed)[..., 0]
    f = {"f": lambda x: x, "f2": torch.square, "f4": lambda x: x ** 4, "abs": torch.abs}[case["transform"]](f)
    B, n = f.shape
    mean = f.mean(dim=1)
    d = f - mean[:, None]
    spec = torch.fft.rfft(d, n=2 * n)
    C = torch.fft.irfft(spec.abs() ** 2, n=2 * n)[:, :n // 2 + 1]
    C = C / (n - torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64))
    tau = 0.5 + torch.cumsum(C[:, 1:] / C[:, :1], dim=1)
    lag = torch.arange(1, n // 2 + 1, device="cuda", dtype=torch.float64)
    done = lag[None, :] >= case["window"] * tau
    done[:, -1] = True
    at = done.int().argmax(dim=1)
    tau = tau.gather(1, at[:, None])[:, 0]
    return [torch.stack([mean, C[:, 0], tau, torch.sqrt(2 * tau * C[:, 0] / n)], dim=1)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "labels":
        return None  # whole numbers
    if kind == "structure":
        return _exact_structure(case, seed)
    if kind == "tau":
        return _exact_tau(case, seed)
    if kind == "adjoint" and _site_steps(case) <= _EXACT_TAPE:
        return _exact_adjoint(case, seed)
    if _site_steps(case) > _EXACT_SITE_STEPS:
        return None
    if (kind == "quench" or case.get("start") == "random") and max(
            min(case.get("steps", FOREVER), c[5]) for c in _configs(case)) > _EXACT_RANDOM_STEPS:
        return None
    out = _exact_forward(case, seed)
    return [None, None] + out if kind == "adjoint" else out
