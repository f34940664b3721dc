"""What a user of this framework has it do: whole calls through its public entry points, over the range of lattices,
boundary kinds, precisions and directions that its configurations, tests and benchmark run.

Kinds of case
  run     init, step(n) and macro of a periodic box (a solver run; convergence studies are many of these)
  box     the same in a Dirichlet box, its boundary data from the exact-solution family or the manufactured solution
  grad    loss and gradients of a periodic run through autograd (fit of the initial field and of the source)
  boxgrad phi(T) of a Dirichlet box and its gradients w.r.t. initial data and every step's boundary jets
  series  a run that reads the diagnostics every few steps (entropy series of a tanh bubble)
  map     the stability map of a batch of velocities

exact() repeats each case in plain torch / numpy in 64 bits, written from the scheme's equations (post-collision
populations f*, pulled and collided; boundary data as sums of complex exponentials, on which every derivative is a
factor)."""
import itertools
import math

import numpy as np
import torch

import paper_2410_13165_gb300 as lhe
from paper_2410_13165_gb300.autograd import LBMBoxFunction, lbm_loss

DEVICE = "cuda"
# velocities of the workloads, by dimension (the half-way scheme is stable at small velocities only)
U = {1: (0.3,), 2: (0.1, 0.05), 3: (0.1, 0.1, 0.1), 4: (0.05, 0.2, 0.08, 0.1), 5: (0.02, 0.04, 0.06, 0.08, 0.1)}
U_HALFWAY = 1e-3


def _run(name, n, **kw):
    c = {**({"name": name} if name else {}), "kind": "run", "n": n, "precision": "fp64", "tau": 0.8, "steps": 20, "source": "none", "R": 0.0, "grad": True}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest solver run: 2D, 200 steps of a grid that one SM's registers could hold; launches and latency
        _run("d2q9_64_fp64", "64x64", steps=200),
        # 2D grid of odd extents in 32 bits, as in the studies of where single precision stops converging
        _run("d2q9_500x333_fp32dev", "500x333", precision="fp32dev", tau=0.5, steps=100, grad=False),
        # a small 3D run on odd extents with a source field (convergence studies; tau above 1)
        _run("d3q19_45x37x51_fp64_source", "45x37x51", tau=1.2, steps=100, source="field", grad=False),
        # the precision workload: 3D, 32-bit deviations
        _run("d3q19_128_fp32dev", "128x128x128", precision="fp32dev", tau=0.5, steps=50),
        # the throughput workload: 3D, 64 bits, the finite-difference gradient formed by the library
        _run("d3q19_256_fp64", "256x256x256", steps=20, grad=False),
        # the largest lattice: 5D, 32-bit deviations
        _run("d5q51_24_fp32dev", "24x24x24x24x24", precision="fp32dev", tau=0.5, steps=5, grad=False),
        # Example 3's travelling sine in a 4D box, full-way scheme
        {"name": "d4q33_32_fullway", "kind": "box", "n": "32x32x32x32", "bc": "fullway", "order": 4, "data": "wave", "R": 0.0,
         "precision": "fp64", "tau": 0.5, "steps": 20},
        # the manufactured solution with its source in a 3D box, half-way scheme
        {"name": "d3q19_48_halfway_sines", "kind": "box", "n": "48x48x48", "bc": "halfway", "order": 4, "data": "sines", "R": 0.0,
         "precision": "fp64", "tau": 0.5, "steps": 50},
        # fitting an initial field and a source: forward and backward through autograd
        {"name": "grad_d3q19_128_fp32dev", "kind": "grad", "n": "128x128x128", "precision": "fp32dev", "tau": 0.5, "steps": 32},
        # gradients w.r.t. boundary data of a 2D box, one block of jets per step
        {"name": "boxgrad_d2q9_48x40_fullway", "kind": "boxgrad", "n": "48x40", "bc": "fullway", "order": 4, "R": 5.0,
         "precision": "fp64", "tau": 0.5, "steps": 32},
        # entropy series of the 3D bubble: the diagnostics every 10 steps
        {"name": "series_d3q19_96_fp64", "kind": "series", "n": "96x96x96", "precision": "fp64", "tau": 0.5, "every": 10, "points": 6},
        # stability map of 3D velocities, 12 wave numbers an axis
        {"name": "map_d3q19", "kind": "map", "d": 3, "points": 24, "nxi": 12, "tau": 0.5},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extents(rng, d, nodes, least):
    side = nodes ** (1.0 / d)
    n = [max(least, int(round(side * rng.uniform(0.75, 1.3)))) for _ in range(d)]
    if rng.random() < 0.3:  # cubes, and rows of a multiple of 8
        n = [max(8, int(round(side / 8)) * 8)] * d
    return n


def draw(rng):
    kind = rng.choice(["run"] * 9 + ["box"] * 5 + ["grad"] * 2 + ["boxgrad"] * 2 + ["series"] * 2 + ["map"] * 2)
    if kind == "map":
        d = rng.choice([1, 2, 2, 3, 3, 4])
        nxi = {1: rng.randint(32, 500), 2: rng.randint(16, 40), 3: rng.randint(6, 12), 4: rng.randint(3, 5)}[d]
        most = min(400, max(2, {1: 600000, 2: 100000, 3: 35000, 4: 6000}[d] // nxi ** d))
        return {"kind": kind, "d": d, "points": int(_log(rng, 2, most)), "nxi": nxi, "tau": rng.choice([0.5, 0.5, 0.8])}
    precision = rng.choice(["fp64", "fp32dev"])
    if kind in ("run", "series"):
        d = rng.choice([1, 2, 2, 3, 3, 3, 4, 5]) if kind == "run" else rng.choice([2, 3, 3, 4])
    else:
        d = rng.choice([2, 3, 3, 4]) if kind == "box" else rng.choice([2, 3])
    q = 2 * d * d + 1
    if kind == "boxgrad":
        nodes = _log(rng, 200, 4000 if d == 2 else 3000)
        n = _extents(rng, d, nodes, 5)
        bc = rng.choice(["fullway", "halfway"])
        return {"kind": kind, "n": "x".join(map(str, n)), "bc": bc, "order": rng.choice([3, 4]), "R": rng.choice([0.0, 5.0]), "precision": precision, "tau": rng.choice([0.5, 0.8]),
                "steps": rng.randint(4, 40 if d == 2 else 12)}
    if kind == "box":
        n = _extents(rng, d, _log(rng, 1000, 8e5), 6)
        nodes = math.prod(n)
        bc = rng.choice(["fullway", "halfway"])
        data = rng.choice(["wave", "sines"])
        return {"kind": kind, "n": "x".join(map(str, n)), "bc": bc, "order": rng.choice([3, 4, 4]), "data": data, "precision": precision,
                "R": rng.choice([0.0, 5.0]) if data == "wave" else 0.0,
                "tau": rng.choice([0.5, 0.5, 0.8]), "steps": max(1, int(min(_log(rng, 5, 150), 1e9 / (nodes * q))))}
    least = 6 if d > 3 else 8
    n = _extents(rng, d, _log(rng, 1000 if d < 4 else 10000, {1: 2e6, 2: 1.2e7, 3: 1.2e7, 4: 5e6, 5: 6e6}[d] / (4 if kind != "run" else 1)), least)
    nodes = math.prod(n)
    steps = max(1, int(min(_log(rng, 5, 200), 5e9 / (nodes * q))))
    tau = rng.choice([0.5, 0.5, 0.6, 0.8, 1.2])
    if kind == "grad":
        return {"kind": kind, "n": "x".join(map(str, n)), "precision": precision, "tau": tau, "steps": max(1, steps // 3)}
    if kind == "series":
        every = rng.randint(2, 20)
        return {"kind": kind, "n": "x".join(map(str, n)), "precision": precision, "tau": tau, "every": every, "points": max(1, min(12, steps // every))}
    return _run("", "x".join(map(str, n)), precision=precision, tau=tau, steps=steps, source=rng.choice(["none", "none", "field"]),
                R=rng.choice([0.0, 0.0, 5.0]), grad=rng.choice([True, False]))


# ------------------------------------------------------------------------------------------------ inputs
def _dims(c):
    return [int(v) for v in c["n"].split("x")]


def _box(c):
    """Extents, spacing, lower and upper corners (a square lattice of spacing dx, the longest side of length `side`) and velocity."""
    n = _dims(c)
    d, bc = len(n), c.get("bc", "periodic")
    side = 2.0 if c["kind"] in ("box", "series") else 1.0
    lo = -1.0 if c["kind"] in ("box", "series") else 0.0
    span = [m - 1 if bc == "fullway" else m for m in n]
    dx = side / max(span)
    hi = [lo + s * dx for s in span]
    u = (U_HALFWAY,) * d if bc == "halfway" else U[d]
    return n, dx, lo, hi, u


def _axes(c):
    n, dx, lo, _, _ = _box(c)
    off = 0.5 if c.get("bc") == "halfway" else 0.0
    return [lo + dx * (torch.arange(m, dtype=torch.float64, device=DEVICE) + off) for m in n]


def _phase(axes, k, shift=0.0):
    """sum_i k_i x_i + shift on the grid, shape (n_d, .., n_1)."""
    d = len(axes)
    out = torch.full((1,) * d, float(shift), dtype=torch.float64, device=DEVICE)
    for i, x in enumerate(axes):
        out = out + (float(k[i]) * x).reshape([-1 if j == d - 1 - i else 1 for j in range(d)])
    return out


def _modes(c, rng, count=6):
    """Fourier modes with integer wave numbers 1..3 of the box (periodic in it): rows (a, kappa, theta)."""
    n, dx, lo, hi, _ = _box(c)
    out = []
    for _ in range(count):
        k = [2 * math.pi * int(rng.integers(1, 4)) / (h - lo) for h in hi]
        out.append((float(rng.uniform(-1, 1)), k, float(rng.uniform(0, 2 * math.pi))))
    return out


def _field(axes, modes, mean=0.0, want_grad=False):
    """The field (a mean keeps it from decaying to rounding where tau damps its modes) and its gradient."""
    phi, grad = mean, [0.0] * len(axes)
    for a, k, th in modes:
        z = _phase(axes, k, th)
        phi = phi + a * torch.sin(z)
        if want_grad:
            cz = a * torch.cos(z)
            grad = [g + k[i] * cz for i, g in enumerate(grad)]
    return phi.reshape(-1).contiguous(), torch.stack([g.reshape(-1) for g in grad]).reshape(-1) if want_grad else None


def _rng(seed, salt=0):
    return np.random.default_rng([2410131650, int(seed), salt])


def _exps(c, seed):
    """Boundary data phi = Re sum_j C_j exp(i kappa_j . x + mu_j t), and what the library is given for it."""
    _, _, lo, hi, u = _box(c)
    d, rng = len(u), _rng(seed, 1)
    if c.get("data") == "sines":
        A, lam, k, th = float(rng.uniform(0.5, 1.5)), 1.0, [math.pi] * d, [float(v) for v in rng.uniform(0, 2 * math.pi, d)]
        terms = []
        for s in itertools.product((1, -1), repeat=d):
            C = A * np.prod(s) / (2j) ** d * np.exp(1j * np.dot(s, th))
            terms.append((complex(C), [a * b for a, b in zip(s, k)], complex(-lam)))
        return terms, {"A": A, "lam": lam, "kappa": k, "theta": th}
    # Example 3's sin(pi sum_i (x_i - u_i t)), its amplitude and phase drawn, and a second mode
    a, kap, th = [], [], []
    for m in range(1 if d == 4 else 2):
        a.append(float(rng.uniform(0.5, 1.5)))
        kap.append([math.pi * (1 if m == 0 else int(rng.integers(1, 3))) for _ in range(d)])
        th.append(float(rng.uniform(0, 2 * math.pi)))
    terms = [(complex(a[m] * np.exp(1j * th[m]) / 1j), kap[m], complex(0, -np.dot(kap[m], u))) for m in range(len(a))]
    return terms, {"a": a, "kappa": kap, "theta": th}


def _exp_field(axes, terms, t, op=None):
    """Re sum_j op_j C_j exp(i kappa_j . x + mu_j t) on the grid; op(kappa, mu) a complex factor."""
    out = 0.0
    for C, k, mu in terms:
        w = C * np.exp(mu * t) * (1.0 if op is None else op(np.asarray(k), mu))
        z = _phase(axes, k)
        out = out + w.real * torch.cos(z) - w.imag * torch.sin(z)
    return out


def _bubble(c, seed):
    """Example 2's tanh bubble, centre and radius drawn, distance to the nearest periodic image."""
    _, dx, lo, hi, _ = _box(c)
    axes, rng = _axes(c), _rng(seed, 2)
    d, r2 = len(axes), 0.0
    for i, x in enumerate(axes):
        L = hi[i] - lo
        y = torch.remainder(x - lo - float(rng.uniform(0, L)) + 0.5 * L, L) - 0.5 * L
        r2 = r2 + (y * y).reshape([-1 if j == d - 1 - i else 1 for j in range(d)])
    r0, w = 0.5 * float(rng.uniform(0.6, 0.9)) * min(h - lo for h in hi) / 2, 0.06
    return (0.5 - 0.5 * torch.tanh((torch.sqrt(r2) - r0) / (2 * w))).reshape(-1).contiguous()


def _sim(c):
    n, dx, lo, hi, u = _box(c)
    return lhe.LBM(len(n), n, lo=lo, hi=hi, u=u, R=c.get("R", 0.0), tau=c["tau"], bc=c.get("bc", "periodic"), bc_order=c.get("order", 4),
                   precision=c["precision"])


def _inputs(c, seed):
    """The arrays of a case, without a handle (exact() starts from the same ones)."""
    kind = c["kind"]
    if kind == "map":
        d, rng = c["d"], _rng(seed)
        sig = rng.uniform(-0.45, 0.45, size=(c["points"], d)) / (1.0 if d < 3 else d - 1.5)
        sig[::3] *= 2.2  # a third of the velocities further out, past the edge of the stable region
        return {"sig": sig}
    axes = _axes(c)
    if kind in ("run", "grad"):
        mean = float(_rng(seed, 6).uniform(0.5, 1.5))
        phi0, grad = _field(axes, _modes(c, _rng(seed)), mean, kind == "run" and c["grad"])
        R = _field(axes, _modes(c, _rng(seed, 3), 3))[0] if kind == "grad" or c["source"] == "field" else None
        out = {"phi0": phi0, "grad": grad, "R": R}
        if kind == "grad":
            out["target"] = _field(axes, _modes(c, _rng(seed, 4)))[0]
        return out
    if kind == "series":
        return {"phi0": _bubble(c, seed)}
    terms, given = _exps(c, seed)
    u = np.asarray(_box(c)[4])
    d = len(u)
    phi0 = _exp_field(axes, terms, 0.0).reshape(-1).contiguous()
    grad = torch.cat([_exp_field(axes, terms, 0.0, lambda k, mu, i=i: 1j * k[i]).reshape(-1) for i in range(d)])
    R0 = None
    if c.get("data") == "sines":
        R0 = _exp_field(axes, terms, 0.0, lambda k, mu: mu + 1j * np.dot(k, u)).reshape(-1).contiguous()
    return {"phi0": phi0, "grad": grad, "R": R0, "terms": terms, "given": given}


def _jets(c, terms, points, t0, dt):
    """Every derivative of order <= 3 in (t, x_1..x_d) at the points, for each step's time: (T, P, length)."""
    d = len(points[0])
    tuples = [tup for q in range(4) for tup in itertools.combinations_with_replacement(range(d + 1), q)]
    out = np.zeros((c["steps"], len(points), len(tuples)))
    R = c.get("R", 0.0)
    for C, k, mu in terms:
        f = [mu] + [1j * v for v in k]
        w = np.array([np.prod([f[v] for v in tup]) if tup else 1.0 for tup in tuples])
        base = C * np.exp(1j * (points @ np.asarray(k)))
        for s in range(c["steps"]):
            out[s] += ((base * np.exp(mu * (s * dt + t0)))[:, None] * w[None, :]).real
    for s in range(c["steps"]):  # the part R t of an exact solution
        out[s, :, 0] += R * (s * dt + t0)
    out[:, :, 1] += R
    return torch.from_numpy(out).to(DEVICE)


def prepare(case, seed):
    c, v = dict(case), _inputs(case, seed)
    if c["kind"] == "map":
        return {"c": c, **v}
    s = {"c": c, "sim": _sim(c), **{k: x for k, x in v.items() if k not in ("terms", "given")}}
    if c["kind"] == "box":
        if c["data"] == "sines":
            s["sim"].set_boundary_sine_product(**v["given"])
        else:
            s["sim"].set_boundary_wave(**v["given"])
    if c["kind"] == "boxgrad":
        points, t0 = s["sim"].boundary_points()
        s["jets"] = _jets(c, v["terms"], points, t0, s["sim"].dt)
        s["cot"] = torch.from_numpy(_rng(seed, 5).standard_normal(s["phi0"].numel())).to(DEVICE)
    return s


def run(s):
    c = s["c"]
    if c["kind"] == "map":
        rho, omin = lhe.stability_map(c["d"], s["sig"], c["nxi"], tau=c["tau"])
        return {"rho": rho, "omega_min": omin}
    sim = s["sim"]
    if c["kind"] in ("run", "box"):
        sim.init(s["phi0"], s["grad"], s["R"])
        sim.step(c["steps"])
        return {"phi": sim.macro()}
    if c["kind"] == "series":
        sim.init(s["phi0"])
        seen = []
        for _ in range(c["points"]):
            sim.step(c["every"])
            seen.append(sim.diagnostics())
        return {"mass": np.array([v["mass"] for v in seen]), "entropy": np.array([v["entropy"] for v in seen]),
                "max": np.array([v["max_abs"] for v in seen]), "nonfinite": np.array([v["nonfinite"] for v in seen]), "phi": sim.macro()}
    if c["kind"] == "grad":
        phi0, R = s["phi0"].detach().requires_grad_(), s["R"].detach().requires_grad_()
        loss = lbm_loss(phi0, R, sim, c["steps"], s["target"])
        g = torch.autograd.grad(loss, (phi0, R))
        return {"loss": loss.detach(), "dphi0": g[0], "dR": g[1]}
    ins = [s[k].detach().requires_grad_() for k in ("phi0", "grad", "jets")]
    phi = LBMBoxFunction.apply(*ins, sim)
    g = torch.autograd.grad(phi, ins, s["cot"])
    return {"phi": phi.detach(), "dphi0": g[0], "dgrad": g[1], "djets": g[2]}


def work(case):
    """Inputs read once, outputs written once; operations: two per population for the collision and one for the moment
    sum, every node and step (the map: a Hessenberg reduction and QR sweeps are one way; the least known is the roots of
    the rank-one-updated diagonal, some ten sweeps of Q^2 complex terms a matrix)."""
    c = case
    if c["kind"] == "map":
        q, total = 2 * c["d"] ** 2 + 1, c["points"] * c["nxi"] ** c["d"]
        return {"bytes": 8 * c["points"] * (c["d"] + 2), "flops": total * 10 * q * q * 8}
    n = _dims(c)
    d, nodes = len(n), math.prod(n)
    q = 2 * d * d + 1
    flops = lambda steps: 3 * q * nodes * steps  # noqa: E731
    if c["kind"] == "run":
        return {"bytes": 8 * nodes * (2 + (d if c["grad"] else 0) + (c["source"] == "field")), "flops": flops(c["steps"])}
    if c["kind"] == "box":
        return {"bytes": 8 * nodes * (2 + d + (c["data"] == "sines")), "flops": flops(c["steps"])}
    if c["kind"] == "series":
        return {"bytes": 8 * nodes * 2, "flops": flops(c["every"] * c["points"]) + 4 * q * nodes * c["points"]}
    if c["kind"] == "grad":
        return {"bytes": 8 * nodes * 5, "flops": flops(2 * c["steps"])}
    full = c["bc"] == "fullway"
    face = sum(1 for x in itertools.product(*[range(m) for m in n]) if any(v in (0, m - 1) for v, m in zip(x, n)))
    rows = face if full else int(face * (3 if d == 2 else 5))
    return {"bytes": 8 * (nodes * (3 + 2 * d) + 2 * c["steps"] * rows * (d + 4) * (d + 3) * (d + 2) // 6), "flops": flops(2 * c["steps"])}


# ------------------------------------------------------------------------------------------------ the same in 64 bits
def _lattice(d):
    e = [[0] * d] + [[int(i == j) for j in range(d)] for i in range(d)] + [[-int(i == j) for j in range(d)] for i in range(d)]
    for i, j in itertools.combinations(range(d), 2):
        for a, b in ((1, 1), (-1, 1), (-1, -1), (1, -1)):
            v = [0] * d
            v[i], v[j] = a, b
            e.append(v)
    return np.array(e)


def _weights(d, s):
    """EDF weights for sigma = u / c with equal fourth moments, halfway between the bounds of the stable interval."""
    e, ss = _lattice(d), float(np.dot(s, s))
    if d == 1:
        m4 = 0.0
    else:
        low = [(2 * d - 6 + 4 * ss) / (3 * d * (d - 1))]
        for i, j in itertools.combinations(range(d), 2):
            low += [(abs(s[i] + s[j]) - 2 * s[i] * s[j]) / 3, (abs(s[i] - s[j]) + 2 * s[i] * s[j]) / 3]
        m4 = 0.5 * (max(low) + min((1 + 2 * v * v - abs((4 - d) * v)) / (3 * (d - 1)) for v in s))
    w = []
    for v in e:
        at = np.nonzero(v)[0]
        if len(at) == 0:
            w.append((3 - d - 2 * ss + 3 * m4 * d * (d - 1) / 2) / 3)
        elif len(at) == 1:
            i = at[0]
            w.append((v[i] * (4 - d) * s[i] + 1 + 2 * s[i] ** 2 - 3 * (d - 1) * m4) / 6)
        else:
            i, j = at
            w.append((3 * m4 + 2 * v[i] * v[j] * s[i] * s[j] + v[i] * s[i] + v[j] * s[j]) / 12)
    return e, np.array(w)


class _Plain:
    """The scheme on one box: post-collision populations as a list of Q tensors of shape (n_d, .., n_1)."""

    def __init__(self, c):
        self.c = c
        self.n, self.dx, _, _, u = _box(c)
        self.d, self.u, self.dt, self.s = len(self.n), np.asarray(u), self.dx, 1.0 / c["tau"]
        self.e, self.w = _weights(self.d, self.u)
        self.shape = tuple(self.n[::-1])
        self.bar = [int(np.nonzero((self.e == -v).all(1))[0][0]) for v in self.e]
        self.dims = tuple(self.d - 1 - i for i in range(self.d))  # tensor dimension of axis i
        self.order = c.get("order", 4)
        bc = c.get("bc", "periodic")
        self.full, self.half = bc == "fullway", bc == "halfway"
        if self.full or self.half:
            self.out = []  # where population k comes from outside the box
            idx = torch.meshgrid(*[torch.arange(m, device=DEVICE) for m in self.shape], indexing="ij")
            for v in self.e:
                o = torch.zeros(self.shape, dtype=torch.bool, device=DEVICE)
                for i in range(self.d):
                    if v[i]:
                        o = o | (idx[self.dims[i]] == (0 if v[i] == 1 else self.n[i] - 1))
                self.out.append(o)

    def fd(self, p):
        return [sum(a * torch.roll(p, -r, self.dims[i]) for r, a in ((2, -1), (1, 8), (-1, -8), (-2, 1))) / (12 * self.dx) for i in range(self.d)]

    def collide(self, f, R):
        phi = sum(f)
        return [(1 - self.s) * f[k] + float(self.w[k]) * (self.s * phi + self.dt * R) for k in range(len(f))]

    def init(self, phi0, grad, R):
        p = phi0.reshape(self.shape)
        g = self.fd(p) if grad is None else list(grad.reshape((self.d,) + self.shape))
        f = [float(self.w[k]) * (p + 0.5 * self.dt * sum(float(self.u[i] - self.e[k][i]) * g[i] for i in range(self.d))) for k in range(len(self.w))]
        return self.collide(f, R)

    def pull(self, fs):
        out = []
        for k, v in enumerate(self.e):
            at = [i for i in range(self.d) if v[i]]
            out.append(torch.roll(fs[k], [int(v[i]) for i in at], [self.dims[i] for i in at]) if at else fs[k])
        return out

    def factor(self, k, kap, mu):
        """What the boundary scheme makes of exp(i kappa . x + mu t) for the unknown population k (without R)."""
        C, dt, P = 1j * np.dot(kap, self.e[k]), self.dt, self.order
        if self.full:
            D = C + mu
            return self.w[k] * (1 - (0.5 * dt * D if P >= 3 else 0) + (dt ** 3 / 24 * D ** 3 if P >= 4 else 0))
        wp, wm = self.w[k] + self.w[self.bar[k]], self.w[k] - self.w[self.bar[k]]
        v = wp * (1 + (0.5 * dt * mu if P >= 2 else 0))
        if P >= 3:
            v -= wp * dt ** 2 / 8 * C * C + wm * dt ** 2 / 4 * C * mu
        if P >= 4:
            v -= wp * (dt ** 3 / 16 * C * C * mu + dt ** 3 / 24 * mu ** 3) + wm * dt ** 3 / 8 * C * mu * mu
        return v * np.exp(-0.5 * dt * C)

    def source_part(self, k):
        """The scheme's factor on R at the node."""
        if self.full:
            return 0.5 * self.dt * self.w[k] if self.order >= 3 else 0.0
        return 0.5 * self.dt * (self.w[k] + self.w[self.bar[k]]) if self.order >= 2 else 0.0

    def with_data(self, fs, data):
        """Pulled populations of a box, the unknown ones from `data[k]` (half-way: minus f*_kbar at the node)."""
        f = self.pull(fs)
        return [f[k] if k == 0 else torch.where(self.out[k], data[k] - (fs[self.bar[k]] if self.half else 0.0), f[k]) for k in range(len(f))]


def _exact_map(c, sig):
    d, m = c["d"], c["nxi"]
    s = 1.0 / c["tau"]
    xi = -math.pi + 2 * math.pi * np.arange(m) / m
    grid = np.stack([g.ravel() for g in np.meshgrid(*[xi] * d, indexing="ij")], 1)
    if len(grid) * len(sig) * (2 * d * d + 1) ** 3 > 6e8:
        return {"rho": None, "omega_min": np.array([_weights(d, v)[1].min() for v in sig])}
    rho, low = [], []
    for v in sig:
        e, w = _weights(d, v)
        low.append(w.min())
        ph = np.exp(-1j * grid @ e.T)  # (points, Q)
        A = ph[:, :, None] * (np.diag(np.full(len(w), 1 - s)) + s * w[:, None])[None]
        rho.append(np.abs(np.linalg.eigvals(A)).max())
    return {"rho": np.array(rho), "omega_min": np.array(low)}


def _nodes(m):
    """Boundary nodes of a box in the library's order: by the faces they lie on (per axis 1 low, 2 high, the first axis the
    lowest digit in base 3), then by index; and for each its (link, unknown) pairs in the order of the links."""
    keyed = []
    for at, x in enumerate(itertools.product(*[range(v) for v in m.n[::-1]])):
        x = x[::-1]
        sign = sum(3 ** i * (1 if x[i] == 0 else 2 if x[i] == m.n[i] - 1 else 0) for i in range(m.d))
        if sign:
            keyed.append((sign, at, x))
    keyed.sort()
    return [(at, [k for k, v in enumerate(m.e) if any(not 0 <= x[i] - v[i] < m.n[i] for i in range(m.d))]) for _, at, x in keyed]


def _jet_rows(m):
    """Weights of the derivatives in each link's record: (Q, length)."""
    tuples = [tup for q in range(4) for tup in itertools.combinations_with_replacement(range(m.d + 1), q)]
    at, dt, P = {t: i for i, t in enumerate(tuples)}, m.dt, m.order
    W = np.zeros((len(m.w), len(tuples)))
    for k, v in enumerate(m.e):
        add = lambda tup, x: W[k].__setitem__(at[tuple(sorted(tup))], W[k][at[tuple(sorted(tup))]] + x)  # noqa: E731
        w = [1.0] + [float(x) for x in v]
        ax = range(1, m.d + 1)
        if m.full:
            add((), m.w[k])
            for a in range(m.d + 1):
                if P >= 3:
                    add((a,), -0.5 * dt * m.w[k] * w[a])
                for b in range(m.d + 1):
                    for g in range(m.d + 1):
                        if P >= 4:
                            add((a, b, g), m.w[k] * dt ** 3 / 24 * w[a] * w[b] * w[g])
            continue
        wp, wm = m.w[k] + m.w[m.bar[k]], m.w[k] - m.w[m.bar[k]]
        add((), wp)
        if P >= 2:
            add((0,), 0.5 * dt * wp)
        if P >= 3:
            for a in ax:
                add((0, a), -wm * dt ** 2 / 4 * w[a])
                for b in ax:
                    add((a, b), -wp * dt ** 2 / 8 * w[a] * w[b])
        if P >= 4:
            add((0, 0, 0), -wp * dt ** 3 / 24)
            for a in ax:
                add((0, 0, a), -wm * dt ** 3 / 8 * w[a])
                for b in ax:
                    add((0, a, b), -wp * dt ** 3 / 16 * w[a] * w[b])
    return torch.from_numpy(W).to(DEVICE)


def exact(case, seed):
    c, v = dict(case), _inputs(case, seed)
    if c["kind"] == "map":
        return _exact_map(c, v["sig"])
    m, R = _Plain(c), c.get("R", 0.0)
    if c["kind"] in ("run", "series"):
        Rf = v["R"].reshape(m.shape) if c["kind"] == "run" and v["R"] is not None else R
        fs = m.init(v["phi0"], v.get("grad"), Rf)
        if c["kind"] == "run":
            for _ in range(c["steps"]):
                fs = m.collide(m.pull(fs), Rf)
            return {"phi": (sum(fs) - m.dt * Rf).reshape(-1)}
        seen = []
        for _ in range(c["points"]):
            for _ in range(c["every"]):
                f = m.pull(fs)
                fs = m.collide(f, Rf)
            phi = sum(fs)
            seen.append([phi.sum().item(), sum((f[k] ** 2).sum().item() / (2 * m.w[k]) for k in range(len(f))), phi.abs().max().item()])
        seen = np.array(seen)
        return {"mass": seen[:, 0], "entropy": seen[:, 1], "max": seen[:, 2], "nonfinite": None, "phi": phi.reshape(-1)}
    if c["kind"] == "box":
        axes, terms = _axes(c), v["terms"]
        sines = c["data"] == "sines"
        # one grid of cos and sin per exponential; a field is then a sum of them
        cs = [(torch.cos(z), torch.sin(z)) for z in (_phase(axes, k) for _, k, _ in terms)]

        def field(t, op):
            ws = [C * np.exp(mu * t) * op(np.asarray(k), mu) for C, k, mu in terms]
            return sum(w.real * a - w.imag * b for w, (a, b) in zip(ws, cs))

        def unknown(q, t):
            v = field(t, lambda k, mu: m.factor(q, k, mu)) + m.source_part(q) * source(t)
            if m.full:  # and the part R t of the solution
                return v + m.w[q] * (R * t - (0.5 * m.dt * R if m.order >= 3 else 0.0))
            return v + (m.w[q] + m.w[m.bar[q]]) * (R * t + (0.5 * m.dt * R if m.order >= 2 else 0.0))

        source = lambda t: field(t, lambda k, mu: mu + 1j * np.dot(k, m.u)) if sines else R  # noqa: E731
        fs = m.init(v["phi0"], v["grad"], source(0.0))
        for n in range(c["steps"]):
            t = (n + 1 if m.full else n) * m.dt
            data = [None] + [unknown(q, t) for q in range(1, len(m.w))]
            fs = m.collide(m.with_data(fs, data), source((n + 1) * m.dt))
        return {"phi": (sum(fs) - m.dt * source(c["steps"] * m.dt)).reshape(-1)}
    if c["kind"] == "grad":
        phi0, Rf = v["phi0"].requires_grad_(), v["R"].requires_grad_()
        fs = m.init(phi0, None, Rf.reshape(m.shape))
        for _ in range(c["steps"]):
            fs = m.collide(m.pull(fs), Rf.reshape(m.shape))
        r = (sum(fs) - m.dt * Rf.reshape(m.shape)).reshape(-1) - v["target"]
        loss = 0.5 * torch.dot(r, r)
        g = torch.autograd.grad(loss, (phi0, Rf))
        return {"loss": loss.detach(), "dphi0": g[0], "dR": g[1]}
    # boxgrad: the records are linear in the jets; their places in the box by (node, link)
    nodes, W = _nodes(m), _jet_rows(m)
    lo = _box(c)[2]
    at = np.array([a for a, _ in nodes])
    coord = np.stack([(at // math.prod(m.n[:i])) % m.n[i] for i in range(m.d)], 1)
    node_x = lo + m.dx * (coord + (0.5 if m.half else 0.0))
    if m.full:
        points, rows = node_x, [(a, k, j) for j, (a, ks) in enumerate(nodes) for k in ks]
    else:
        rows, points, j = [], [], 0
        for q, (a, ks) in enumerate(nodes):
            for k in ks:
                rows.append((a, k, j))
                points.append(node_x[q] - 0.5 * m.dx * m.e[k])
                j += 1
        points = np.array(points)
    places = [([a for a, kk, _ in rows if kk == k], [j for _, kk, j in rows if kk == k]) for k in range(len(m.w))]
    jets = _jets(c, v["terms"], points, m.dt if m.full else 0.0, m.dt).requires_grad_()
    phi0, grad = v["phi0"].requires_grad_(), v["grad"].requires_grad_()
    fs = m.init(phi0, grad, R)
    size = phi0.numel()
    for n in range(c["steps"]):
        data = [None]
        for k in range(1, len(m.w)):
            a, j = (torch.tensor(q, dtype=torch.long, device=DEVICE) for q in places[k])
            rec = jets[n][j] @ W[k] + m.source_part(k) * R
            data.append(torch.zeros(size, dtype=torch.float64, device=DEVICE).index_put((a,), rec).reshape(m.shape))
        fs = m.collide(m.with_data(fs, data), R)
    phi = (sum(fs) - m.dt * R).reshape(-1)
    cot = torch.from_numpy(_rng(seed, 5).standard_normal(size)).to(DEVICE)
    g = torch.autograd.grad(phi, (phi0, grad, jets), cot)
    return {"phi": phi.detach(), "dphi0": g[0], "dgrad": g[1], "djets": g[2]}
