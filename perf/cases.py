"""Performance cases of the MMVM library: what its users run, through the
public Python binding of the C ABI.

A case is one pass of a user's program: load a state that is already on the
device (or on the host, where the call takes host arrays), run the solver,
take the state out.  The kinds:

* ``steps``: classic RK4 steps of one simulation (``mmvm_set_state_device``,
  ``mmvm_step``, ``mmvm_get_state_device``), the benchmark's own unit of work;
* ``rhs``: one right-hand side for a program with its own integrator
  (``mmvm_set_state_device``, ``mmvm_rhs_device``);
* ``adaptive``: Dormand-Prince integration at the tolerance of the paper's
  experiments (``mmvm_integrate``);
* ``served``: a burst of independent simulations through the
  continuous-batching server (``Server.submit`` / ``wait``);
* ``vorticity``: the field of a state on a grid of points
  (``mmvm_vorticity``).

The states are the repository's workloads, drawn here from the seed: a
single Lamb-Oseen core with a quadrupole, particles in a disk, two co-rotating
patches, the coarse-grid tripole.
"""
import math

import numpy as np
import torch

import paper_1010_2475_gb300 as mm

DISK_R, DISK_SIGMA = 10.0, 0.5        # random disk: radius and core size
PATCH_R, PATCH_SEP = 2.0, 6.0         # two patches: radius and separation


def listed():
    return [
        # one vortex core relaxing towards axisymmetry: the paper's single-particle
        # experiments, thousands of tiny right-hand sides one after another
        {"name": "single_m10", "kind": "steps", "state": "single", "n": 1, "order": 10,
         "precision": "fp64", "sigma": 1.0, "dt": 0.01, "steps": 100},
        # the high-order limit of one core: a single right-hand side
        {"name": "single_m60", "kind": "rhs", "state": "single", "n": 1, "order": 60,
         "precision": "fp64", "sigma": 1.0},
        # the coarse-grid tripole of the paper, adaptive steps at 1e-8: small n, host
        # decisions between steps
        {"name": "tripole_adaptive", "kind": "adaptive", "state": "tripole", "n": 36, "order": 2,
         "precision": "fp64", "sigma": 1.0, "t_end": 0.5},
        # a plot of a state: every particle seen from every grid point
        {"name": "vorticity_n4096", "kind": "vorticity", "state": "disk", "n": 4096, "order": 4,
         "precision": "fp64", "sigma": 0.5, "grid": 121},
        # the plain FP64 form, the accuracy reference of every study
        {"name": "patches_2048_fp64", "kind": "rhs", "state": "patches", "n": 2048, "order": 6,
         "precision": "fp64", "sigma": 0.1},
        # a small low-order simulation (about the median of the served sizes)
        {"name": "disk_700_m2", "kind": "steps", "state": "disk", "n": 700, "order": 2,
         "precision": "mixed", "sigma": 0.5, "dt": 0.01, "steps": 4},
        # the N = 4096, M = 4 random disk
        {"name": "disk_4096_m4", "kind": "steps", "state": "disk", "n": 4096, "order": 4,
         "precision": "mixed", "sigma": 0.5, "dt": 0.01, "steps": 1},
        # the highest order with many particles, a ragged size
        {"name": "disk_2011_m8", "kind": "steps", "state": "disk", "n": 2011, "order": 8,
         "precision": "mixed", "sigma": 0.5, "dt": 0.01, "steps": 1},
        # low order, larger n at the density of 8192 particles in the disk (the largest served)
        {"name": "disk_30011_m2", "kind": "steps", "state": "disk", "n": 30011, "order": 2,
         "precision": "mixed", "sigma": 0.5, "dt": 0.01, "steps": 1},
        # two patches at a ragged size of a parameter study
        {"name": "patches_5003_m6", "kind": "steps", "state": "patches", "n": 5003, "order": 6,
         "precision": "mixed", "sigma": 0.1, "dt": 0.05, "steps": 1},
        # the benchmark workload
        {"name": "patches_65536_m6", "kind": "steps", "state": "patches", "n": 65536, "order": 6,
         "precision": "mixed", "sigma": 0.1, "dt": 0.05, "steps": 1},
        # a burst of the served stream: sizes log-uniform in [64, 8192], orders 2, 4, 8
        {"name": "served_burst", "kind": "served", "requests": 16, "n_min": 64, "n_max": 8192,
         "precision": "mixed", "sigma": 0.5, "dt": 0.01, "steps": 4},
    ]


def _log_int(rng, lo, hi):
    """Log-uniform integer, odd half of the time."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, n | 1) if rng.random() < 0.5 else n


def draw(rng):
    pick = rng.random()
    if pick < 0.12:  # one particle, through the moment tables (to order 16)
        return {"kind": "steps", "state": "single", "n": 1, "order": rng.randint(2, 16),
                "precision": "fp64", "sigma": rng.choice([0.5, 1.0, 2.0]), "dt": 0.01,
                "steps": rng.randint(20, 100)}
    if pick < 0.20:  # one particle, separable self term
        return {"kind": "rhs", "state": "single", "n": 1, "order": rng.randint(17, 60),
                "precision": "fp64", "sigma": 1.0}
    if pick < 0.28:
        return {"kind": "adaptive", "state": "tripole", "n": rng.choice([16, 25, 36, 49]),
                "order": rng.randint(0, 4), "precision": "fp64", "sigma": 1.0,
                "t_end": rng.choice([0.25, 0.5])}
    if pick < 0.36:
        return {"kind": "vorticity", "state": "disk", "n": _log_int(rng, 36, 4096),
                "order": rng.randint(0, 4), "precision": "fp64", "sigma": 0.5,
                "grid": rng.randint(32, 121)}
    if pick < 0.48:
        return {"kind": "rhs", "state": rng.choice(["disk", "patches"]),
                "n": _log_int(rng, 64, 2048), "order": rng.randint(0, 8), "precision": "fp64",
                "sigma": 0.5 if rng.random() < 0.5 else 0.1}
    if pick < 0.70:
        return {"kind": "steps", "state": "disk", "n": _log_int(rng, 64, 8192),
                "order": rng.choice([2, 4, 8]), "precision": "mixed", "sigma": 0.5,
                "dt": 0.01, "steps": rng.randint(1, 2)}
    if pick < 0.94:
        n = _log_int(rng, 2048, 65536)
        return {"kind": "steps", "state": "patches", "n": n, "order": rng.randint(0, 8 if n < 16384 else 6),
                "precision": "mixed", "sigma": 0.1, "dt": 0.05, "steps": 1}
    return {"kind": "served", "requests": rng.randint(4, 16), "n_min": 64,
            "n_max": rng.choice([1024, 4096, 8192]), "precision": "mixed", "sigma": 0.5,
            "dt": 0.01, "steps": rng.randint(2, 4)}


# ------------------------------------------------------------------ states
def _n_moments(order):
    return (order + 1) * (order + 2) // 2


def _col(k1, k2):
    return (k1 + k2) * (k1 + k2 + 1) // 2 + k2


def _weights(order, lam):
    """w_k = 2^|k| k1! k2! / lam^(2|k|), by moment column."""
    return np.array([2.0 ** s * math.factorial(s - k2) * math.factorial(k2) / lam ** (2 * s)
                     for s in range(order + 1) for k2 in range(s + 1)])


def _single(order, sigma, seed):
    rng = np.random.default_rng(seed)
    m = np.zeros((1, _n_moments(order)))
    m[0, 0] = 1.0
    eps = 10.0 ** rng.uniform(-2.0, -1.0) * sigma ** 2
    m[0, _col(2, 0)], m[0, _col(0, 2)], m[0, _col(1, 1)] = eps, -eps, 2.0 * eps
    return rng.normal(size=(1, 2)), m, 1.0 / rng.uniform(500.0, 5000.0)


def _disk(n, order, sigma, seed):
    """Uniform in a disk of radius 10 (larger above 8192 particles, at their
    density), circulations N(0, 1) with the mean removed, moments of order >= 2
    1 % of the circulation in the weighted norm."""
    rng = np.random.default_rng(seed)
    r = DISK_R * max(1.0, math.sqrt(n / 8192.0)) * np.sqrt(rng.random(n))
    th = 2.0 * math.pi * rng.random(n)
    g = rng.standard_normal(n)
    g = np.where(np.abs(g) < 0.1, np.where(g < 0, -0.1, 0.1), g)
    g = g - g.mean() if n > 1 else g
    m = np.zeros((n, _n_moments(order)))
    m[:, 0] = g
    if order >= 2:
        m[:, 3:] = (0.01 * rng.standard_normal((n, m.shape[1] - 3)) * np.abs(g)[:, None]
                    / np.sqrt(_weights(order, sigma)[3:])[None, :])
    return np.stack([r * np.cos(th), r * np.sin(th)], 1), m, 1.0 / rng.uniform(100.0, 5000.0)


def _patches(n, order, sigma, seed):
    """Two disks of radius 2 at (+-3, 0), circulations exp(-r^2) normalised per
    patch; moments of order >= 2 as after some steps (1 % in the weighted norm)."""
    rng = np.random.default_rng(seed)
    xs, gs = [], []
    for c, cnt in ((-PATCH_SEP / 2, n // 2), (PATCH_SEP / 2, n - n // 2)):
        r = PATCH_R * np.sqrt(rng.random(cnt))
        th = 2.0 * math.pi * rng.random(cnt)
        xs.append(np.stack([c + r * np.cos(th), r * np.sin(th)], 1))
        w = np.exp(-r ** 2)
        gs.append(w / w.sum())
    g = np.concatenate(gs)
    m = np.zeros((n, _n_moments(order)))
    m[:, 0] = g
    if order >= 2:
        m[:, 3:] = (0.01 * rng.standard_normal((n, m.shape[1] - 3)) * g[:, None]
                    / np.sqrt(_weights(order, sigma)[3:])[None, :])
    return np.concatenate(xs), m, 1.0 / rng.uniform(1000.0, 4000.0)


def _tripole(n, order, sigma, seed):
    """A square grid of centres on [-1, 1]^2 sampling a perturbed Lamb-Oseen core."""
    rng = np.random.default_rng(seed)
    side = math.isqrt(n)
    q = np.linspace(-1.0, 1.0, side)
    x = np.stack([a.ravel() for a in np.meshgrid(q, q, indexing="ij")], 1)
    delta = rng.uniform(0.05, 0.25)
    r2 = (x ** 2).sum(1)
    w = np.exp(-r2 / sigma ** 2) / (math.pi * sigma ** 2)
    w = w * (1.0 + 16.0 * delta * (x[:, 0] ** 2 - x[:, 1] ** 2) / sigma ** 4)
    m = np.zeros((side * side, _n_moments(order)))
    h = 2.0 / (side - 1)
    m[:, 0] = np.where(w == 0.0, 1e-3, w) * h * h
    return x, m, 1.0 / rng.uniform(500.0, 2000.0)


def _state(case, seed):
    make = {"single": lambda: _single(case["order"], case["sigma"], seed),
            "disk": lambda: _disk(case["n"], case["order"], case["sigma"], seed),
            "patches": lambda: _patches(case["n"], case["order"], case["sigma"], seed),
            "tripole": lambda: _tripole(case["n"], case["order"], case["sigma"], seed)}
    return make[case["state"]]()


def _requests(case, seed):
    """(x, moments, order, nu) of each served request; the sizes and orders of
    a burst are those of its case, the states come from the seed."""
    sizes = np.random.default_rng(case["requests"])
    out = []
    for i in range(case["requests"]):
        u = (i + sizes.random()) / case["requests"]
        n = int(round(case["n_min"] * (case["n_max"] / case["n_min"]) ** u))
        order = (2, 4, 8)[i % 3]
        x, m, nu = _disk(n, order, case["sigma"], seed * 1000 + i)
        out.append((x, m, order, nu))
    return out


# ------------------------------------------------------------------ passes
def prepare(case, seed):
    precision = mm.MMVM_FP64 if case["precision"] == "fp64" else mm.MMVM_MIXED_FP32
    if case["kind"] == "served":
        return {"case": case, "server": mm.Server(precision), "requests": _requests(case, seed)}
    x, m, nu = _state(case, seed)
    ctx = mm.Context(case["order"], case["sigma"], nu, precision)
    s = {"case": case, "ctx": ctx}
    ctx.set_state(x, m, 0.0)
    if case["kind"] == "vorticity":
        q = np.linspace(-12.0, 12.0, case["grid"])
        s["pts"] = np.stack([a.ravel() for a in np.meshgrid(q, q, indexing="ij")], 1)
        return s
    dev = torch.device("cuda", 0)
    s["x"], s["m"] = torch.from_numpy(x).to(dev), torch.from_numpy(m).to(dev)
    s["out_x"], s["out_m"] = torch.empty_like(s["x"]), torch.empty_like(s["m"])
    torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "served":
        srv = s["server"]
        tickets = [srv.submit(x, m, order, case["sigma"], nu, case["dt"], case["steps"])
                   for x, m, order, nu in s["requests"]]
        done = [srv.wait(t) for t in tickets]
        return [(x, m) for x, m, _ in done]
    ctx = s["ctx"]
    if case["kind"] == "vorticity":
        return ctx.vorticity(s["pts"])
    h = ctx.handle
    mm.mmvm_set_state_device(h, s["x"].shape[0], s["x"].data_ptr(), s["m"].data_ptr(), 0.0)
    if case["kind"] == "rhs":
        mm.mmvm_rhs_device(h, s["out_x"].data_ptr(), s["out_m"].data_ptr())
    else:
        if case["kind"] == "steps":
            mm.mmvm_step(h, case["dt"], case["steps"])
        else:
            mm.mmvm_integrate(h, case["t_end"], h0=0.05, rtol=1e-8, atol=1e-8)
        mm.mmvm_get_state_device(h, s["out_x"].data_ptr(), s["out_m"].data_ptr())
    return s["out_x"], s["out_m"]


def work(case):
    """State read and written, and the multiply-adds of the per-particle moment
    equation: no evaluation of the pair sums, however fast, does without
    these.  (Per right-hand side: at least one multiply-add for each of the K
    moments of a particle with each of the 2M orders of the velocity jet.)"""
    if case["kind"] == "served":
        parts = [(x.shape[0], order, 4 * case["steps"]) for x, _, order, _ in _requests(case, 0)]
    else:
        rhs = {"steps": 4 * case.get("steps", 1), "rhs": 1, "adaptive": 6 * 8, "vorticity": 0}
        parts = [(case["n"], case["order"], rhs[case["kind"]])]
    nbytes = sum(2.0 * 8 * n * (2 + _n_moments(o)) for n, o, _ in parts)
    flops = sum(2.0 * n * _n_moments(o) * max(2 * o, 1) * max(r, 0) for n, o, r in parts)
    if case["kind"] == "vorticity":
        pts = case["grid"] ** 2
        nbytes = 8.0 * (case["n"] * (2 + _n_moments(case["order"])) + 3 * pts)
        flops = 2.0 * pts * _n_moments(case["order"])
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ 64-bit values
def _terms(order, sources):
    """(k, l, beta1, beta2, coefficient) of the moment equation in units
    2 lambda^2 = 1: dM_k = sum coef a_l Psi[beta] over the source columns l."""
    out = []
    cols = [(s - k2, k2) for s in range(order + 1) for k2 in range(s + 1)]
    f = math.factorial
    for k, (k1, k2) in enumerate(cols):
        for l in sources:
            l1, l2 = cols[l]
            sg = -1.0 if (k1 + k2 + l1 + l2) & 1 else 1.0
            for i in range(min(l1, k1) + 1):
                for q in range(min(l2, k2) + 1):
                    p = sg * math.comb(l1, i) * math.comb(l2, q) * 4.0 ** (i + q + 1 - k1 - k2)
                    if i <= k1 - 1:
                        out.append((k, l, k1 + l1 - 2 * i - 1, k2 + l2 - 2 * q + 1,
                                    -p / (f(k1 - i - 1) * f(k2 - q))))
                    if q <= k2 - 1:
                        out.append((k, l, k1 + l1 - 2 * i + 1, k2 + l2 - 2 * q - 1,
                                    p / (f(k1 - i) * f(k2 - q - 1))))
    return out


def _psi0(a1, a2):
    """D^(a1, a2) of the stream function of a unit Gaussian vortex at its centre."""
    if (a1 | a2) & 1 or a1 + a2 == 0:
        return 0.0
    p, q = a1 // 2, a2 // 2
    f = math.factorial
    v = f(2 * p) // f(p) * (f(2 * q) // f(q))
    return (-1.0 if (p + q) % 2 == 0 else 1.0) * v / (4.0 * math.pi * (p + q))


def _jets(b1, b2, top):
    """{(a1, a2): D^a psi} for 1 <= a1 + a2 <= top at the separations (b1, b2)."""
    x = b1 * b1 + b2 * b2
    e = torch.exp(-x)
    P = top - 1
    near = x < max(P, 1)
    xs = torch.where(near, x, torch.ones_like(x))
    term = torch.full_like(x, 1.0 / (P + 1))
    acc = term.clone()
    for k in range(1, 100):
        term = term * xs / (P + 1 + k)
        acc = acc + term
    down = [None] * (P + 1)
    down[P] = torch.exp(-xs) * acc
    for k in range(P, 0, -1):
        down[k - 1] = (xs * down[k] + torch.exp(-xs)) / k
    xf = torch.where(near, torch.full_like(x, 2.0 * P + 1.0), x)
    ints, up = [], (1.0 - torch.exp(-xf)) / xf
    for k in range(P + 1):
        if k:
            up = (k * up - torch.exp(-xf)) / xf
        ints.append(torch.where(near, down[k], up))
    h1, h2 = [torch.exp(-b1 * b1) / math.pi], [torch.exp(-b2 * b2)]
    for h, b in ((h1, b1), (h2, b2)):
        h.append(-2.0 * b * h[0])
        for k in range(1, top):
            h.append(-2.0 * b * h[k] - 2.0 * k * h[k - 1])
    zr, zi = torch.ones_like(x), torch.zeros_like(x)
    out = {}
    for n in range(1, top + 1):
        zr, zi = zr * b1 + zi * b2, zi * b1 - zr * b2  # conj(z)^n
        s = (-1.0 if (n - 1) & 1 else 1.0) / (4.0 * math.pi)
        dr, di = s * zr * ints[n - 1], s * zi * ints[n - 1]
        chi = [0.0, 0.0]
        for a in range(2, n + 1):
            chi.append(h1[a - 2] * h2[n - a] - chi[a - 2])
            w = math.comb(n, a) * 2.0 ** -n
            r = (n - a) & 3
            if r == 0:
                dr = dr - w * chi[a]
            elif r == 1:
                di = di + w * chi[a]
            elif r == 2:
                dr = dr + w * chi[a]
            else:
                di = di - w * chi[a]
        seed = ((2 * dr, 2 * di), (-2 * di, 2 * dr), (-2 * dr, -2 * di), (2 * di, -2 * dr))[n & 3]
        for a in range(n + 1):
            out[(a, n - a)] = (-1.0 if (a >> 1) & 1 else 1.0) * seed[a & 1] + chi[a]
    return out


class _Exact:
    """The moment equation of n particles in FP64, every pair summed directly."""

    def __init__(self, order, lam0, nu, n, moments):
        self.order, self.lam0, self.nu, self.n = order, lam0, nu, n
        self.cols = [(s - k2, k2) for s in range(order + 1) for k2 in range(s + 1)]
        K = len(self.cols)
        src = range(K) if order <= 16 else [l for l in range(K) if moments[0, l] != 0.0]
        t = _terms(order, src)
        self.top = 2 * order if order else 1
        self.betas = {}
        for s in range(1, self.top + 1):
            for b2 in range(s + 1):
                self.betas[(s - b2, b2)] = len(self.betas)
        self.k = torch.tensor([v[0] for v in t], dtype=torch.int64)
        self.l = torch.tensor([v[1] for v in t], dtype=torch.int64)
        self.b = torch.tensor([self.betas[v[2], v[3]] for v in t], dtype=torch.int64)
        self.c = torch.tensor([v[4] for v in t], dtype=torch.float64)
        self.src = list(src)
        self.dev = torch.device("cuda" if torch.cuda.is_available() and n > 1 else "cpu")
        if n == 1:
            self.p0 = {}
            for (a1, a2), i in self.betas.items():
                self.p0[i] = [(l, _psi0(self.cols[l][0] + a1, self.cols[l][1] + a2))
                              for l in self.src]

    def __call__(self, x, m, t):
        c = 2.0 * (self.lam0 ** 2 + 4.0 * self.nu * t)
        s = torch.tensor([c ** (-0.5 * (k1 + k2)) for k1, k2 in self.cols], dtype=torch.float64,
                         device=x.device)
        a = m * s
        psi = torch.zeros((x.shape[0], len(self.betas)), dtype=torch.float64, device=x.device)
        if self.n == 1:
            for i, ps in self.p0.items():
                psi[0, i] = sum(float(a[0, l]) * v for l, v in ps if v)
        else:
            z = x / math.sqrt(c)
            rows = max(1, int(3e6) // x.shape[0])
            for r0 in range(0, x.shape[0], rows):
                d = z[r0:r0 + rows, None, :] - z[None, :, :]
                for (a1, a2), j in _jets(d[..., 0], d[..., 1], self.top + self.order).items():
                    v = j @ a  # every moment against this derivative
                    for l, (m1, m2) in enumerate(self.cols):
                        i = self.betas.get((a1 - m1, a2 - m2))
                        if i is not None and a1 >= m1 and a2 >= m2:
                            psi[r0:r0 + rows, i] += v[:, l]
        vel = torch.zeros((x.shape[0], 2), dtype=torch.float64, device=x.device)
        if self.n > 1:
            for l, (m1, m2) in enumerate(self.cols):
                sg = -1.0 if (m1 + m2) & 1 else 1.0
                vel[:, 0] -= sg * a[:, l] * psi[:, self.betas[m1, m2 + 1]]
                vel[:, 1] += sg * a[:, l] * psi[:, self.betas[m1 + 1, m2]]
        k, l, b, w = (v.to(x.device) for v in (self.k, self.l, self.b, self.c))
        dm = torch.zeros_like(m)
        for e in range(0, len(k), 4096):
            q = slice(e, e + 4096)
            dm.index_add_(1, k[q], w[q] * a[:, l[q]] * psi[:, b[q]])
        for i, (k1, k2) in enumerate(self.cols):
            if k1:
                dm[:, i] += vel[:, 0] * a[:, _col(k1 - 1, k2)] / m[:, 0]
            if k2:
                dm[:, i] += vel[:, 1] * a[:, _col(k1, k2 - 1)] / m[:, 0]
        return vel / (math.sqrt(c) * m[:, :1]), dm / (s * c)


# nodes, stage weights and 5th minus 4th order weights of Dormand-Prince 5(4)
_DP_C = (0.0, 1 / 5, 3 / 10, 4 / 5, 8 / 9, 1.0, 1.0)
_DP_A = ((), (1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
         (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
         (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
         (35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84))
_DP_E = (35 / 384 - 5179 / 57600, 0.0, 500 / 1113 - 7571 / 16695, 125 / 192 - 393 / 640,
         -2187 / 6784 + 92097 / 339200, 11 / 84 - 187 / 2100, -1 / 40)


def _adaptive(f, x, m, t_end, h, tol):
    t, k = 0.0, [f(x, m, 0.0)]
    while t < t_end:
        last = t + h >= t_end
        h = t_end - t if last else h
        for s in range(1, 7):
            yx = x + h * sum(w * v[0] for w, v in zip(_DP_A[s], k))
            ym = m + h * sum(w * v[1] for w, v in zip(_DP_A[s], k))
            k.append(f(yx, ym, t + _DP_C[s] * h))
        err = 0.0
        for y, y5, p in ((x, yx, 0), (m, ym, 1)):
            e = (h * sum(w * v[p] for w, v in zip(_DP_E, k))).abs()
            err = max(err, float((e / (tol + tol * torch.maximum(y.abs(), y5.abs()))).max()))
        fac = 0.9 * err ** -0.2 if err > 0.0 else 5.0
        if err <= 1.0:
            x, m, t, k = yx, ym, (t_end if last else t + h), [k[6]]
            h *= min(5.0, max(0.2, fac))
        else:
            k = [k[0]]
            h *= min(1.0, max(0.2, fac))
    return x, m


def _vorticity(x, m, lam, order, pts):
    """The field at pts, particles beyond the reach of double precision included."""
    out = torch.zeros(pts.shape[0], dtype=torch.float64, device=x.device)
    rows = max(1, int(1e7) // x.shape[0])
    for r0 in range(0, pts.shape[0], rows):
        t = (pts[r0:r0 + rows, None, :] - x[None, :, :]) / lam
        g = torch.exp(-(t * t).sum(-1)) / (math.pi * lam * lam)
        h = []
        for d in range(2):
            u = t[..., d]
            p = [torch.ones_like(u), 2.0 * u]
            for q in range(1, order):
                p.append(2.0 * u * p[q] - 2.0 * q * p[q - 1])
            h.append(p)
        for s in range(order + 1):
            for k2 in range(s + 1):
                w = m[:, _col(s - k2, k2)] * (-1.0 / lam) ** s
                out[r0:r0 + rows] += (h[0][s - k2] * h[1][k2] * g) @ w
    return out


def exact(case, seed):
    if case["kind"] == "served" or (case["kind"] == "steps" and case["n"] > 1
                                    and case["n"] ** 2 * (case["order"] + 2) ** 3 * case["steps"] > 2.5e10):
        return None  # every pair in FP64 takes too long
    x, m, nu = _state(case, seed)
    n, lam0 = x.shape[0], case["sigma"]
    dev = torch.device("cuda" if torch.cuda.is_available() and n > 1 else "cpu")
    x, m = torch.from_numpy(x).to(dev), torch.from_numpy(m).to(dev)
    if case["kind"] == "vorticity":
        q = np.linspace(-12.0, 12.0, case["grid"])
        pts = np.stack([a.ravel() for a in np.meshgrid(q, q, indexing="ij")], 1)
        return _vorticity(x, m, lam0, case["order"], torch.from_numpy(pts).to(dev)).cpu().numpy()
    f = _Exact(case["order"], lam0, nu, n, m)
    if case["kind"] == "rhs":
        return f(x, m, 0.0)
    if case["kind"] == "adaptive":
        return _adaptive(f, x, m, case["t_end"], 0.05, 1e-8)
    h, t = case["dt"], 0.0
    for _ in range(case["steps"]):
        k1 = f(x, m, t)
        k2 = f(x + 0.5 * h * k1[0], m + 0.5 * h * k1[1], t + 0.5 * h)
        k3 = f(x + 0.5 * h * k2[0], m + 0.5 * h * k2[1], t + 0.5 * h)
        k4 = f(x + h * k3[0], m + h * k3[1], t + h)
        x, m = (y + h / 6.0 * (a + 2.0 * b + 2.0 * c + d)
                for y, a, b, c, d in zip((x, m), k1, k2, k3, k4))
        t += h
    return x, m
