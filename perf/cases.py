"""The work that users of this package have it do, as measurable cases.

A pass of a case is what a program does between having new data and using the
result: it hands the state to the solver it keeps (`set_state`), advances it,
and reads the fields and the energy, mass and gradient sums back.  Every pass
starts from the same state, so it costs the same however often it is repeated.

Kinds of case ("kind"):
  run       one PFCSolver (any precision, any initial iterate, constant or
            variable mobility)
  ensemble  runs of up to three grid sizes, one PFCBatch per size, advanced
            together by one PFCGroup
  adjoint   adjoint.rollout, forward and backward, as a training loop calls it

Grids are cubes of n = 2^k m cells a side (m = 1, 3, 5, 7), 16^3 to 256^3;
boxes, time steps, tolerances and multigrid settings are those of the
package's workloads (smooth mode, noise start, growth, polycrystal, ensemble,
gradient) and the library's defaults.
"""

import math

import numpy as np
import torch

from paper_1611_06288_gb300 import adjoint, binding
from paper_1611_06288_gb300.solver import PFCBatch, PFCGroup, PFCSolver

# Multigrid settings of the package's workloads, as a program passes them.
STIFF = {"nu1": 0, "nu2": 1, "inner_cycles": 2, "jacobi_factor": 4, "coarse_sweeps": 2}
SOFT = {"nu1": 1, "nu2": 2, "inner_cycles": 3, "jacobi_factor": 3, "coarse_sweeps": 2}
SMALL = {"nu1": 1, "nu2": 2, "inner_cycles": 2, "jacobi_factor": 3, "coarse_sweeps": 2}
FP64 = {"nu1": 0, "nu2": 1, "jacobi_factor": 2}
SETTINGS = ("nu1", "nu2", "inner_cycles", "jacobi_factor", "coarse_sweeps", "cluster_tail",
            "guess", "coarsest")


def _run(name, field, n, L, eps, dt, steps, tol=1e-9, precision="mixed", each=False, prev=False,
         m2=0.0, **settings):
    """A "run" case: `steps` steps from one field of the kind `field`; each:
    the sums are read after every step (else after the last); prev: the state
    comes with the field of the step before; m2: mobility 1 + m2 phi^2."""
    return {"name": name, "kind": "run", "field": field, "n": n, "L": L, "eps": eps, "dt": dt,
            "steps": steps, "tol": tol, "precision": precision, "each": each, "prev": prev,
            "m2": m2, **settings}


def listed():
    return [
        # the smallest call: the 16^3 noise start with the library's own cycle,
        # 10 steps; latency of launches and of the coarse levels
        _run("noise16", "noise", 16, 32.0, 0.025, 0.01, 10, tol=1e-10),
        # a program that owns the fields and has single steps taken from them
        # (coupling, restarts): one step from phi^k, phi^{k-1} at 64^3
        _run("restart64", "smooth", 64, 32.0, 0.025, 0.0125, 1, prev=True, each=True, **STIFF,
             guess="extrapolate_all", cluster_tail=2),
        # the package's headline: a smooth 128^3 run followed step by step
        _run("smooth128", "smooth", 128, 32.0, 0.025, 0.0125, 20, each=True, **STIFF,
             guess="extrapolate_all", cluster_tail=2),
        # the same run on the largest grid
        _run("smooth256", "smooth", 256, 32.0, 0.025, 0.0125, 8, each=True, **STIFF,
             guess="extrapolate_all"),
        # growth of a polycrystal from a nearly uniform field on a grid that
        # is no power of two, advanced without looking at every step
        _run("growth96", "start", 96, 64.0, 0.25, 0.01, 10, **SOFT, guess="extrapolate_all"),
        # crystal seeds in a liquid, the package's largest workload
        _run("polycrystal256", "crystal", 256, 256 * math.pi / 4, 0.25, 0.1, 3, each=True, **SOFT,
             guess="extrapolate_all"),
        # parameter study: 96 runs of uneven sizes advanced together
        {"name": "ensemble96", "kind": "ensemble", "m32": 28, "m48": 26, "m64": 42, "L": 32.0,
         "dt": 0.05, "steps": 5, "tol": 1e-9},
        # PFCSolver as it comes: double precision, V(2,2), 32^3
        _run("default32", "smooth", 32, 32.0, 0.025, 0.0125, 10, precision="fp64"),
        # double precision with its tuned cycle at the headline's size
        _run("fp64_128", "smooth", 128, 32.0, 0.025, 0.0125, 6, precision="fp64", each=True,
             **FP64, guess="extrapolate_all"),
        # the double-float outer loop at the headline's size
        _run("df128", "smooth", 128, 32.0, 0.025, 0.0125, 10, precision="mixed_df", each=True,
             **STIFF, cluster_tail=2),
        # concentration-dependent mobility 1 + phi^2/2, no power of two
        _run("mobility80", "start", 80, 64.0, 0.25, 0.01, 10, m2=0.5, **SOFT, coarsest=10),
        # gradient of a loss through 20 steps, as fitting eps and phi^0 does
        {"name": "adjoint64", "kind": "adjoint", "n": 64, "L": 32.0, "eps": 0.15, "dt": 0.05,
         "steps": 20, "every": 10},
    ]


def _log_size(rng, lo, hi, odd=(1, 3, 5, 7)):
    """A grid size 2^k m in [lo, hi], near a point drawn over the logarithm."""
    sizes = [m << k for m in odd for k in range(2, 9) if lo <= m << k <= hi]
    at = rng.uniform(math.log(lo), math.log(hi))
    return min(sizes, key=lambda n: abs(math.log(n) - at))


def _coarsest(n):
    """The last even size that halving n reaches (the library's `coarsest`)."""
    while n % 4 == 0:
        n //= 2
    return n


def draw(rng):
    kind = rng.choice(["smooth", "smooth", "growth", "growth", "polycrystal", "noise", "fp64",
                       "fp64", "df", "mobility", "ensemble", "adjoint"])
    each = rng.random() < 0.5
    eps = round(rng.uniform(0.02, 0.3), 4)

    def steps(n, most=12):
        return max(2, min(most, rng.randint(4, 12), int(3 * 256 ** 3 / n ** 3)))

    def case(*args, **kw):
        c = _run("", *args, **kw)
        del c["name"]
        return c

    if kind == "ensemble":
        return {"kind": "ensemble", "m32": rng.randint(0, 24), "m48": rng.randint(1, 16),
                "m64": rng.randint(0, 24), "L": 32.0, "dt": round(rng.uniform(0.02, 0.05), 4),
                "steps": rng.randint(1, 5), "tol": 1e-9}
    if kind == "adjoint":
        n = _log_size(rng, 16, 64, odd=(1, 3))
        s = rng.randint(4, 12)
        return {"kind": "adjoint", "n": n, "L": 32.0, "eps": eps,
                "dt": round(rng.uniform(0.02, 0.05), 4), "steps": s, "every": rng.randint(2, s)}
    if kind == "noise":
        n = _log_size(rng, 16, 32)
        return case("noise", n, 2.0 * n, eps, 0.01, steps(n), tol=1e-10, each=each,
                    coarsest=_coarsest(n))
    if kind == "growth":
        n = _log_size(rng, 32, 192)
        return case("start", n, n / 2.0, eps, round(rng.uniform(0.005, 0.02), 4), steps(n),
                    each=each, **SOFT, guess=rng.choice(["extrapolate_all", "previous"]),
                    coarsest=_coarsest(n))
    if kind == "polycrystal":
        n = _log_size(rng, 48, 256)
        return case("crystal", n, n * math.pi / 4, 0.25, 0.1, min(3, steps(n)), each=each, **SOFT,
                    guess=rng.choice(["extrapolate_all", "previous"]), coarsest=_coarsest(n))
    if kind == "mobility":
        n = _log_size(rng, 32, 128)
        return case("start", n, n / 2.0, eps, 0.01, steps(n), each=each,
                    m2=round(rng.uniform(0.1, 0.8), 3), **SOFT, coarsest=_coarsest(n))
    # the smooth mode on the box of side 32 in the three precisions
    n = _log_size(rng, 24, 256 if kind == "smooth" else 128, odd=(1, 3) if kind == "fp64" else
                  (1, 3, 5, 7))
    dt = round(rng.uniform(0.008, 0.0125), 5)
    if kind == "fp64":
        tuned = rng.random() < 0.5
        kw = dict(FP64, guess="extrapolate_all") if tuned else {}
        return case("smooth", n, 32.0, eps, dt, steps(n, 6), precision="fp64", each=each, **kw,
                    coarsest=_coarsest(n))
    kw = dict(STIFF if n >= 64 else SMALL, coarsest=_coarsest(n))
    if n >= 64 and n < 256 and n % 8 == 0:
        kw["cluster_tail"] = 2
    if kind == "df":
        return case("smooth", n, 32.0, eps, dt, steps(n), precision="mixed_df", each=each, **kw)
    return case("smooth", n, 32.0, eps, dt, steps(n), each=each,
                guess=rng.choice(["extrapolate_all", "previous"]), prev=rng.random() < 0.3, **kw)


# ---------------------------------------------------------------------------
# Inputs, drawn on the GPU from the seed
# ---------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, shape):
    """U(-1, 1) per cell."""
    return 2.0 * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 1.0


def _field(kind, n, L, seed):
    g = _generator(seed)
    h = L / n
    x = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * h
    if kind == "noise":        # 0.07 + 0.07 U(-1, 1) per cell
        return 0.07 + 0.07 * _uniform(g, (n, n, n))
    if kind == "start":        # 0.2 + 0.005 U[0, 1] per cell
        return 0.2 + 0.0025 * (1.0 + _uniform(g, (n, n, n)))
    if kind == "smooth":       # one mode of amplitude about 0.1 in random place, on a mean
        a, b, c, d, e = (2.0 * torch.rand(5, generator=g, device="cuda",
                                          dtype=torch.float64) - 1.0).tolist()
        k = 2.0 * math.pi / L
        sx, sy, sz = (torch.sin(k * x + math.pi * p) for p in (a, b, c))
        return 0.03 + 0.01 * d + 0.1 * (1.0 + 0.1 * e) * sz[:, None, None] * sy[:, None] * sx
    # liquid at -0.25 with noise and six one-mode BCC seeds of radius 10 h in
    # random places and orientations
    r = np.random.default_rng(seed)
    phi = -0.25 + 0.01 * torch.randn((n, n, n), generator=g, device="cuda", dtype=torch.float64)
    qs = np.array([[1, 1, 0], [1, -1, 0], [1, 0, 1], [1, 0, -1], [0, 1, 1], [0, 1, -1]])
    for _ in range(6):
        cx, cy, cz = r.uniform(0.0, L, 3)
        rot, _ = np.linalg.qr(r.standard_normal((3, 3)))
        dx, dy, dz = ((x - p + 0.5 * L) % L - 0.5 * L for p in (cx, cy, cz))
        inside = (dz ** 2)[:, None, None] + (dy ** 2)[:, None] + dx ** 2 <= (10.0 * h) ** 2
        for q in (qs / math.sqrt(2.0)) @ rot.T:
            wave = torch.cos((q[2] * dz)[:, None, None] + (q[1] * dy)[:, None] + q[0] * dx)
            phi = torch.where(inside, phi + 0.3 * wave, phi)
    return phi


def _fields(case, seed):
    """(phi^k, phi^{k-1} or None) of a run."""
    phi = _field(case["field"], case["n"], case["L"], seed)
    if not case["prev"]:
        return phi, None
    mean = phi.mean()
    return phi, mean + 1.001 * (phi - mean)


def _members(case, seed):
    """{n: (eps list, phi0 of the members)}: eps ~ U[0.02, 0.3], phi0 = mean +
    0.05 U(-1, 1) with the mean ~ U[-0.3, 0.1]."""
    r, g, out = np.random.default_rng(seed), _generator(seed), {}
    for n in (32, 48, 64):
        m = case["m%d" % n]
        if m:
            mean = torch.tensor(r.uniform(-0.3, 0.1, m), device="cuda")[:, None, None, None]
            out[n] = (r.uniform(0.02, 0.3, m).tolist(), mean + 0.05 * _uniform(g, (m, n, n, n)))
    return out


def _gradient_inputs(case, seed):
    """phi^0 and the gradient of the loss with respect to the last field."""
    n, g = case["n"], _generator(seed)
    phi0 = -0.1 + 0.05 * _uniform(g, (n, n, n))
    return phi0, (case["L"] / n) ** 3 * _uniform(g, (n, n, n))


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def prepare(case, seed):
    if case["kind"] == "adjoint":
        phi0, gout = _gradient_inputs(case, seed)
        return {"case": case, "phi0": phi0.requires_grad_(True), "gout": gout,
                "eps": torch.tensor(case["eps"], dtype=torch.float64, requires_grad=True)}
    if case["kind"] == "ensemble":
        kw = dict(SOFT, tol=case["tol"], max_cycles=100, guess="extrapolate_all")
        members = _members(case, seed)
        batches = {n: PFCBatch(n, case["L"], eps, case["dt"], phi0, **kw)
                   for n, (eps, phi0) in members.items()}
        return {"case": case, "batches": batches, "group": PFCGroup(list(batches.values())),
                "phi0": {n: phi0 for n, (_, phi0) in members.items()}}
    phi, prev = _fields(case, seed)
    kw = {k: case[k] for k in SETTINGS if k in case}
    if case["m2"]:
        kw["mobility"] = (1.0, case["m2"])
    solver = PFCSolver(case["n"], case["L"], case["eps"], case["dt"], phi, prev,
                       precision=case["precision"], tol=case["tol"], max_cycles=100,
                       step_diagnostics=case["each"], **kw)
    return {"case": case, "solver": solver, "phi": phi, "prev": prev}


def _sums(d):
    return [d["energy"], d["modified_energy"], d["mass"], d["grad_sq"]]


def run(state):
    case = state["case"]
    if case["kind"] == "adjoint":
        phi0, eps = state["phi0"], state["eps"]
        phi0.grad = eps.grad = None
        phi = adjoint.rollout(phi0, eps, case["n"], case["L"], case["dt"], case["steps"],
                              every=case["every"])
        phi.backward(state["gout"])
        return {"phi": phi.detach(), "phi0_grad": phi0.grad, "eps_grad": eps.grad}
    if case["kind"] == "ensemble":
        batches = state["batches"]
        for n, b in batches.items():
            binding.pfc_set_state(b.ctx, state["phi0"][n])
        state["group"].step(case["steps"])
        return {str(n): {"phi": b.phi(), "mu": b.mu(), "omega": b.omega(),
                         "sums": np.array([_sums(d) for d in b.diagnostics()])}
                for n, b in batches.items()}
    s, sums = state["solver"], []
    s.set_state(state["phi"], state["prev"])
    if case["each"]:
        for _ in range(case["steps"]):
            s.step(1)
            sums.append(_sums(s.diagnostics()))
    else:
        s.step(case["steps"])
        sums.append(_sums(s.diagnostics()))
    return {"phi": s.phi(), "mu": s.mu(), "omega": s.omega(), "sums": np.array(sums)}


def work(case):
    """What a step cannot do without: phi^k, phi^{k-1}, mu and omega read, the
    new phi, mu and omega written, and one evaluation of the three rows of the
    scheme (Eqs. 5.4-5.10: five Laplacians and the cubic term, 60 operations a
    cell).  An adjoint pass takes each step twice forwards (the backward pass
    recomputes it) and once backwards."""
    if case["kind"] == "ensemble":
        cells = sum(case["m%d" % n] * n ** 3 for n in (32, 48, 64))
    else:
        cells = case["n"] ** 3
    steps = case["steps"] * (3 if case["kind"] == "adjoint" else 1)
    return {"bytes": 56.0 * cells * steps, "flops": 60.0 * cells * steps}


# ---------------------------------------------------------------------------
# The same numbers in 64 bits by plain torch: every step of the scheme is
# solved for phi (mu and omega eliminated) by residual correction with a
# constant-coefficient operator inverted by FFT, to rounding.
# ---------------------------------------------------------------------------

AXES = (-1, -2, -3)


def _lap(v, h):
    s = -6.0 * v
    for a in AXES:
        s += torch.roll(v, 1, a)
        s += torch.roll(v, -1, a)
    return s / (h * h)


def _inverse(n, h, c1, dt, q, m):
    """x -> (I - dt m Lap (q + c1 + Lap^2 / 2))^{-1} x on fields of n^3 cells."""
    k = torch.arange(n, device="cuda", dtype=torch.float64) * (math.pi / n)
    s = -4.0 / (h * h) * torch.sin(k) ** 2
    lam = s[:, None, None] + s[:, None] + s[: n // 2 + 1]
    sym = 1.0 - dt * m * lam * (q + c1 + 0.5 * lam * lam)

    def inv(x):
        return torch.fft.irfftn(torch.fft.rfftn(x, dim=(-3, -2, -1)) / sym, s=(n, n, n),
                                dim=(-3, -2, -1))
    return inv


def _solve(x, residual, inv):
    """x with residual(x) = 0, by x += inv(residual(x)) until it stalls."""
    last = math.inf
    for it in range(200):
        dx = inv(residual(x))
        x = x + dx
        size, top = dx.abs().max().item(), x.abs().max().item()
        if size <= 1e-16 * top or (size <= 1e-13 * top and size > 0.7 * last):
            break
        last = size
    return x


def _slope(a, b):
    return 0.75 * a * a + 0.5 * a * b + 0.25 * b * b


def _middle(v):
    """The middle of the values' range, per member."""
    d = (-3, -2, -1)
    return 0.5 * (v.amax(dim=d, keepdim=True) + v.amin(dim=d, keepdim=True))


def _advance(b, c, n, h, c1, dt, m2=0.0):
    """phi^{k+1}, mu, omega from b = phi^k, c = phi^{k-1}; c1 = (1 - eps)/2 (a
    number, or one per member)."""
    lb = _lap(b, h)
    s2 = c1 * b + 3.0 * lb - _lap(c, h)
    star = 1.5 * b - 0.5 * c

    def others(p):
        om = 0.5 * (lb + _lap(p, h))
        mu = s2 + 0.25 * (p + b) * (p * p + b * b) + c1 * p + _lap(om, h)
        return mu, om

    def flux(mu):
        if not m2:
            return _lap(mu, h)
        out = torch.zeros_like(mu)
        for a in AXES:
            face = 0.5 * (star + torch.roll(star, -1, a))
            f = (1.0 + m2 * face * face) * (torch.roll(mu, -1, a) - mu)
            out += f - torch.roll(f, 1, a)
        return out / (h * h)

    m = 1.0 + m2 * _middle(star * star)
    inv = _inverse(n, h, c1, dt, _middle(_slope(b, b)), m)
    p = _solve(2.0 * b - c, lambda v: b + dt * flux(others(v)[0]) - v, inv)
    return (p, *others(p))


def _energy_sums(a, b, h, c1):
    """Energy, modified energy, mass and squared gradient per member."""
    d = (-3, -2, -1)

    def grad_sq(v):
        return sum(((torch.roll(v, -1, x) - v) ** 2).sum(dim=d) for x in AXES) * h

    c1 = c1.reshape(-1) if torch.is_tensor(c1) else c1
    h3, g = h ** 3, grad_sq(a)
    energy = (0.25 * h3 * (a ** 4).sum(dim=d) + c1 * h3 * (a * a).sum(dim=d) - g
              + 0.5 * h3 * (_lap(a, h) ** 2).sum(dim=d))
    return torch.stack([energy, energy + 0.5 * grad_sq(a - b), h3 * a.sum(dim=d), g], dim=-1)


def _exact_steps(b, c, n, L, c1, dt, steps, m2=0.0, each=True):
    h, sums = L / n, []
    for _ in range(steps):
        p, mu, om = _advance(b, c, n, h, c1, dt, m2)
        b, c = p, b
        sums.append(_energy_sums(b, c, h, c1))
    return {"phi": b, "mu": mu, "omega": om,
            "sums": torch.stack(sums) if each else torch.stack(sums[-1:])}


def _exact_adjoint(case, seed):
    n, dt = case["n"], case["dt"]
    h, c1 = case["L"] / n, 0.5 * (1.0 - case["eps"])
    phi0, g = _gradient_inputs(case, seed)
    path = [phi0, phi0]                       # phi^{-1} := phi^0
    for _ in range(case["steps"]):
        path.append(_advance(path[-1], path[-2], n, h, c1, dt)[0])
    gc, geps = torch.zeros_like(g), 0.0
    # step k maps (phi^k, phi^{k-1}) to phi^{k+1} with G(phi^{k+1}; phi^k,
    # phi^{k-1}) = 0, so dL/dphi^k and dL/dphi^{k-1} gain -G_b^T w and
    # -G_c^T w with G_a^T w = dL/dphi^{k+1}
    for k in range(case["steps"] - 1, -1, -1):
        a, b = path[k + 2], path[k + 1]
        inv = _inverse(n, h, c1, dt, _middle(_slope(a, b)), 1.0)
        slope = _slope(a, b) + c1

        def rest(w):
            l1 = _lap(w, h)
            return g - w + dt * (slope * l1 + 0.5 * _lap(_lap(l1, h), h))

        w = _solve(inv(g), rest, inv)
        l1 = _lap(w, h)
        l2 = _lap(l1, h)
        fb = 0.25 * (a * a + 2.0 * a * b + 3.0 * b * b)
        geps -= 0.5 * dt * (l1 * (a + b)).sum()
        gb = gc + w + dt * ((fb + c1) * l1 + 3.0 * l2 + 0.5 * _lap(l2, h))
        g, gc = gb, -dt * l2
    return {"phi": path[-1], "phi0_grad": g + gc, "eps_grad": geps}


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    if case["kind"] == "ensemble":
        out = {}
        for n, (eps, phi0) in _members(case, seed).items():
            c1 = 0.5 * (1.0 - torch.tensor(eps, device="cuda")[:, None, None, None])
            r = _exact_steps(phi0, phi0, n, case["L"], c1.double(), case["dt"], case["steps"])
            out[str(n)] = dict(r, sums=r["sums"][-1])
        return out
    phi, prev = _fields(case, seed)
    return _exact_steps(phi, phi if prev is None else prev, case["n"], case["L"],
                        0.5 * (1.0 - case["eps"]), case["dt"], case["steps"], case["m2"],
                        case["each"])
