"""Measured cases: what a user of this library has it do, through its public entry points.

Four kinds of pass, all on device-resident data:

* ``steps``     -- start a flow from its fields, advance it n time steps, take a copy of the state;
* ``ensemble``  -- the same for many independent D2Q9 domains held in one batch;
* ``gradient``  -- a rollout that keeps its states, the kinetic energy of its end, and the reverse
  sweep back to the initial populations;
* ``fields``    -- fields to populations and populations back to fields (start and output of a run).

Flows are periodic Taylor-Green vortices, the doubly periodic shear layer and random solenoidal
Fourier modes (the developed flow, where most nodes lie further from equilibrium), made on the GPU
from the seed.  ``exact`` restates the whole path in 64 bits with plain torch.
"""
import math

import torch

from paper_2203_12946_gb300 import elbm as E

DEV = "cuda"
VIEW = {"f64": torch.float64, "f32": torch.float32, "f32dev": torch.float32, "f16dev": torch.float16,
        "bf16dev": torch.bfloat16}
BYTES = {"f64": 8, "f32": 4, "f32dev": 4, "f16dev": 2, "bf16dev": 2}
SIDES = (64, 96, 128, 192, 256, 384, 512)  # of an ensemble's domains


def _steps(name, lattice, dims, storage, beta, flow, amp, n):
    return {"name": name, "kind": "steps", "lattice": lattice, "nx": dims[0], "ny": dims[1], "nz": dims[2],
            "storage": storage, "beta": beta, "flow": flow, "amp": amp, "n": n}


def _gradient(name, lattice, dims, beta, amp, n):
    return {"name": name, "kind": "gradient", "lattice": lattice, "nx": dims[0], "ny": dims[1], "nz": dims[2],
            "storage": "f32", "beta": beta, "flow": "modes", "amp": amp, "n": n}


def listed():
    return [
        # the 64^2 validation vortex: the smallest domain anybody runs, all latency
        _steps("d2_tgv64", 9, (64, 64, 1), "f32", 0.9, "tgv", 0.01, 100),
        # a small box in three dimensions (a test run, one member of a parameter scan)
        _steps("d3_tgv32", 27, (32, 32, 32), "f32", 0.999, "tgv", 0.05, 50),
        # the shear layer of the accuracy study: a state that fits the L2
        _steps("d2_shear1024", 9, (1024, 1024, 1), "f32", 0.9995, "shear", 0.04, 50),
        # the same flow at production size
        _steps("d2_shear4096", 9, (4096, 4096, 1), "f32", 0.9995, "shear", 0.04, 20),
        # odd sides, a developed flow, the storage that holds 1e-5 over long runs
        _steps("d2_modes_f32dev", 9, (1501, 997, 1), "f32dev", 0.995, "modes", 0.04, 20),
        # the benchmark flow near its start: most of a three-dimensional user's time
        _steps("d3_tgv256", 27, (256, 256, 256), "f32", 0.999, "tgv", 0.05, 20),
        # a developed flow in three dimensions on a ragged box: the longer coefficient forms
        _steps("d3_modes", 27, (203, 150, 131), "f32", 0.999, "modes", 0.02, 20),
        # half the memory for twice the box
        _steps("d3_modes_f16dev", 27, (176, 144, 160), "f16dev", 0.995, "modes", 0.03, 20),
        # many small domains of mixed sizes at once (training data for a surrogate)
        {"name": "ensemble64", "kind": "ensemble", "lattice": 9, "domains": 64, "storage": "f32", "amp": 0.03, "n": 50},
        # sensitivity of the final kinetic energy to the initial state, in two and three dimensions
        _gradient("grad_d2_256", 9, (256, 256, 1), 0.9, 0.02, 32),
        _gradient("grad_d3", 27, (60, 52, 44), 0.95, 0.02, 8),
        # fields in and fields out: restart from fields, output for analysis
        {"name": "fields_d3", "kind": "fields", "lattice": 27, "nx": 201, "ny": 160, "nz": 150, "storage": "f32",
         "beta": 0.999, "flow": "modes", "amp": 0.05},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, lattice, nodes):
    """Sides of about `nodes` nodes, aspect ratios within a factor of two, odd ones among them."""
    d = 2 if lattice == 9 else 3
    side = nodes ** (1.0 / d)
    dims = [max(8, int(round(side * _log(rng, 0.75, 1.33)))) for _ in range(d)]
    if rng.random() < 0.5:  # sides that divide well, as many users choose them
        q = 32 if d == 2 else 16
        dims = [max(q, q * round(v / q)) for v in dims]
    return (dims + [1])[:3]


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "steps", "gradient", "ensemble", "fields"])
    beta = round(rng.choice([rng.uniform(0.9, 0.99), 1.0 - _log(rng, 5e-4, 1e-2)]), 5)
    amp = round(rng.uniform(0.01, 0.05), 4)
    lattice = rng.choice([9, 27])
    if kind == "ensemble":
        return {"kind": kind, "lattice": 9, "domains": rng.randint(4, 64), "storage": rng.choice(["f32", "f32", "f32dev", "f16dev"]),
                "amp": amp, "n": rng.randint(10, 60)}
    if kind == "gradient":
        nx, ny, nz = _box(rng, lattice, _log(rng, 64 ** 2, 512 ** 2) if lattice == 9 else _log(rng, 20 ** 3, 72 ** 3))
        return {"kind": kind, "lattice": lattice, "nx": nx, "ny": ny, "nz": nz, "storage": "f32",
                "beta": round(rng.uniform(0.9, 0.99), 5), "flow": "modes", "amp": amp, "n": rng.randint(3, 12)}
    if kind == "fields":
        nx, ny, nz = _box(rng, lattice, _log(rng, 64 ** 2, 2048 ** 2))
        return {"kind": kind, "lattice": lattice, "nx": nx, "ny": ny, "nz": nz, "storage": rng.choice(["f32", "f32", "f32dev"]),
                "beta": beta, "flow": rng.choice(["tgv", "modes"]), "amp": amp}
    storage = rng.choice(["f32", "f32", "f32", "f32dev", "f16dev", "bf16dev", "f64"])
    nodes = _log(rng, 48 ** 2, 3500 ** 2) if lattice == 9 else _log(rng, 16 ** 3, 200 ** 3)
    if storage == "f64":  # the 64-bit path serves checks: small boxes
        nodes = min(nodes, _log(rng, 48 ** 2, 300 ** 2))
    nx, ny, nz = _box(rng, lattice, nodes)
    most = 0.4 * 20 * 27 * 256 ** 3 / (lattice * nx * ny * nz * (8 if storage == "f64" else 1))
    n = max(1, int(min(_log(rng, 1, 100), most)))
    flow = rng.choice(["tgv", "modes", "shear"] if lattice == 9 else ["tgv", "modes", "modes"])
    case = _steps("", lattice, (nx, ny, nz), storage, beta, flow, amp, n)
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _flow(flow, dims, amp, seed):
    """rho (N) and u (D, N) in 64 bits, nodes in the order (z, y, x)."""
    nx, ny, nz = dims
    d = 2 if nz == 1 else 3
    g = torch.Generator().manual_seed(int(seed) * 7919 + 13)
    r = lambda *s: torch.rand(*s, generator=g, dtype=torch.float64)  # noqa: E731
    x = torch.arange(nx, device=DEV, dtype=torch.float64).view(1, 1, nx) / nx
    y = torch.arange(ny, device=DEV, dtype=torch.float64).view(1, ny, 1) / ny
    z = torch.arange(nz, device=DEV, dtype=torch.float64).view(nz, 1, 1) / nz
    full = (nz, ny, nx)
    ph = [2.0 * math.pi * float(v) for v in r(3)]  # the flow's place in the box
    a = amp * (0.9 + 0.2 * float(r(1)))
    tau = 2.0 * math.pi
    if flow == "tgv":
        X, Y, Z = tau * x + ph[0], tau * y + ph[1], tau * z + ph[2]
        if d == 2:
            u = [a * torch.sin(X) * torch.cos(Y), -a * torch.cos(X) * torch.sin(Y)]
            rho = 1.0 - 0.75 * a * a * (torch.cos(2 * X) + torch.cos(2 * Y))
        else:
            u = [a * torch.sin(X) * torch.cos(Y) * torch.cos(Z), -a * torch.cos(X) * torch.sin(Y) * torch.cos(Z),
                 torch.zeros(1, 1, 1, device=DEV, dtype=torch.float64)]
            rho = 1.0 + 3.0 * a * a / 16.0 * (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0)
    elif flow == "shear":
        w, delta = 0.05, 0.05
        s = torch.remainder(y + ph[1] / tau, 1.0)
        u = [torch.where(s <= 0.5, a * torch.tanh((4 * s - 1) / w), a * torch.tanh((3 - 4 * s) / w)),
             a * delta * torch.sin(tau * (x + 0.25) + ph[0]), torch.zeros(1, 1, 1, device=DEV, dtype=torch.float64)][:d]
        rho = torch.ones(1, 1, 1, device=DEV, dtype=torch.float64)
    else:  # solenoidal Fourier modes of wavelengths down to about 24 nodes, rms speed a
        modes, u = 10, [torch.zeros(full, device=DEV, dtype=torch.float64) for _ in range(d)]
        amps = []
        for _ in range(modes):
            k = torch.tensor([math.floor(float(r(1)) * (2 * m + 1)) - m for m in (max(1, n // 24) for n in dims[:d])], dtype=torch.float64)
            if not k.any():
                k[0] = 1.0
            kk = k / torch.tensor(dims[:d], dtype=torch.float64)  # per node
            v = r(d) - 0.5
            v -= (v @ kk) / (kk @ kk) * kk
            if v.norm() < 1e-3:
                v = torch.zeros(d, dtype=torch.float64)
                v[0], v[1] = -kk[1], kk[0]
            amps.append((k, v / v.norm(), tau * float(r(1))))
        for k, v, p in amps:
            arg = tau * (k[0] * x + k[1] * y + (k[2] * z if d == 3 else 0.0)) + p
            c = torch.cos(arg) * (a * math.sqrt(2.0 / modes))
            for b in range(d):
                u[b] += float(v[b]) * c
        rho = torch.ones(1, 1, 1, device=DEV, dtype=torch.float64)
    return (rho.expand(full).reshape(-1).contiguous(),
            torch.stack([v.expand(full).reshape(-1) for v in u]).contiguous())


def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _members(case, seed):
    """Sides and betas of an ensemble's domains."""
    g = torch.Generator().manual_seed(4242 + case["domains"])  # the batch's shape belongs to the case
    sides = [SIDES[int(i)] for i in torch.randint(len(SIDES), (case["domains"],), generator=g)]
    betas = (0.9 + 0.099 * torch.rand(case["domains"], generator=g, dtype=torch.float64)).tolist()
    return sides, betas


def prepare(case, seed):
    if case["kind"] == "ensemble":
        sides, betas = _members(case, seed)
        ens = E.Ensemble(9, [(s, s, 1) for s in sides], betas, storage=case["storage"])
        fields = [_flow("modes", (s, s, 1), case["amp"], seed * 64 + k) for k, s in enumerate(sides)]
        out = torch.empty(sum(9 * s * s for s in sides), dtype=VIEW[case["storage"]], device=DEV)
        torch.cuda.synchronize()  # the batch has a stream of its own
        return {"case": case, "ens": ens, "fields": fields, "out": out}
    rho, u = _flow(case["flow"], _dims(case), case["amp"], seed)
    sim = E.Simulation(case["lattice"], _dims(case), case["beta"], storage=case["storage"],
                       cutoff=case["kind"] != "gradient")
    return {"case": case, "sim": sim, "rho": rho, "u": u}


def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        ens, out, at = state["ens"], state["out"], 0
        for k, (rho, u) in enumerate(state["fields"]):
            E.elbm_batch_init_equilibrium(ens.b, k, rho, u, E.ELBM_MEM_DEVICE)
        ens.step(case["n"])
        for k in range(len(ens.dims)):
            size = 9 * ens.nodes(k)
            E.elbm_batch_get_populations(ens.b, k, out[at:at + size], E.ELBM_MEM_DEVICE)
            at += size
        return out
    sim = state["sim"]
    sim.init_equilibrium(state["rho"], state["u"])
    if case["kind"] == "fields":
        rho, u = sim.moments()
        return {"rho": rho, "u": u}
    if case["kind"] == "gradient":
        kept = [sim.state_copy()]
        for _ in range(case["n"]):
            sim.step(1)
            kept.append(sim.state_copy())
        L, g = sim.kinetic_energy(with_grad=True)
        for t in range(case["n"] - 1, -1, -1):
            g = sim.adjoint_step(kept[t], g)
        return {"L": L, "g": g, "f": kept[-1].view(VIEW[case["storage"]]).view(sim.Q, sim.N)}
    sim.step(case["n"])
    return sim.state_copy().view(VIEW[case["storage"]]).view(sim.Q, sim.N)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Fields read once and results written once, and the arithmetic of the collisions (short power series of
    the path-length coefficients); the reverse step is counted as twice the forward one."""
    if case["kind"] == "ensemble":
        nodes, q, s, d = sum(v * v for v in _members(case, 0)[0]), 9, BYTES[case["storage"]], 2
    else:
        nodes, q, s = case["nx"] * case["ny"] * case["nz"], case["lattice"], BYTES[case["storage"]]
        d = 2 if q == 9 else 3
    fields, pops, node = 8.0 * (1 + d) * nodes, float(q) * s * nodes, 27.0 * q + 80.0 + 30.0 * (d - 2)
    if case["kind"] == "fields":
        return {"bytes": 2 * fields + 2 * pops, "flops": nodes * (6.0 * q + 60.0)}
    if case["kind"] == "gradient":  # every kept state is written and read again
        return {"bytes": fields + pops * (2 * case["n"] + 2), "flops": 3.0 * node * nodes * case["n"]}
    return {"bytes": fields + pops, "flops": node * nodes * case["n"]}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------

def _lattice(q):
    d = 2 if q == 9 else 3
    c = [[(i // 3 ** (d - 1 - a)) % 3 - 1 for a in range(d)] for i in range(q)]
    w = [math.prod(4.0 / 6.0 if v == 0 else 1.0 / 6.0 for v in ci) for ci in c]
    return d, c, w


def _equilibrium64(q, rho, u):
    d, c, _ = _lattice(q)
    ax = []
    for a in range(d):
        s = torch.sqrt(1.0 + 3.0 * u[a] * u[a])
        zz = (2.0 * u[a] + s) / (1.0 - u[a])
        ax.append({-1: (2.0 - s) / (6.0 * zz), 0: (2.0 - s) * (4.0 / 6.0), 1: (2.0 - s) * zz / 6.0})
    out = []
    for ci in c:
        v = rho
        for a in range(d):
            v = v * ax[a][ci[a]]
        out.append(v)
    return torch.stack(out)


def _moments64(q, f):
    d, c, _ = _lattice(q)
    rho = f.sum(0)
    j = [sum((ci[a] * f[i] for i, ci in enumerate(c) if ci[a]), torch.zeros_like(rho)) for a in range(d)]
    return rho, [v / rho for v in j]


def _root(a, b, c):
    return 2.0 * c / (b + torch.sqrt(b * b - 4.0 * a * c))


def _collide64(q, f, beta, cutoff):
    rho, u = _moments64(q, f)
    x = _equilibrium64(q, rho, u) / f - 1.0
    fx2 = f * x * x
    b1, c1 = 0.5 * fx2.sum(0), (2.0 * fx2 / (2.0 + x)).sum(0)
    c = (fx2 * (60.0 + x * (60.0 + 11.0 * x)) / (60.0 + x * (90.0 + x * (36.0 + 3.0 * x)))).sum(0)
    xm, xp = x.clamp(max=0.0), x.clamp(min=0.0)
    p = fx2 * xm
    s3, p = p.sum(0), p * xm
    s4, p = p.sum(0), p * xm
    s5, p = p.sum(0), p * xm
    s6 = p.sum(0)
    aL = _root(0.5 * s3, b1, c1)
    t = aL * beta * xp
    bp = (fx2 * xp * (2.0 / (4.0 + t) + 1.0 / (4.0 + 2.0 * t) + 2.0 / (4.0 + 3.0 * t))).sum(0)
    b = b1 - 2.0 / 15.0 * aL * beta * beta * bp
    hb = _root(beta * beta * s3 / 6.0, b, c) * beta
    a = beta * beta * (s3 / 6.0 - hb * s4 / 12.0 + hb * hb * s5 / 20.0 - hb ** 3 * s6 / 5.0)
    alpha = _root(a, b, c)
    if cutoff:
        alpha = torch.where(x.abs().amax(0) < 1e-3, torch.full_like(alpha, 2.0), alpha)
    amax = -1.0 / (beta * x.amin(0).clamp(max=-1e-300))
    half = 0.5 * (1.0 + amax)
    alpha = torch.where(alpha > amax, torch.where(half > amax, 0.5 * amax, half), alpha)
    return f + alpha * beta * x * f


def _step64(q, dims, f, beta, cutoff):
    d, c, _ = _lattice(q)
    shape = dims[::-1]
    pulled = [torch.roll(f[i].view(shape), [v for v in ci[::-1]], list(range(3 - d, 3))).reshape(-1) for i, ci in enumerate(c)]
    return _collide64(q, torch.stack(pulled), beta, cutoff)


def _reference64(q, storage):
    """What a deviation storage subtracts from every population."""
    d, _, w = _lattice(q)
    if storage in ("f64", "f32"):
        return None
    unit = float(torch.tensor(6.0 ** -d, dtype=torch.float32))
    return torch.tensor([round(v * 6 ** d) * unit for v in w], dtype=torch.float64, device=DEV).view(-1, 1)


def _run64(q, dims, storage, beta, rho, u, n):
    f = _equilibrium64(q, rho, u)
    for _ in range(n):
        f = _step64(q, dims, f, beta, True)
    c = _reference64(q, storage)
    return f if c is None else f - c


def exact(case, seed):
    if case["kind"] == "ensemble":
        sides, betas = _members(case, seed)
        return torch.cat([_run64(9, (s, s, 1), case["storage"], betas[k], *_flow("modes", (s, s, 1), case["amp"], seed * 64 + k), case["n"]).reshape(-1)
                          for k, s in enumerate(sides)])
    q, dims = case["lattice"], _dims(case)
    rho, u = _flow(case["flow"], dims, case["amp"], seed)
    if case["kind"] == "fields":
        return {"rho": rho, "u": u}
    if case["kind"] == "gradient":
        f0 = _equilibrium64(q, rho, u).requires_grad_(True)
        f = f0
        for _ in range(case["n"]):
            f = _step64(q, dims, f, case["beta"], False)
        r, v = _moments64(q, f)
        L = 0.5 * (r * sum(a * a for a in v)).sum()
        (g,) = torch.autograd.grad(L, f0)
        return {"L": float(L.detach()), "g": g, "f": f.detach()}
    return _run64(q, dims, case["storage"], case["beta"], rho, u, case["n"])
