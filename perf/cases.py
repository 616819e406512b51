"""What this library is measured on: the calls that a simulation program makes.

A program creates a context, loads a state, runs many steps with mpcd_step, and
reads the state (and the observables of its protocol) back every so often.  The
"run" cases do that: `steps` whole steps, then mpcd_get_state into pinned host
buffers, each pass continuing the trajectory of the last one.  The "transfer"
cases load and read a state, the "collide" cases are the allocation-free solvent
collision on tensors that the caller owns.
"""
import functools
import math

import numpy as np
import torch

from paper_2604_14307_gb300 import binding as B
from paper_2604_14307_gb300 import inputs as I

RUN = dict(kind="run", Lx=10, Ly=10, Lz=10, n_rep=1, density=5.0, radius=3.0, level=3, phi=0.0, rule="srd",
           thermostat=2, precision="p32", angular=0, steps=20, force=0.0, pairs=0, lags=0, layout="box")
COLLIDE = dict(kind="collide", Lx=16, Ly=16, Lz=16, n=20480, rule="srd", thermostat=2, step=7)


def _run(name=None, **kw):
    return {**({"name": name} if name else {}), **RUN, **kw}


def listed():
    return [
        # one 162-site colloid in a small box for a long time: the validation case, all latency
        _run("single_sphere_L10", radius=2.0, level=2, phi=0.033, thermostat=0, steps=100),
        # a mid-size MPCD-AT suspension, 221 spheres of 642 sites
        _run("suspension_L50_at", Lx=50, Ly=50, Lz=50, phi=0.2, rule="at", steps=50),
        # the headline workload: 80 M solvent particles, 8952 spheres, SRD with its thermostat
        _run("suspension_L200_srd", Lx=200, Ly=200, Lz=200, density=10.0, radius=4.0, phi=0.3, steps=60),
        # sedimentation in an elongated box with odd edges: forced bodies, balanced solvent
        _run("sedimentation_63x63x129", Lx=63, Ly=63, Lz=129, phi=0.1, thermostat=1, force=0.5, steps=50),
        # an ensemble of small boxes, one colloid each, sampled for its velocity autocorrelations
        _run("ensemble_512_spheres", n_rep=512, radius=2.0, level=2, layout="single", thermostat=0, steps=50, lags=50),
        # an ensemble of mixed spheres, dumbbells and rods in boxes of 20 to 40 cells, MPCD-AT
        _run("ensemble_48_mixed", n_rep=48, layout="mixed", rule="at", steps=20),
        # the shear-viscosity protocol on its box: 17.28 M particles, 100 exchanged pairs a step
        _run("viscosity_120x240x120", Lx=120, Ly=240, Lz=120, pairs=100, steps=40),
        # the angular-momentum-conserving rule with colloids
        _run("angular_L60", Lx=60, Ly=60, Lz=60, phi=0.1, angular=1, steps=20),
        # the plain FP64 form, with which the FP32 one is compared
        _run("suspension_L40_fp64", Lx=40, Ly=40, Lz=40, phi=0.2, thermostat=1, precision="p64", steps=4),
        # a restart file of 10 M particles and 1119 colloids in, a snapshot out
        _run("transfer_L100", kind="transfer", Lx=100, Ly=100, Lz=100, density=10.0, radius=4.0, phi=0.3),
        # one collision of a small box in a host code's loop
        dict(COLLIDE, name="collide_17x13x19", Lx=17, Ly=13, Lz=19, n=20992, thermostat=1),
        # one MPCD-AT collision of the largest kind of box that call takes
        dict(COLLIDE, name="collide_40_at", Lx=40, Ly=40, Lz=40, n=640000, rule="at", thermostat=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any box of 10 to 180 cells an edge (at most 4 M cells), any form and rule."""
    kind = rng.choice(["run", "run", "run", "ensemble", "mixed", "viscosity", "angular", "fp64", "transfer", "collide"])
    rule = rng.choice(["srd", "srd", "at"])
    thermostat = rng.choice([0, 1, 2]) if rule == "srd" else 0
    if kind == "collide":
        L = [_log_int(rng, 6, 40) for _ in range(3)]
        n = max(4, int(math.prod(L) * rng.uniform(3, 20)) // 4 * 4)
        return dict(COLLIDE, Lx=L[0], Ly=L[1], Lz=L[2], n=n, rule=rule, thermostat=thermostat, step=rng.randrange(1000))
    if kind == "ensemble":
        return _run(n_rep=_log_int(rng, 7, 700), radius=2.0, level=2, layout="single", rule=rule, thermostat=thermostat,
                    steps=rng.randrange(20, 60), lags=rng.choice([0, 20, 50]))
    if kind == "mixed":
        return _run(n_rep=_log_int(rng, 3, 60), layout="mixed", rule=rule, thermostat=thermostat,
                    steps=rng.randrange(5, 30))
    if kind == "viscosity":
        return _run(Lx=_log_int(rng, 15, 130), Ly=2 * _log_int(rng, 10, 120), Lz=_log_int(rng, 15, 130),
                    pairs=rng.choice([10, 100, 300]), rule=rule, thermostat=thermostat, steps=rng.randrange(10, 50))
    top = dict(run=180, transfer=150, angular=90, fp64=60)[kind]
    base = _log_int(rng, 14, top)
    L = [min(top, max(14, int(base * rng.uniform(0.7, 1.4)))) for _ in range(3)]
    radius, level = rng.choice([(2.0, 2), (3.0, 3), (4.0, 3)])
    case = _run(Lx=L[0], Ly=L[1], Lz=L[2], density=rng.choice([5.0, 10.0]), radius=radius, level=level,
                phi=rng.choice([0.0, 0.05, 0.2, 0.3]), rule=rule, thermostat=thermostat, steps=rng.randrange(8, 50))
    if kind == "transfer":
        case.update(kind="transfer")
    elif kind == "angular":
        case.update(angular=1, steps=rng.randrange(4, 21))
    elif kind == "fp64":
        case.update(precision="p64", steps=rng.randrange(2, 6))
    elif rng.random() < 0.3 and case["phi"] > 0:
        case.update(force=0.3)
    return case


# ------------------------------------------------------------------ inputs
def _params(case, seed):
    return I.Params(kT=1.0, dt=0.1, alpha_deg=130.0, rule=I.SRD if case["rule"] == "srd" else I.AT,
                    thermostat=case["thermostat"], precision=I.P64 if case.get("precision") == "p64" else I.P32,
                    seed=1 + seed, angular=case.get("angular", 0))


@functools.lru_cache(maxsize=8)
def _mixed_boxes(n):
    """Random sequential addition of mixed shapes, up to 6 layouts (it is slow) used in turn."""
    few = I.batched_mixed_shapes(min(n, 6), seed=5)
    return few.shapes, [(few.replicas[i % len(few.replicas)], few._placements[i % len(few.replicas)]) for i in range(n)]


def _lattice(rng, L, n, d):
    """n spheres of diameter d in random order on a cubic lattice, shifted at random as far as they stay clear."""
    n_ax = [max(1, int(a / (d + 0.2))) for a in L]
    n = min(n, math.prod(n_ax))
    while True:     # the coarsest lattice that holds them
        k = max(range(3), key=lambda a: n_ax[a] / L[a])
        if math.prod(n_ax) // n_ax[k] * (n_ax[k] - 1) < n or n_ax[k] == 1:
            break
        n_ax[k] -= 1
    step = np.array(L) / n_ax
    at = rng.permutation(math.prod(n_ax))[:n]
    ijk = np.stack(np.unravel_index(at, n_ax), axis=1)
    play = np.maximum(0.0, (step - d - 0.2) / 2)
    return ((ijk + 0.5) * step + rng.uniform(-1, 1, (n, 3)) * play) % np.array(L, dtype=float)


def _system(case, seed):
    """The system and its bodies' positions and orientations."""
    rng = np.random.default_rng([17, seed])
    prm = _params(case, seed)
    if case["layout"] == "mixed":
        shapes, boxes = _mixed_boxes(case["n_rep"])
        reps = [I.Replica(L=r.L, n_solvent=r.n_solvent, body_shapes=list(r.body_shapes), id=i)
                for i, (r, _) in enumerate(boxes)]
        return I.System(prm, shapes, reps), np.concatenate([p[0] for _, p in boxes]), \
            np.concatenate([p[1] for _, p in boxes])
    shapes = [I.sphere_shape(case["radius"], case["level"], case["density"])]
    if case["layout"] == "single":
        edges = np.random.default_rng(3).choice([12, 16, 20, 24], size=case["n_rep"])
        reps = [I.Replica(L=(int(a),) * 3, n_solvent=int(case["density"] * a ** 3), body_shapes=[0], id=i)
                for i, a in enumerate(edges)]
        R = np.repeat(edges[:, None] / 2.0, 3, axis=1)
    else:
        L = (case["Lx"], case["Ly"], case["Lz"])
        R = _lattice(rng, L, I.n_bodies_for_phi(L, case["phi"], case["radius"]), 2 * case["radius"])
        reps = [I.Replica(L=L, n_solvent=int(case["density"] * math.prod(L)), body_shapes=[0] * len(R))]
    return I.System(prm, shapes, reps), R, I.random_quaternions(rng, len(R))


def _state(case, seed, system, R, q):
    """The initial state in pinned host buffers: uniform solvent, Maxwell-Boltzmann velocities."""
    real = torch.float64 if system.params.precision == I.P64 else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng([29, seed])
    n, nb = system.n_solvent, system.n_bodies
    L = system.L_array().astype(np.float64)
    counts = torch.tensor([r.n_solvent for r in system.replicas], device="cuda")
    edges = torch.repeat_interleave(torch.tensor(L, device="cuda", dtype=real), counts, dim=0) if len(L) > 1 else \
        torch.tensor(L, device="cuda", dtype=real)
    x = torch.rand(n, 3, generator=gen, device="cuda", dtype=real) * edges
    x = torch.where(x < edges, x, torch.zeros_like(x))
    v = torch.randn(n, 3, generator=gen, device="cuda", dtype=real)
    v -= v.mean(0)
    b = {}
    for k, t in (("x", x), ("v", v)):
        b[k] = torch.empty((n, 3), dtype=real, pin_memory=True)
        b[k].copy_(t)
    del x, v, edges
    M = np.array([s.m.sum() for s in system.shapes])
    Ibar = np.array([I.shape_inertia_diag(s).mean() for s in system.shapes])
    shape = system.body_shape_array()
    body = dict(R=np.asarray(R, dtype=np.float64).reshape(nb, 3), q=np.asarray(q, dtype=np.float64).reshape(nb, 4),
                P=rng.standard_normal((nb, 3)) * np.sqrt(M[shape])[:, None],
                Lm=rng.standard_normal((nb, 3)) * np.sqrt(Ibar[shape])[:, None])
    for k, a in body.items():
        b[k] = torch.empty(a.shape, dtype=torch.float64, pin_memory=True)
        b[k].copy_(torch.from_numpy(a))
    return {k: t.numpy() for k, t in b.items()}, b


def _collide_inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, L = case["n"], (case["Lx"], case["Ly"], case["Lz"])
    x = []
    for a in L:
        t = torch.rand(n, generator=gen, device="cuda") * a
        x.append(torch.where(t < a, t, torch.zeros_like(t)))
    v = [torch.randn(n, generator=gen, device="cuda") for _ in range(3)]
    return L, x, v, torch.arange(n, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    if case["kind"] == "collide":
        L, x, v, tag = _collide_inputs(case, seed)
        return dict(case=case, prm=_params(case, seed), L=L, x=x, v=v, tag=tag, step=case["step"])
    system, R, q = _system(case, seed)
    buf, own = _state(case, seed, system, R, q)
    sim = B.Simulation(system)
    sim.set_state_buffers(buf)
    if case["force"]:
        sim.set_body_force((case["force"], 0.0, 0.0))
    if case["pairs"]:
        sim.set_rnemd(y_a=0.0, y_b=case["Ly"] / 2.0, max_pairs=case["pairs"])
    if case["lags"]:
        sim.set_vacf(case["lags"])
    st = dict(case=case, sim=sim, buf=buf, own=own)
    if case["kind"] == "transfer":
        st["own_out"] = {k: torch.empty_like(t, pin_memory=True) for k, t in own.items()}
        st["out"] = {k: t.numpy() for k, t in st["own_out"].items()}
    return st


# -------------------------------------------------------------------- a pass
def run(state):
    case = state["case"]
    if case["kind"] == "collide":
        B.collide_solvent_static(state["prm"], state["L"], *state["x"], *state["v"], state["tag"], step=state["step"])
        state["step"] += 1
        return dict(zip(("vx", "vy", "vz"), state["v"]))
    sim = state["sim"]
    if case["kind"] == "transfer":
        sim.set_state_buffers(state["buf"])
        sim.get_state_buffers(state["out"])
        return {k: a for k, a in state["out"].items() if a.size}
    sim.step(case["steps"])
    sim.get_state_buffers(state["buf"])
    out = {k: a for k, a in state["buf"].items() if a.size}
    if case["pairs"]:
        out["p_moved"], out["pairs"] = sim.rnemd_totals()
        out["mass"], out["momentum"] = sim.velocity_profile(case["Ly"])
    if case["lags"]:
        out["ct"], out["cr"], out["origins"] = sim.vacf()
    return out


def _sizes(case):
    """(solvent, cells) of all boxes."""
    if case["kind"] == "collide":
        return case["n"], case["Lx"] * case["Ly"] * case["Lz"]
    if case["layout"] == "mixed":
        reps = [r for r, _ in _mixed_boxes(case["n_rep"])[1]]
        return sum(r.n_solvent for r in reps), sum(math.prod(r.L) for r in reps)
    if case["layout"] == "single":
        c = int((np.random.default_rng(3).choice([12, 16, 20, 24], size=case["n_rep"]) ** 3).sum())
    else:
        c = case["Lx"] * case["Ly"] * case["Lz"]
    return int(case["density"] * c), c


def work(case):
    """Bytes: a step reads and writes every solvent particle's position and velocity once, a snapshot
    reads and writes them once more; a collision reads both and writes the velocities.  Operations:
    the cell sums (10), the rule (40; the +a correction 60 more) and the streaming (6) of a particle."""
    n, _ = _sizes(case)
    row = 48.0 if case.get("precision") == "p64" else 24.0
    if case["kind"] == "collide":
        return {"bytes": 1.5 * row * n, "flops": 50.0 * n}
    if case["kind"] == "transfer":
        return {"bytes": 2 * row * n, "flops": 1.0}
    per = 56.0 + (60.0 if case["angular"] else 0.0)
    return {"bytes": 2 * row * n * (case["steps"] + 1), "flops": per * n * case["steps"]}


# ------------------------------------------------------ the same in 64 bits
def _philox(key, step, ids, tag, j=0):
    """Philox4x32-10 (Salmon et al., SC'11): four words of 32 bits for each id."""
    c = [np.full(len(ids), step & 0xFFFFFFFF, np.uint64), ids.astype(np.uint64), np.full(len(ids), tag, np.uint64),
         np.full(len(ids), j, np.uint64)]
    k0, k1, low = key & 0xFFFFFFFF, key >> 32, np.uint64(0xFFFFFFFF)
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & low, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _u(w):
    return (w.astype(np.float64) + 0.5) * 2.0 ** -32


def _normals(key, step, ids, tag):
    w = [_u(a) for a in _philox(key, step, ids, tag)]
    r1, r2, t = np.sqrt(-2 * np.log(w[0])), np.sqrt(-2 * np.log(w[2])), 2 * np.pi
    return np.stack([r1 * np.cos(t * w[1]), r1 * np.sin(t * w[1]), r2 * np.cos(t * w[3])], axis=1)


def _gamma(key, step, cells, n, thermostat):
    """Gamma((3 n - 3) / 2) of each cell: a sum of exponentials, or Marsaglia and Tsang's rejection."""
    dof = 3 * (n - 1)
    g = np.zeros(len(cells))
    if thermostat == 1:
        for j in range(int(-(-(dof.max() // 2) // 4))):
            for k, w in enumerate(_philox(key, step, cells, 3, j)):
                g += np.where(4 * j + k < dof // 2, -np.log(_u(w)), 0.0)
        w = _philox(key, step, cells, 4)
        return g + np.where(dof % 2 == 1, -np.log(_u(w[0])) * np.cos(2 * np.pi * _u(w[1])) ** 2, 0.0)
    left = np.arange(len(cells))
    for j in range(64):
        if not len(left):
            break
        w = [_u(a) for a in _philox(key, step, cells[left], 7, j)]
        d = 0.5 * dof[left] - 1 / 3
        r = np.sqrt(-2 * np.log(w[0]))
        done = np.zeros(len(left), dtype=bool)
        for x, u in ((r * np.cos(2 * np.pi * w[1]), w[2]), (r * np.sin(2 * np.pi * w[1]), w[3])):
            t = 1 + x / np.sqrt(9 * d)
            v = np.where(t > 0, t, 1.0) ** 3
            ok = ~done & (t > 0) & (np.log(u) < 0.5 * x * x + d - d * v + d * np.log(v))
            g[left[ok]] = (d * v)[ok]
            done |= ok
        left = left[~done]
    return g


def _collision(case, key, step, L, x, v, m, draw_ids):
    """The rule on all members (positions x, velocities v, masses m; kT = 1): the new velocities."""
    w = _philox(key, step, np.zeros(1), 1)
    S = np.array([int(a[0]) >> 12 for a in w[:3]]) - (1 << 19)
    c = ((np.floor(x * 1048576.0).astype(np.int64) - S) >> 20) % np.array(L)
    cell = c[:, 0] + L[0] * (c[:, 1] + L[1] * c[:, 2])
    C = math.prod(L)

    def add(a):
        return np.bincount(cell, weights=a, minlength=C)

    n, M = np.bincount(cell, minlength=C), add(m)
    some = np.maximum(M, 1e-300)
    u = np.stack([add(m * v[:, k]) for k in range(3)], axis=1) / some[:, None]
    rel = v - u[cell]
    lone = (n < 2)[cell][:, None]
    if case["rule"] == "at":
        xi = _normals(key, step, draw_ids, 6) / np.sqrt(m)[:, None]
        mean = np.stack([add(m * xi[:, k]) for k in range(3)], axis=1) / some[:, None]
        return np.where(lone, v, u[cell] + xi - mean[cell])
    ids = np.arange(C)
    w = _philox(key, step, ids, 2)
    z, ph = 2 * _u(w[0]) - 1, 2 * np.pi * _u(w[1])
    rho = np.sqrt(1 - z * z)
    axis = np.stack([rho * np.cos(ph), rho * np.sin(ph), z], axis=1)[cell]
    kappa = np.ones(C)
    if case["thermostat"]:
        on = np.flatnonzero(n >= 2)
        erel = 0.5 * add(m * (rel * rel).sum(1))[on]
        kappa[on] = np.sqrt(_gamma(key, step, on, n[on], case["thermostat"]) / erel)
    ca, sa = math.cos(math.radians(130.0)), math.sin(math.radians(130.0))
    dot = (axis * rel).sum(1, keepdims=True)
    new = u[cell] + kappa[cell][:, None] * (rel * ca + np.cross(axis, rel) * sa + axis * dot * (1 - ca))
    return np.where(lone, v, new)


def _matrices(q):
    w, x, y, z = q.T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                     1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                     1 - 2 * (x * x + y * y)], axis=1).reshape(-1, 3, 3)


def _exact_run(case, seed):
    """Whole steps of one box of spheres, none of them within reach of another (the lattice keeps them apart)."""
    system, R, q = _system(case, seed)
    b = {k: a.copy() for k, a in _state(case, seed, system, R, q)[0].items()}
    L, sh, key, dt = np.array(system.replicas[0].L), system.shapes[0], 1 + seed, 0.1
    n, nb, ns = system.n_solvent, system.n_bodies, sh.n_sites
    M = sh.m.sum()
    inertia = np.array([(sh.m * ((sh.b ** 2).sum(1) - sh.b[:, k] ** 2)).sum() for k in range(3)])
    ids = np.arange(n + nb * ns)
    m = np.concatenate([np.ones(n), np.tile(sh.m, nb)])

    def spin(Q, ang):       # angular velocity of an angular momentum
        return np.einsum("bij,bj->bi", Q, np.einsum("bji,bj->bi", Q, ang) / inertia)

    for step in range(case["steps"]):
        b["x"] = (b["x"] + dt * b["v"]) % L
        b["R"] = (b["R"] + dt * b["P"] / M) % L
        for k, h in ((2, 0.5), (1, 0.5), (0, 1.0), (1, 0.5), (2, 0.5)):     # free rotations about body axes
            half = 0.5 * dt * h * np.einsum("bj,bj->b", _matrices(b["q"])[:, :, k], b["Lm"]) / inertia[k]
            r, i = b["q"][:, [0]], b["q"][:, 1:]
            e = np.zeros(3)
            e[k] = 1.0
            c, s = np.cos(half)[:, None], np.sin(half)[:, None]
            b["q"] = np.concatenate([r * c - i[:, [k]] * s, i * c + s * (r * e + np.cross(i, e))], axis=1)
        b["q"] /= np.linalg.norm(b["q"], axis=1, keepdims=True)
        Q = _matrices(b["q"])
        d = np.einsum("bij,sj->bsi", Q, sh.b)
        ms = sh.m[None, :, None]
        th = _normals(key, step, ids[n:], 5).reshape(nb, ns, 3) / np.sqrt(ms)
        V = b["P"] / M - (ms * th).sum(1) / M
        W = spin(Q, b["Lm"]) - spin(Q, np.cross(d, ms * th).sum(1))
        vs = th + V[:, None] + np.cross(W[:, None], d)
        xs = (b["R"][:, None] + d) % L
        v = _collision(case, key, step, tuple(int(a) for a in L), np.concatenate([b["x"], xs.reshape(-1, 3)]),
                       np.concatenate([b["v"], vs.reshape(-1, 3)]), m, ids)
        dp = ms * (v[n:].reshape(nb, ns, 3) - vs)
        b["v"], b["P"], b["Lm"] = v[:n], b["P"] + dp.sum(1), b["Lm"] + np.cross(d, dp).sum(1)
    return {k: a for k, a in b.items() if a.size}


def exact(case, seed):
    """None for the FP32 runs: within a few steps a particle within a rounding of a cell face lands in
    another cell than in 64 bits, and from there the two trajectories part, whatever the arithmetic."""
    if case["kind"] == "collide":
        L, x, v, _ = _collide_inputs(case, seed)
        x = np.stack([t.double().cpu().numpy() for t in x], axis=1)
        v = np.stack([t.double().cpu().numpy() for t in v], axis=1)
        new = _collision(case, 1 + seed, case["step"], L, x, v, np.ones(case["n"]), np.arange(case["n"]))
        return {k: new[:, i] for i, k in enumerate(("vx", "vy", "vz"))}
    if case["kind"] == "transfer":
        buf, _ = _state(case, seed, *_system(case, seed))
        return {k: a.astype(np.float64) for k, a in buf.items() if a.size}
    if case["precision"] == "p64" and case["n_rep"] == 1 and case["steps"] <= 6 and _sizes(case)[0] <= 600000:
        return _exact_run(case, seed)
    return None
