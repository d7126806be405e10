"""Performance cases of the tree-gravity framework: what its users run, over the range of sizes and options they run it at.

listed() names the cases that are timed, draw(rng) gives further ones from the same ranges, prepare(case, seed) makes a
program's state before the call, run(state) is one pass through the public entry points, work(case) the bytes and flops no
implementation can do without, and exact(case, seed) the result in 64 bits (direct sums, plain torch) where that is feasible.

Kinds:
  step       one captured kick-drift-kick step with energies of a star cluster or an ensemble (rv_kdk_step_graph)
  kdk        one kick-drift-kick step launched kernel by kernel (rv_kdk_step)
  forces     tree build and tree forces (rv_build_tree, rv_tree_forces)
  rel        tree build and forces under the relative criterion (rv_build_tree, rv_tree_forces_rel)
  system     the whole force pass of a galaxy with an SMBH or an SMBH pair (rv_system_forces)
  blocks     one dt_max of hierarchical block steps (rv_block_steps)
  substep    the perturbers' pull inside a chain integrator's substep (rv_chain_perturber_forces)
  search     the k nearest perturbers of a chain (rv_select_perturbers)
  network    inference of the cell-force network (rv_mlp_forward)
  gradient   a minibatch's loss and gradient (rv_mlp_gradient)
"""
import math
import random

import numpy as np
import torch

from paper_1507_01009_gb300 import rv

GALAXY = {"theta": 0.5, "eps": 0.005, "n_leaf": 24, "group": 64, "tile": 96, "quad": True, "softening": 0}


def listed():
    return [
        # a chain integrator's own force evaluation: dozens of these per tree step, each a few microseconds of work
        {"name": "substep_pair_k256", "kind": "substep", "n": 65536, "k": 256, "pair": True},
        # the smallest system the framework is used on: a star cluster, captured step with energies; latency and launches count
        {"name": "step_cluster_4096", "kind": "step", "profile": "plummer", "n": 4096, "members": 1, "pair": False, "theta": 0.5,
         "eps": 0.01, "n_leaf": 16, "group": 32, "tile": 96, "quad": True, "softening": 0},
        # a library user with the default configuration and an odd star count: build and forces
        {"name": "forces_default_100003", "kind": "forces", "n": 100003, "theta": 0.5, "eps": 0.01, "n_leaf": 16, "group": 32,
         "tile": 64, "quad": True, "softening": 0},
        # the galaxy with one SMBH, perturbers within a radius: the whole force pass
        {"name": "system_smbh_1m", "kind": "system", "n": 1 << 20, "pair": False, "mode": 1, "radius": 0.02, "k": 0, **GALAXY},
        # the same galaxy under the relative opening criterion with the previous step's accelerations
        {"name": "forces_relative_1m", "kind": "rel", "n": 1 << 20, "alpha": 1e-3, **GALAXY},
        # the galaxy with a central SMBH pair, its 256 nearest stars as perturbers and the pair's quadrupole on the others
        {"name": "system_pair_4m", "kind": "system", "n": 1 << 22, "pair": True, "mode": 2, "radius": 0.0, "k": 256, **GALAXY},
        # the largest galaxy of the benchmark, one step
        {"name": "step_galaxy_16m", "kind": "kdk", "n": 1 << 24, **dict(GALAXY, theta=0.8)},
        # an ensemble of uneven galaxies, each with an SMBH pair, stepped together by one graph
        {"name": "step_ensemble_16", "kind": "step", "profile": "hernquist", "n": 0, "members": 16, "lo": 8192, "hi": 65536,
         "size_seed": 4, "pair": True, **GALAXY},
        # hierarchical block steps: sixteen substeps, each rebuilding the tree and walking the active groups
        {"name": "blocks_200001", "kind": "blocks", "n": 200001, "max_level": 4, **GALAXY},
        # the perturber search on its own, as a chain integrator calls it between tree steps
        {"name": "search_nearest_1m", "kind": "search", "n": 1 << 20, "k": 256},
        # the cell-force network: inference on the (group, cell) pairs of a force pass, and a training minibatch
        {"name": "network_4m_rows", "kind": "network", "rows": 4000003},
        {"name": "gradient_8192_rows", "kind": "gradient", "rows": 8192},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["substep", "step", "step", "forces", "forces", "rel", "system", "system", "kdk", "blocks", "search",
                       "network", "gradient"])
    tree = {"theta": round(rng.uniform(0.4, 0.9), 3), "eps": rng.choice([0.005, 0.01]), "n_leaf": rng.choice([16, 24, 32]),
            "group": rng.choice([32, 64, 64]), "tile": rng.choice([64, 96, 128]), "quad": rng.random() < 0.85,
            "softening": 1 if rng.random() < 0.15 else 0}
    if kind == "substep":
        return {"kind": kind, "n": _log(rng, 8192, 1 << 18), "k": _log(rng, 16, 5000), "pair": rng.random() < 0.5}
    if kind == "search":
        return {"kind": kind, "n": _log(rng, 5000, 1 << 22), "k": _log(rng, 1, 5000)}
    if kind == "network":
        return {"kind": kind, "rows": _log(rng, 1000, 1 << 23)}
    if kind == "gradient":
        return {"kind": kind, "rows": _log(rng, 64, 65536)}
    if kind == "step" and rng.random() < 0.5:
        return {"kind": kind, "profile": "plummer", "n": _log(rng, 1000, 65536), "members": 1, "pair": False, **tree}
    if kind == "step":
        return {"kind": kind, "profile": "hernquist", "n": 0, "members": rng.randint(2, 48), "lo": 4096, "hi": 65536,
                "size_seed": rng.randrange(1 << 20), "pair": True, **dict(tree, quad=True, softening=0)}
    if kind == "rel":
        return {"kind": kind, "n": _log(rng, 10000, 1 << 21), "alpha": round(math.exp(rng.uniform(math.log(5e-4), math.log(5e-3))), 6),
                **tree}
    if kind == "system":
        near = rng.random() < 0.5
        return {"kind": kind, "n": _log(rng, 10000, 1 << 21), "pair": rng.random() < 0.5, "mode": 2 if near else 1,
                "radius": 0.0 if near else 0.02, "k": _log(rng, 16, 2000) if near else 0, **tree}
    if kind == "blocks":
        return {"kind": kind, "n": _log(rng, 10000, 1 << 18), "max_level": rng.randint(2, 4), **dict(tree, softening=0)}
    return {"kind": kind, "n": _log(rng, 1000, 1 << 22), **tree}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _isotropic(g, n):
    c, p = 2.0 * _uniform(g, n) - 1.0, 2.0 * math.pi * _uniform(g, n)
    s = torch.sqrt(1.0 - c * c)
    return torch.stack([s * torch.cos(p), s * torch.sin(p), c])


def _stars(g, n, profile="hernquist"):
    """Positions and velocities (3, n) in FP32 and masses of a unit-mass Hernquist sphere (enclosed-mass fraction up to 0.99) or
    Plummer sphere; speeds Gaussian at about the local dispersion, cut at the escape speed."""
    if profile == "plummer":
        u = (_uniform(g, n) * 0.999).clamp_min(1e-12)
        r = 1.0 / torch.sqrt(u ** (-2.0 / 3.0) - 1.0)
        vesc = math.sqrt(2.0) * (1.0 + r * r) ** -0.25
    else:
        s = torch.sqrt(_uniform(g, n) * 0.99)
        r = s / (1.0 - s)
        vesc = torch.sqrt(2.0 / (1.0 + r))
    pos = _isotropic(g, n) * r
    vel = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64) * (0.25 * vesc)
    vel *= torch.clamp(0.99 * vesc / vel.norm(dim=0).clamp_min(1e-12), max=1.0)
    return pos.float(), vel.float(), torch.full((n,), 1.0 / n, dtype=torch.float32, device="cuda")


def _sizes(case):
    if case["members"] == 1:
        return [case["n"]]
    r = random.Random(case["size_seed"])
    return [_log(r, case["lo"], case["hi"]) for _ in range(case["members"])]


def _bodies(case, seed):
    """Stars of every member, member offsets, and the chains' masses, positions and velocities (FP64, or None)."""
    g = _gen(seed)
    sizes = _sizes(case) if case["kind"] == "step" else [case["n"]]
    parts = [_stars(g, n, case.get("profile", "hernquist")) for n in sizes]
    pos, vel, m = (torch.cat([p[k] for p in parts], dim=-1) for k in range(3))
    off = [0]
    for n in sizes:
        off.append(off[-1] + n)
    if "pair" not in case or (case["kind"] == "step" and not case["pair"]):
        return pos, vel, m, off, None
    if case["pair"]:   # a = 0.01, e = 0.1, at apocentre, masses 0.005
        sep, v = 0.011, math.sqrt(0.01 * 0.9 / 0.011)
        cm, cx, cv = [0.005, 0.005], [[sep / 2, 0, 0], [-sep / 2, 0, 0]], [[0, v / 2, 0], [0, -v / 2, 0]]
    else:              # one SMBH on a circular orbit at r = 0.5
        cm, cx, cv = [0.005], [[0.5, 0, 0]], [[0, math.sqrt(0.5) / 1.5, 0]]
    k = len(sizes)
    chain = tuple(torch.tensor(t, dtype=torch.float64, device="cuda").repeat(*([k] + [1] * (d - 1)))
                  for t, d in ((cm, 1), (cx, 2), (cv, 2)))
    return pos, vel, m, off, chain


def _rows(case, seed):
    """Features and targets as the walk's accepted cells have them: direction, s/|r|, eps/|r|, Q/(M s^2), octupole terms."""
    g, n = _gen(seed), case["rows"]
    x = torch.zeros(n, 16, dtype=torch.float64, device="cuda")
    x[:, 0:3] = _isotropic(g, n).T
    x[:, 3] = 0.05 + 0.75 * _uniform(g, n)
    x[:, 4] = 0.1 * _uniform(g, n) ** 4
    x[:, 5:14] = torch.randn(n, 9, generator=g, device="cuda", dtype=torch.float64) * 0.05
    t = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64) * 0.02
    return x.float(), t.float()


def _reference(pos):
    """Accelerations of the previous step, as the Hernquist model has them."""
    r = pos.double().norm(dim=0).clamp_min(1e-6)
    return (-pos.double() / (r * (1.0 + r) ** 2)).float()


def _levels(case, pos):
    """Block levels by radius: the inner stars on the finest levels, most of the galaxy on the coarse ones."""
    r = pos.double().norm(dim=0)
    return torch.clamp(torch.floor(-1.5 * torch.log2(r.clamp_min(1e-6))), 0, case["max_level"]).to(torch.int8)


def _context(case, n, **kw):
    return rv.Context(n, theta=case["theta"], eps_star=case["eps"], n_leaf=case["n_leaf"], group=case["group"],
                      quadrupole=case["quad"], tile=case["tile"], softening=case["softening"], **kw)


_STREAM = []


def _stream():
    """The program's one stream for captured steps."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


DT = 1e-3
DT_MAX = 1.0 / 64
DT_SUB = 1e-4


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("network", "gradient"):
        x, t = _rows(case, seed)
        return {"case": case, "net": rv.Mlp(seed=7), "x": x, "t": t}
    pos, vel, m, off, chain = _bodies(case, seed)
    s = {"case": case, "pos": pos.contiguous(), "m": m}
    n = off[-1]
    if kind in ("forces", "rel"):
        s["ctx"] = _context(case, n)
        if kind == "rel":
            s["ref"] = _reference(pos).contiguous()
        return s
    if kind == "search":
        s["ctx"] = rv.Context(n)
        return s
    extra = {}
    if chain is not None:
        mode = case.get("mode", 2)
        extra = dict(chain_m=chain[0], chain_x=chain[1], chain_v=chain[2], pert_mode=mode, pert_radius=case.get("radius", 0.0),
                     pert_k=case.get("k", 256))
    if kind == "step" and case["members"] > 1:
        extra["member_offsets"] = np.array(off, dtype=np.int64)
    s["sys"] = rv.System(pos, vel, m, **extra)
    s["ctx"] = rv.Context(n, theta=0.8, eps_star=0.005, n_leaf=24, group=64) if kind == "substep" else _context(case, n)
    if kind == "step":
        s["stream"] = _stream()
        s["energy"] = torch.zeros(10 * case["members"], dtype=torch.float64, device="cuda")
    if kind in ("kdk", "substep"):
        s["ctx"].system_forces(s["sys"])
    if kind == "substep":   # the chain a little further on its orbit than at the force pass
        s["at"] = (chain[1] + DT_SUB * chain[2]).contiguous()
    if kind == "blocks":
        s["blocks"] = rv.Blocks(n, DT_MAX, case["max_level"], eps=case["eps"], adapt=False, level=_levels(case, pos))
        s["ctx"].block_start(s["sys"], s["blocks"])
    return s


def _state(sys):
    out = {"pos": sys.state[0:3], "vel": sys.state[3:6], "acc": sys.state[6:9], "pot": sys.state[9]}
    if sys.n_chain:
        out["chain_a"], out["chain_pot"] = sys.chain_a, sys.chain_pot
    return out


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "network":
        return state["net"].forward(state["x"])
    if kind == "gradient":
        return list(state["net"].gradient(state["x"], state["t"]))
    ctx = state["ctx"]
    if kind == "forces":
        ctx.build_tree(*state["pos"], state["m"])
        return list(ctx.tree_forces())
    if kind == "rel":
        ctx.build_tree(*state["pos"], state["m"])
        return list(ctx.tree_forces_rel(case["alpha"], state["ref"]))
    if kind == "search":
        idx, count = ctx.select_perturbers(*state["pos"], (0.0, 0.0, 0.0), 2, k=case["k"])
        return [idx[:case["k"]], count]
    sys = state["sys"]
    if kind == "substep":
        return list(ctx.chain_perturber_forces(sys, DT_SUB, state["at"]))
    if kind == "system":
        ctx.system_forces(sys)
        out = _state(sys)
        return {k: out[k] for k in out if k not in ("pos", "vel")}
    if kind == "step":
        ctx.kdk_step_graph(sys, DT, 1, state["energy"], stream=state["stream"])
        return dict(_state(sys), energy=state["energy"])
    if kind == "kdk":
        ctx.kdk_step(sys, DT)
    else:
        ctx.block_steps(sys, state["blocks"], 1 << case["max_level"])
    return _state(sys)


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _interactions(n, case):
    """Star-star and star-cell interactions a star has in such a sphere under the opening test: a fit to the walk's counters, within
    about a third over the ranges above (the relative criterion acts like an angle that grows with its tolerance)."""
    th = 0.72 * (case["alpha"] / 1e-3) ** 0.2 if case["kind"] == "rel" else case["theta"]
    cells = 1850.0 / th ** 1.7 / (1.0 + (7e4 / n) ** 0.9)
    stars = 1500.0 / th ** 1.2 * math.sqrt(case["n_leaf"] * case["group"] / 1536.0)
    return min(stars, float(n)), cells


def _pass_work(n, case):
    stars, cells = _interactions(n, case)
    return {"bytes": 32.0 * n, "flops": n * (20.0 * stars + (54.0 if case["quad"] else 18.0) * cells)}


def work(case):
    kind = case["kind"]
    if kind in ("network", "gradient"):
        n, f = case["rows"], 2.0 * (14 * 64 + 64 * 64 + 64 * 3)
        if kind == "network":
            return {"bytes": n * (14 * 4 + 3 * 4), "flops": n * f}
        return {"bytes": n * (14 * 4 + 3 * 4) + 2 * 4 * 5768, "flops": n * (3.0 * f - 2.0 * 14 * 64)}
    n = case["n"]
    if kind == "search":
        return {"bytes": 12.0 * n + 4 * case["k"], "flops": 8.0 * n}
    if kind == "substep":
        c = 2 if case["pair"] else 1
        return {"bytes": (28 + 4) * case["k"] + 56 * c, "flops": case["k"] * (6.0 + 20.0 * c)}
    if kind == "step":
        w = [_pass_work(k, case) for k in _sizes(case)]
        n = sum(_sizes(case))
        return {"bytes": sum(q["bytes"] for q in w) + 60.0 * n, "flops": sum(q["flops"] for q in w) + 40.0 * n}
    w = _pass_work(n, case)
    if kind == "kdk":
        w["bytes"] += 60.0 * n
    if kind == "rel":
        w["bytes"] += 12.0 * n
    if kind == "blocks":   # level l is active 2^l times; most stars sit on the coarse levels
        subs, r = 1 << case["max_level"], [2.0 ** (-l / 1.5) for l in range(case["max_level"] + 1)]
        inside = [q * q / (1 + q) ** 2 / 0.99 for q in r]      # mass within the radius where level l begins
        updates = 1.0 + sum(inside[l] * (2 ** l - 2 ** (l - 1)) for l in range(1, case["max_level"] + 1))
        return {"bytes": subs * 36.0 * n + updates * 28.0 * n, "flops": updates * w["flops"]}
    return w


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _spline(r2, m, h):
    """m f / h^3 and m P / h of the cubic-spline kernel of support h; Newton beyond it."""
    r = torch.sqrt(r2)
    u = (r / h).clamp(1e-9, 1.0)
    a = 32 / 3 + u * u * (-192 / 5 + 32 * u)
    b = 64 / 3 - 48 * u + 192 / 5 * u * u - 32 / 3 * u ** 3 - 1 / (15 * u ** 3)
    p = -14 / 5 + u * u * (16 / 3 + u * u * (-48 / 5 + 32 / 5 * u))
    q = -16 / 5 + 1 / (15 * u) + u * u * (32 / 3 + u * (-16 + u * (48 / 5 - 32 / 15 * u)))
    f, w = torch.where(u < 0.5, a, b) / h ** 3, torch.where(u < 0.5, p, q) / h
    out = r >= h
    rinv = 1.0 / r.clamp_min(1e-30)
    return m * torch.where(out, rinv ** 3, f), m * torch.where(out, -rinv, w)


def _direct(x, m, eps, soft, at=None, unsoftened=False, skip_self=True):
    """Accelerations (3, k) and potentials of all points `at` (default: the bodies themselves) by direct summation."""
    at = x if at is None else at
    k, n = at.shape[1], x.shape[1]
    acc, pot = torch.empty(3, k, dtype=torch.float64, device="cuda"), torch.empty(k, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 26) // n)
    for i in range(0, k, step):
        p = at[:, i:i + step]
        d = [x[a][None, :] - p[a][:, None] for a in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        if soft == 1 and not unsoftened:
            f, w = _spline(r2, m[None, :], 2.8 * eps)
        else:
            rinv = torch.rsqrt(r2 + (0.0 if unsoftened else eps * eps))
            rinv = torch.where(torch.isfinite(rinv), rinv, torch.zeros_like(rinv))
            f, w = m[None, :] * rinv ** 3, -m[None, :] * rinv
        if skip_self:
            own = torch.arange(i, i + p.shape[1], device="cuda")
            w[torch.arange(p.shape[1], device="cuda"), own] = 0.0
        for a in range(3):
            acc[a, i:i + step] = (f * d[a]).sum(1)
        pot[i:i + step] = w.sum(1)
    return acc, pot


def _resolved(case, x, m, off, cx, cm):
    """Forces on the stars of every member and on its chain members: star pairs softened, every pair with an SMBH not."""
    eps, soft = float(np.float32(case["eps"])), case["softening"]
    acc, pot, ca, cp = [], [], [], []
    members = len(off) - 1
    for k in range(members):
        xs, ms = x[:, off[k]:off[k + 1]], m[off[k]:off[k + 1]]
        a, p = _direct(xs, ms, eps, soft)
        if cx is not None:
            per = cx.shape[0] // members
            xc, mc = cx[k * per:(k + 1) * per].T, cm[k * per:(k + 1) * per]
            b, q = _direct(xc, mc, 0.0, 0, at=xs, unsoftened=True, skip_self=False)
            a, p = a + b, p + q
            b, q = _direct(xs, ms, 0.0, 0, at=xc, unsoftened=True, skip_self=False)
            b2, q2 = _direct(xc, mc, 0.0, 0, unsoftened=True)
            ca.append((b + b2).T.reshape(-1))
            cp.append(q + q2)
        acc.append(a)
        pot.append(p)
    out = {"acc": torch.cat(acc, 1), "pot": torch.cat(pot)}
    if cx is not None:
        out["chain_a"], out["chain_pot"] = torch.cat(ca), torch.cat(cp)
    return out


def _energies(x, v, m, pot, off, cx, cv, cm, cp):
    out, members = [], len(off) - 1
    for k in range(members):
        s = slice(off[k], off[k + 1])
        X, V, M, P = x[:, s], v[:, s], m[s], pot[s]
        if cx is not None:
            per = cx.shape[0] // members
            c = slice(k * per, (k + 1) * per)
            X, V, M, P = torch.cat([X, cx[c].T], 1), torch.cat([V, cv[c].T], 1), torch.cat([M, cm[c]]), torch.cat([P, cp[c]])
        ek, ep = 0.5 * (M * (V * V).sum(0)).sum(), 0.5 * (M * P).sum()
        out.append(torch.stack([ek, ep, ek + ep, *(M * V).sum(1), *(M * torch.linalg.cross(X, V, dim=0)).sum(1), M.sum()]))
    return torch.cat(out)


def _splitmix(x):
    x = x + np.uint64(0x9E3779B97F4A7C15)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return x ^ (x >> np.uint64(31))


def _weights(seed):
    """The network's initial weights rounded to bfloat16 (Glorot-uniform from SplitMix64; biases zero), FP64."""
    with np.errstate(over="ignore"):
        u = (_splitmix(np.uint64(seed) ^ (np.uint64(0xA5A5A5A5) + np.arange(5768, dtype=np.uint64))) >> np.uint64(40)) / 16777216.0
    u = 2.0 * torch.from_numpy(u.astype(np.float32)).cuda() - 1.0
    w1 = torch.tensor(math.sqrt(6 / 78), dtype=torch.float32) .cuda() * u[:1024].view(16, 64)
    w2 = torch.tensor(math.sqrt(6 / 128), dtype=torch.float32).cuda() * u[1088:5184].view(64, 64)
    w3 = torch.tensor(math.sqrt(6 / 67), dtype=torch.float32).cuda() * u[5248:5760].view(64, 8)
    w1[14:] = 0.0
    w3[:, 3:] = 0.0
    return tuple(w.bfloat16().double() for w in (w1, w2, w3))


def _network(case, seed):
    x, t = _rows(case, seed)
    w1, w2, w3 = _weights(7)
    rnd = lambda v: v.float().bfloat16().double()  # noqa: E731
    out, g, loss = [], [torch.zeros_like(w1), torch.zeros_like(w2), torch.zeros_like(w3)], 0.0
    gb = [torch.zeros(w.shape[1], dtype=torch.float64, device="cuda") for w in (w1, w2, w3)]
    n = case["rows"]
    for i in range(0, n, 1 << 18):
        a = rnd(x[i:i + (1 << 18)])
        z1 = a @ w1
        s1 = torch.sigmoid(z1)
        h1 = rnd(z1 * s1)
        z2 = h1 @ w2
        s2 = torch.sigmoid(z2)
        h2 = rnd(z2 * s2)
        y = h2 @ w3
        out.append(y[:, :3])
        if case["kind"] == "gradient":
            e = y[:, :3] - t[i:i + (1 << 18)].double()
            loss = loss + (e * e).sum() / (3 * n)
            dy = torch.zeros_like(y)
            dy[:, :3] = 2.0 / (3 * n) * e
            d2 = (dy @ w3.T) * s2 * (1 + z2 * (1 - s2))
            d1 = (d2 @ w2.T) * s1 * (1 + z1 * (1 - s1))
            for k, (h, d) in enumerate(((a, d1), (h1, d2), (h2, dy))):
                g[k] += h.T @ d
                gb[k] += d.sum(0)
    if case["kind"] == "network":
        return torch.cat(out)
    return [torch.cat([v for k in range(3) for v in (g[k].reshape(-1), gb[k])]), loss.reshape(1)]


def _nearest(pos, centre, k):
    d = pos - centre.float()[:, None]
    d2 = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]
    return torch.sort(d2, stable=True).indices[:k]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("network", "gradient"):
        return _network(case, seed)
    if kind in ("search", "blocks"):   # whole numbers; sixteen substeps of direct sums
        return None
    members = _sizes(case) if kind == "step" else [case["n"]]
    if kind != "substep" and sum(n * n for n in members) * (2 if kind in ("step", "kdk") else 1) > 3 << 34:
        return None
    pos, vel, m, off, chain = _bodies(case, seed)
    x, v, md = pos.double(), vel.double(), m.double()
    cm, cx, cv = chain if chain is not None else (None, None, None)
    if kind == "substep":
        com = (cm[:, None] * cx).sum(0) / cm.sum()
        p = _nearest(pos, com, case["k"])
        a, q = _direct(x[:, p] + DT_SUB * v[:, p], md[p], 0.0, 0, at=(cx + DT_SUB * cv).T, unsoftened=True, skip_self=False)
        return [a.T.reshape(-1), q]
    if kind in ("forces", "rel", "system"):
        f = _resolved(case, x, md, off, cx, cm)
        return f if kind == "system" else [*f["acc"], f["pot"]]
    f = _resolved(case, x, md, off, cx, cm)
    v = v + f["acc"] * (DT / 2)
    x = x + v * DT
    if cx is not None:
        cv = cv + f["chain_a"].view(-1, 3) * (DT / 2)
        cx = cx + cv * DT
    f = _resolved(case, x, md, off, cx, cm)
    v = v + f["acc"] * (DT / 2)
    if cx is not None:
        cv = cv + f["chain_a"].view(-1, 3) * (DT / 2)
    out = dict(f, pos=x, vel=v)
    if kind == "step":
        out["energy"] = _energies(x, v, md, f["pot"], off, cx, cv, cm, f.get("chain_pot"))
    return out
