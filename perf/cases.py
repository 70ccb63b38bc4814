"""Performance cases: the work a user of this package has it do, at the sizes they do it.

Each case is one pass through the public calls of ``paper_2506_05362_gb300.pd``: a
stretch of velocity-Verlet steps from a given state (set the state, step, read the
state back), one step of a coupled program, the bond set-up of a new body, or the
surrogate network's inference and training.  Bodies and sizes are those of
``scenarios``, the tests and ``bench.py``.

The mixed path's forces are FP32 numbers that the C ABI hands over as doubles, and the
positions and velocities they move are as good as those forces: the outputs of the
mixed cases are given in FP32, those of the all-FP64 path in FP64.  The network stores
its weights and activations in BF16 (8 bits); its predictions and trained weights are
given in FP16 (11 bits), which keeps all that this leaves of them.
"""
import math

import numpy as np
import torch

from paper_2506_05362_gb300 import pd, scenarios as S, surrogate

DIMS = (109, 256, 256, 256, 256, 6)  # the surrogate network of bench.py and surrogate.train
DEV = "cuda"


def listed():
    return [
        # the smallest simulation: one glass sphere between two plates, a whole run of 200 steps;
        # a step is a few microseconds of work, so launches, barriers and latency are what counts
        {"name": "sphere_200", "kind": "crush", "inner": 0, "outer": 10, "steps": 200, "cracks": 0},
        # the benchmark's plate under impact: the ordinary single-body fracture run, horizon 4h
        {"name": "plate_128", "kind": "plate", "length": 100, "height": 200, "precision": "mixed", "steps": 128},
        # the hollow sphere being crushed, already cracked: horizon 3h, a third of a million nodes,
        # part of the bonds broken, a checkpointed state to go on from
        {"name": "shell_cracked_64", "kind": "crush", "inner": 35, "outer": 50, "steps": 64, "cracks": 3},
        # one strain record of a representative volume: touching grains with contact damping,
        # six moving walls, then stress, damage and the number of contacts (surrogate.rve_aggregate)
        {"name": "rve_record", "kind": "packing", "shape": "jack", "side": 4, "steps": 64, "zeta": 0.5, "mu": 0.0,
         "record": True},
        # the largest body: a thousand touching spheres in a box, 2.1 million nodes
        {"name": "packing_1000", "kind": "packing", "shape": "sphere", "side": 10, "steps": 16, "zeta": 0.0, "mu": 0.0,
         "record": False},
        # the all-FP64 path, which users run to check the mixed one, on the benchmark's plate cut
        {"name": "plate_fp64", "kind": "plate", "length": 40, "height": 60, "precision": "fp64", "steps": 24},
        # a program coupled step by step: the state in, one step, the state out (bench.py's end to end)
        {"name": "coupled_step", "kind": "coupled", "length": 100, "height": 200},
        # the set-up of a new body: bond lists, kernel choice, and the lists read back
        {"name": "build_bonds", "kind": "build", "inner": 21, "outer": 30},
        # the surrogate evaluated on a full batch, and on one run's 49 windows
        {"name": "infer_65536", "kind": "infer", "batch": 65536},
        {"name": "infer_49", "kind": "infer", "batch": 49},
        # training at the benchmark's batch, and one epoch in minibatches with a ragged last one
        {"name": "train_65536", "kind": "train", "samples": 65536, "batch": 65536, "passes": 4},
        {"name": "train_epoch", "kind": "train", "samples": 9751, "batch": 4096, "passes": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["crush", "crush", "plate", "plate", "packing", "packing", "coupled", "build", "infer", "infer",
                       "train", "train"])
    if kind in ("crush", "build"):
        outer = _log(rng, 6, 50 if kind == "crush" else 30)
        inner = rng.choice([0, int(0.7 * outer)]) if outer <= 30 else int(0.7 * outer)
        if kind == "build":
            return {"kind": kind, "inner": inner, "outer": outer}
        return {"kind": kind, "inner": inner, "outer": outer, "steps": rng.randint(20, 100),
                "cracks": rng.choice([0, rng.randint(1, 4)])}
    if kind == "plate":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        length = _log(rng, 16, 100 if precision == "mixed" else 40)
        return {"kind": kind, "length": length, "height": int(length * rng.uniform(1.2, 2.0)), "precision": precision,
                "steps": rng.randint(8, 24) if precision == "fp64" else rng.randint(8, 128)}
    if kind == "coupled":
        length = _log(rng, 16, 100)
        return {"kind": kind, "length": length, "height": int(length * rng.uniform(1.2, 2.0))}
    if kind == "packing":
        return {"kind": kind, "shape": rng.choice(["sphere", "shell", "jack"]), "side": rng.randint(2, 8),
                "steps": rng.randint(8, 48), "zeta": rng.choice([0.0, 0.5, rng.uniform(0.1, 0.9)]),
                "mu": rng.choice([0.0, 0.0, 0.3]), "record": rng.choice([True, False])}
    if kind == "infer":
        return {"kind": kind, "batch": _log(rng, 1, 65536)}
    samples = _log(rng, 64, 65536)
    return {"kind": kind, "samples": samples, "batch": rng.choice([samples, 4096]), "passes": 1}


# ---- bodies ---------------------------------------------------------------------
def _body(case):
    """The body: always the same for a case, as a program's mesh is; the seed draws the state it is in."""
    kind, seed = case["kind"], 0
    if kind in ("crush", "build"):
        if case["inner"]:
            sc = S.hollow(seed=seed, outer_cells=case["outer"], inner_cells=case["inner"])
        else:
            sc = S.sphere(seed=seed, radius_cells=case["outer"])
    elif kind in ("plate", "coupled"):
        L, H = case["length"] * 1e-3, case["height"] * 1e-3
        sc = S.kalthoff(length=L, height=H, notch_len=0.5 * L, notch_gap=max(0.25 * H, 8e-3))
    else:
        # radius 8h: the extreme nodes of two neighbours lie 0.55 h apart, inside the contact radius 0.6 h
        sc = S.shape_study(case["shape"], n_side=case["side"], seed=seed, gap_cells=-1.45)
        if case["zeta"] > 0:
            sc.material.beta_d = surrogate.damping_coefficient(sc.material, sc.horizon, float(sc.vol.mean()),
                                                               case["zeta"])
        sc.material.mu = case["mu"]
        if case["record"]:  # every wall moves inward, as in the isotropic pre-compression
            p = S.walls_array(sc.walls)[:, 3:6]
            for k, w in enumerate(sc.walls):
                a = k // 2
                w.velocity = tuple(1e3 * (p[2 * a + 1, a] - p[2 * a, a]) * np.array(w.normal))
        else:
            for w in sc.walls:
                w.velocity = (0.0, 0.0, 0.0)
    return sc


def _state(sc, seed):
    """u and v to start from: a smooth strain of some 1e-4, every grain's own velocity, and node noise."""
    rng = np.random.default_rng(seed + 1)
    u = (sc.x - sc.x.mean(0)) @ rng.normal(0.0, 5e-5, (3, 3)) + rng.normal(0.0, 2e-6 * sc.h, sc.x.shape)
    v = sc.v0 + rng.normal(0.0, 1.0, (int(sc.grain.max()) + 1, 3))[sc.grain] + rng.normal(0.0, 1e-2, sc.x.shape)
    return u, v


def _crack_planes(case, sc, seed):
    """Half-planes (normal, offset, direction) whose crossing bonds are broken at the start."""
    rng = np.random.default_rng(seed + 2)
    out = []
    for _ in range(case.get("cracks", 0)):
        n = rng.normal(size=3)
        n /= np.linalg.norm(n)
        d = rng.normal(size=3)
        out.append((n, rng.uniform(-0.3, 0.3) * float(np.abs(sc.x).max()), d / np.linalg.norm(d)))
    return out


def _cracked(planes, x, i, j):
    """Whether the bonds (i, j) cross a crack (x: torch FP64; i, j: torch indices)."""
    hit = torch.zeros(i.shape, dtype=torch.bool, device=x.device)
    for n, c, d in planes:
        side = x @ torch.tensor(n, device=x.device) > c
        open_ = x @ torch.tensor(d, device=x.device) > 0
        hit |= (side[i] != side[j]) & open_[i] & open_[j]
    return hit


def _pinned(shape, dtype):
    return torch.zeros(shape, dtype=dtype, pin_memory=True)


def _weights(seed):
    """A parameter vector of the network: per layer W (out x in) and b."""
    rng = np.random.default_rng(seed + 3)
    parts = []
    for a, b in zip(DIMS[:-1], DIMS[1:]):
        parts += [rng.uniform(-1, 1, b * a) / math.sqrt(a), rng.uniform(-0.1, 0.1, b)]
    return np.concatenate(parts).astype(np.float32)


def _samples(rows, seed):
    g = torch.Generator(DEV).manual_seed(seed + 4)
    X = torch.randn(rows, DIMS[0], device=DEV, generator=g)
    return X, torch.tanh(X[:, :DIMS[-1]] + 0.5 * torch.randn(rows, DIMS[-1], device=DEV, generator=g))


def _order(case, seed):
    """Sample order of each pass over the data (None: the whole batch as it is)."""
    if case["batch"] >= case["samples"]:
        return [None] * case["passes"]
    g = torch.Generator().manual_seed(seed + 5)
    return [torch.randperm(case["samples"], generator=g).to(DEV) for _ in range(case["passes"])]


# ---- one pass -------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("infer", "train"):
        net = pd.MLP(DIMS, seed=seed)
        net.set_params(_weights(seed))
        if kind == "infer":
            X, _ = _samples(case["batch"], seed)
            return {"case": case, "net": net, "X": X, "Y": torch.empty(case["batch"], DIMS[-1], device=DEV),
                    "Y16": torch.empty(case["batch"], DIMS[-1], device=DEV, dtype=torch.float16)}
        X, T = _samples(case["samples"], seed)
        return {"case": case, "net": net, "X": X, "T": T, "order": _order(case, seed),
                "loss": torch.zeros(1, device=DEV)}
    sc = _body(case)
    if kind == "build":  # nodes come in a mesh generator's order, not in ours
        p = np.random.default_rng(seed).permutation(sc.n)
        ctx = pd.Context(sc.x[p], sc.vol[p], sc.grain[p], sc.material, v0=sc.v0[p])
        ctx.set_walls(S.walls_array(sc.walls))
        return {"case": case, "ctx": ctx, "horizon": sc.horizon, "filters": sc.filters}
    # a representative volume fixes its kernel, as surrogate does; other runs leave the choice to the library
    fixed = {"lanes": 8, "tiles": -1} if case.get("record") else {}
    ctx = pd.Context.from_scenario(sc, precision=case.get("precision", "mixed"), **fixed)
    u0, v0 = _state(sc, seed)
    words = (ctx.B + 31) // 32
    st = {"case": case, "ctx": ctx, "dt": 0.8 * ctx.stable_dt(), "walls": S.walls_array(sc.walls),
          "moving": any(any(w.velocity) for w in sc.walls)}
    for name, values in (("u0", u0), ("v0", v0)):
        st[name] = _pinned(values.shape, torch.float64)
        st[name].copy_(torch.from_numpy(values))
    st["bits0"] = _pinned(words, torch.int32)
    planes = _crack_planes(case, sc, seed)
    if planes:
        rp, col = ctx.bonds()
        i = torch.repeat_interleave(torch.arange(sc.n, device=DEV), torch.from_numpy(np.diff(rp)).to(DEV))
        hit = torch.zeros(32 * words, dtype=torch.int64, device=DEV)
        hit[:ctx.B] = _cracked(planes, torch.from_numpy(sc.x).to(DEV), i, torch.from_numpy(col).to(DEV).long())
        packed = (hit.view(-1, 32) << torch.arange(32, device=DEV)).sum(1)
        st["bits0"].copy_((packed - ((packed >> 31) << 32)).to(torch.int32))
    for name, like in (("u", st["u0"]), ("v", st["v0"])):
        st[name] = _pinned(like.shape, torch.float64)
        st[name + "32"] = torch.zeros(like.shape, dtype=torch.float32)
    st["bits"] = _pinned(words, torch.int32)
    if case.get("record"):
        p = st["walls"][:, 3:6]
        L = np.array([p[1, 0] - p[0, 0], p[3, 1] - p[2, 1], p[5, 2] - p[4, 2]])
        st["areas"] = np.array([L[1] * L[2]] * 2 + [L[0] * L[2]] * 2 + [L[0] * L[1]] * 2)
    if kind == "coupled":  # the coupled program starts from this state and keeps it in its own buffers
        st["u"].copy_(st["u0"])
        st["v"].copy_(st["v0"])
        pd.pd_set_state_packed(ctx.h, st["u"].numpy(), st["v"].numpy(), st["bits"].numpy().view(np.uint32))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "infer":
        st["net"].forward_device(st["X"], st["Y"])
        return st["Y16"].copy_(st["Y"])
    if kind == "train":
        net, X, T = st["net"], st["X"], st["T"]
        for order in st["order"]:
            if order is None:
                net.train_step_device(X, T, 1e-3, st["loss"])
                continue
            for b0 in range(0, len(order), case["batch"]):
                idx = order[b0:b0 + case["batch"]]
                net.train_step_device(X.index_select(0, idx), T.index_select(0, idx), 1e-3, st["loss"])
        return {"loss": st["loss"], "weights": torch.from_numpy(net.get_params()).to(torch.float16)}
    ctx = st["ctx"]
    if kind == "build":
        ctx.build_bonds(st["horizon"], st["filters"])
        rowptr, col = ctx.bonds()
        return {"rowptr": rowptr, "col": col}
    u, v, bits = st["u"].numpy(), st["v"].numpy(), st["bits"].numpy().view(np.uint32)
    if kind == "coupled":
        pd.pd_set_state_packed(ctx.h, u, v, bits)
        ctx.step(st["dt"], 1)
    else:
        if st["moving"]:
            ctx.set_walls(st["walls"])
        pd.pd_set_state_packed(ctx.h, st["u0"].numpy(), st["v0"].numpy(), st["bits0"].numpy().view(np.uint32))
        ctx.step(st["dt"], case["steps"])
    out = {}
    if case.get("record"):
        sigma, _, _ = ctx.bulk_stress_mean(st["areas"])
        # the record holds the number of contacts (it varies with the state, the list's length with it)
        out = {"sigma": sigma.astype(np.float32), "damage": ctx.damage(), "contacts": len(ctx.contacts())}
    pd.pd_get_state_packed(ctx.h, ctx.n, ctx.B, u, v, bits)
    out["broken"] = st["bits"]
    for name in ("u", "v"):
        out[name] = st[name] if case.get("precision") == "fp64" else st[name + "32"].copy_(st[name])
    return out


# ---- what a pass cannot do without -----------------------------------------------
def _lattice(case):
    """(nodes, directed bonds) of a case's body on its undisturbed lattice."""
    kind = case["kind"]
    cells, copies = 3, 1
    if kind in ("crush", "build"):
        r = np.arange(-case["outer"], case["outer"] + 1)
        rr = r[:, None, None] ** 2 + r[None, :, None] ** 2 + r[None, None, :] ** 2
        m = (rr < case["outer"] ** 2) & (rr >= case["inner"] ** 2)
    elif kind in ("plate", "coupled"):
        cells, m = 4, np.ones((case["length"], case["height"], 9), bool)
    else:
        r = np.arange(-8, 9)
        p = np.rint(S.shape_particle(case["shape"], 1e-3, 1e-3 / 8) / (1e-3 / 8)).astype(int) + 8
        m = np.zeros((len(r),) * 3, bool)
        m[tuple(p.T)] = True
        copies = case["side"] ** 3
    bonds = 0
    c = np.arange(-cells, cells + 1)
    for a in c:
        for b in c:
            for d in c:
                if 0 < a * a + b * b + d * d < cells * cells:
                    lo = [slice(max(0, -s), m.shape[k] - max(0, s)) for k, s in enumerate((a, b, d))]
                    hi = [slice(max(0, s), m.shape[k] - max(0, -s)) for k, s in enumerate((a, b, d))]
                    bonds += int((m[tuple(lo)] & m[tuple(hi)]).sum())
    return copies * int(m.sum()), copies * bonds


def work(case):
    kind = case["kind"]
    if kind in ("infer", "train"):
        macs = sum(a * b for a, b in zip(DIMS[:-1], DIMS[1:]))
        params = macs + sum(DIMS[1:])
        if kind == "infer":
            return {"bytes": 4.0 * case["batch"] * (DIMS[0] + DIMS[-1]) + 4.0 * params, "flops": 2.0 * case["batch"] * macs}
        steps = case["passes"] * -(-case["samples"] // case["batch"])
        return {"bytes": 4.0 * case["passes"] * case["samples"] * (DIMS[0] + DIMS[-1]) + 24.0 * steps * params,
                "flops": case["passes"] * case["samples"] * 2.0 * (3 * macs - DIMS[0] * DIMS[1])}
    n, B = _lattice(case)
    if kind == "build":  # positions, volumes and grains in; rows and columns out
        return {"bytes": 36.0 * n + 8.0 * n + 4.0 * B, "flops": 8.0 * B}
    # a step: the neighbour index and broken bit of every directed bond, x, V, u, v, F and the row of every node;
    # some 46 operations for an undirected bond.  The state goes in and out once.
    steps = case.get("steps", 1)
    size = 2 if case.get("precision") == "fp64" else 1
    return {"bytes": steps * (4.125 * B + 170.0 * size * n) + 2.0 * (48.0 * n + B / 8.0), "flops": steps * 23.0 * B}


# ---- the same in 64 bits ---------------------------------------------------------
def _pairs(x, cut):
    """Ordered pairs (i, j), i != j, with |x_j - x_i| < cut (torch indices on x's device)."""
    cell = torch.floor((x - x.min(0).values) / (cut * (1 + 1e-9))).long() + 1
    dims = cell.max(0).values + 2
    key = (cell[:, 0] * dims[1] + cell[:, 1]) * dims[2] + cell[:, 2]
    order = torch.argsort(key)
    skey = key[order]
    out = []
    for a in (-1, 0, 1):
        for b in (-1, 0, 1):
            for d in (-1, 0, 1):
                want = key + (a * dims[1] + b) * dims[2] + d
                s, e = torch.searchsorted(skey, want), torch.searchsorted(skey, want, right=True)
                cnt = e - s
                i = torch.repeat_interleave(torch.arange(len(x), device=x.device), cnt)
                j = order[torch.arange(len(i), device=x.device) - torch.repeat_interleave(cnt.cumsum(0) - cnt - s, cnt)]
                d2 = (x[j] - x[i]).square()
                keep = (((d2[:, 0] + d2[:, 1]) + d2[:, 2]) < cut * cut) & (i != j)
                out.append(torch.stack([i[keep], j[keep]]))
    return torch.cat(out, 1)


def _filtered(sc, x, i, j):
    """Bonds that the notch and inner-sphere filters take out."""
    drop = torch.zeros(i.shape, dtype=torch.bool, device=x.device)
    for kind, a in sc.filters:
        if kind == S.FILTER_SPHERE:
            inside = (x - torch.tensor(a[:3], device=x.device, dtype=torch.float64)).square().sum(1) < a[3] ** 2
            drop |= inside[i] | inside[j]
        else:
            p, q = x[torch.minimum(i, j)], x[torch.maximum(i, j)]
            n = torch.tensor(a[:3], device=x.device, dtype=torch.float64)
            t = -(p @ n + a[3]) / ((q - p) @ n)
            at = p + t[:, None] * (q - p)
            lo, hi = (torch.tensor(a[k:k + 3], device=x.device, dtype=torch.float64) for k in (4, 7))
            box = (at >= lo).all(1) & (at <= hi).all(1)
            drop |= (t > 0) & (t < 1) & box
    return drop


def _steps64(case, seed):
    """u, v and the mean wall forces after the case's steps, in FP64.

    Contact is the spring between nodes of different grains: no two nodes of one grain come within R_c here."""
    sc = _body(case)
    m, f64 = sc.material, torch.float64
    x, V = torch.tensor(sc.x, device=DEV), torch.tensor(sc.vol, device=DEV)
    grain = torch.tensor(sc.grain, device=DEV)
    u, v = (torch.tensor(a, device=DEV) for a in _state(sc, seed))
    K, d = 2 * m.E / 3, sc.horizon
    c, s0, Kn = 18 * K / (math.pi * d ** 4), math.sqrt(5 * m.G0 / (9 * K * d)), m.contact_factor * 18 * K / (math.pi * d ** 5)
    i, j = _pairs(x, d)
    keep = (grain[i] == grain[j]) & ~_filtered(sc, x, i, j)
    i, j = i[keep], j[keep]
    xi = x[j] - x[i]
    L = xi.norm(dim=1)
    dt = 0.8 * float((2 * m.rho / torch.zeros_like(V).index_add_(0, i, V[j] * c / L)).sqrt().min())
    intact = ~_cracked(_crack_planes(case, sc, seed), x, i, j)
    Rc = m.contact_radius
    ci, cj = _pairs(x + u, 1.5 * Rc)
    other = grain[ci] != grain[cj]
    ci, cj = ci[other], cj[other]
    walls = S.walls_array(sc.walls)
    wn, wp, wv = (torch.tensor(walls[:, 3 * k:3 * k + 3], device=DEV) for k in range(3))
    impulse = torch.zeros(len(walls), 3, device=DEV, dtype=f64)

    def accel(wp):
        nonlocal intact
        y = xi + (u[j] - u[i])
        l = y.norm(dim=1)
        s = (l - L) / L
        intact = intact & ~(s > s0)
        F = torch.zeros_like(u).index_add_(0, i, torch.where(intact, c * s * V[j] / l, 0.0)[:, None] * y)
        e = (x[cj] - x[ci]) + (u[cj] - u[ci])
        dn = e.norm(dim=1)
        e = e / dn[:, None]
        g = -Kn * (Rc - dn) + m.beta_d * ((v[cj] - v[ci]) * e).sum(1)
        F.index_add_(0, ci, torch.where(dn < Rc, g * V[cj], 0.0)[:, None] * e)
        react = torch.zeros_like(impulse)
        for k in range(len(walls)):
            q = (x + u - wp[k]) @ wn[k]
            near = q < Rc
            q = q[near]
            cap = math.pi / 3 * (Rc - q) ** 2 * (2 * Rc + q)
            mag = Kn * (Rc - math.pi / 4 * (Rc * Rc - q * q) ** 2 / cap) * cap
            mag = mag + m.beta_d * ((wv[k] - v[near]) @ wn[k]) * cap
            F[near] += mag[:, None] * wn[k]
            react[k] = -(mag * V[near]).sum() * wn[k]
        return F / m.rho, react

    a, _ = accel(wp)
    for _ in range(case.get("steps", 1)):
        v = v + 0.5 * dt * a
        u = u + dt * v
        wp = wp + dt * wv
        a, react = accel(wp)
        impulse += dt * react
        v = v + 0.5 * dt * a
    return u, v, impulse / (dt * case.get("steps", 1)), wn


def _net64(theta, X):
    h, at, keep = X, 0, []
    for k, (a, b) in enumerate(zip(DIMS[:-1], DIMS[1:])):
        W, c = theta[at:at + a * b].view(b, a), theta[at + a * b:at + a * b + b]
        at += a * b + b
        z = h @ W.t() + c
        h = z if k == len(DIMS) - 2 else torch.nn.functional.gelu(z)
    return h


def exact(case, seed):
    kind = case["kind"]
    if kind == "build":
        return None  # lists of whole numbers
    if kind in ("infer", "train"):
        theta = torch.tensor(_weights(seed), device=DEV, dtype=torch.float64)
        if kind == "infer":
            return _net64(theta, _samples(case["batch"], seed)[0].double())
        X, T = (t.double() for t in _samples(case["samples"], seed))
        m1, m2, t = torch.zeros_like(theta), torch.zeros_like(theta), 0
        for order in _order(case, seed):
            for b0 in range(0, case["samples"], case["batch"]):
                idx = slice(None) if order is None else order[b0:b0 + case["batch"]]
                theta = theta.detach().requires_grad_(True)
                loss = (_net64(theta, X[idx]) - T[idx]).square().mean()
                g, = torch.autograd.grad(loss, theta)
                t += 1
                m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
                theta = theta - 1e-3 * (m1 / (1 - 0.9 ** t)) / ((m2 / (1 - 0.999 ** t)).sqrt() + 1e-8)
        return {"loss": loss.detach().view(1), "weights": theta.detach()}
    if case.get("mu", 0.0) > 0:
        return None  # friction: stick and slip part at the last bit
    u, v, R, wn = _steps64(case, seed)
    out = {"broken": None, "u": u, "v": v}
    if case.get("record"):
        p = S.walls_array(_body(case).walls)[:, 3:6]
        L = np.array([p[1, 0] - p[0, 0], p[3, 1] - p[2, 1], p[5, 2] - p[4, 2]])
        sig = torch.zeros(3, 3, device=DEV, dtype=torch.float64)
        for k in range(6):  # column of the wall's axis: its force over its area, outward normal -n
            a = k // 2
            sig[:, a] += R[k] * torch.sign(wn[k, a]) / (2 * L.prod() / L[a])
        sig = 0.5 * (sig + sig.t())
        sigma = torch.stack([sig[0, 0], sig[1, 1], sig[2, 2], sig[1, 2], sig[0, 2], sig[0, 1]])
        out = {"sigma": sigma, "damage": None, "contacts": None, **out}
    return out
