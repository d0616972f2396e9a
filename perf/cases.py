"""The work that users have this library do, as cases whose time and results can be compared.

Every case goes through the package's public entry points on inputs drawn on the GPU from
a seed: the density models of ``ics`` (Plummer sphere, NFW halo, Andromeda-like galaxy)
with analytic |a_old| and speeds near equilibrium.  The kinds of work:

  force      the whole force evaluation of one system: tree build, then every particle's force
  tree       the tree build alone (keys, sort, permutation, octree, pseudo j-particles)
  walk       forces of some of the particles on a tree that is there
  steps      a restart: load a checkpoint, take block steps, read the state back
  integrate  a caller-driven integration: prediction of all, correction of the active
  batch      one captured force evaluation of many independent systems
  serve      requests of several sizes through the continuous-batching server
  sort       the allocation-free sort of (key, value) pairs
"""
import ctypes
import math

import numpy as np
import torch

from paper_1610_07279_gb300 import gothic as g

MACS = {"angle": g.GT_MAC_OPENING_ANGLE, "acceleration": g.GT_MAC_ACCELERATION, "multipole": g.GT_MAC_MULTIPOLE}
CURVES = {"morton": g.GT_KEY_MORTON, "hilbert": g.GT_KEY_HILBERT}
EPS = {"plummer": 1.0 / 64.0, "nfw": 1.0 / 256.0, "galaxy": 0.01}
LEVELS = 8
T_RESTART = 11  # the restarts' clock: the next block steps are 12, 13, 14, 15 (levels >= 5, 7, >= 6, 7)
DIRECT_PAIRS = 1 << 37  # the largest direct sum in 64 bits that exact() makes


def listed():
    return [
        # the smallest system of the paper's accuracy study: 8192 particles, all active, every launch counts
        {"name": "force_plummer_8192", "kind": "force", "model": "plummer", "n": 8192, "leaf": 16, "group": 64,
         "mac": "acceleration", "curve": "morton"},
        # the rebuild of a mid-sized halo between block steps
        {"name": "tree_nfw_1m", "kind": "tree", "model": "nfw", "n": 1 << 20, "leaf": 16, "curve": "morton"},
        # the rebuild of the benchmark's galaxy, the largest tree
        {"name": "tree_galaxy_16m", "kind": "tree", "model": "galaxy", "n": 1 << 24, "leaf": 32, "curve": "morton"},
        # a step in which every particle is due, benchmark's leaf and group sizes: the start-up and the
        # longest block steps
        {"name": "walk_galaxy_4m_all", "kind": "walk", "model": "galaxy", "n": 1 << 22, "leaf": 32, "group": 64,
         "mac": "acceleration", "curve": "morton", "active": 1.0},
        # the commonest block step of the benchmark: only the finest level, 0.6 % of the particles, is due
        {"name": "walk_galaxy_16m_sparse", "kind": "walk", "model": "galaxy", "n": 1 << 24, "leaf": 32, "group": 32,
         "mac": "acceleration", "curve": "morton", "active": 0.006},
        # a tenth of a halo of ragged size with the opening-angle criterion (the bootstrap pass's)
        {"name": "walk_nfw_odd_angle", "kind": "walk", "model": "nfw", "n": 1000003, "leaf": 16, "group": 64,
         "mac": "angle", "curve": "morton", "active": 0.1},
        # three block steps of the halo from a checkpoint, automatic rebuild interval (the default)
        {"name": "steps_nfw_1m_auto", "kind": "steps", "model": "nfw", "n": 1 << 20, "leaf": 16, "group": 64,
         "rebuild": 0, "steps": 3},
        # four block steps of the benchmark's galaxy from a checkpoint, one rebuild in four steps
        {"name": "steps_galaxy_16m", "kind": "steps", "model": "galaxy", "n": 1 << 24, "leaf": 32, "group": 64,
         "rebuild": 4, "steps": 4},
        # a caller that computes its own forces: prediction of an odd number of particles, a third corrected
        {"name": "integrate_galaxy_12m_odd", "kind": "integrate", "model": "galaxy", "n": 12345677, "active": 0.3},
        # the benchmark's batch: 64 systems of 2^12 to 2^18 particles in one captured evaluation
        {"name": "batch_64", "kind": "batch", "count": 64, "lo": 12.0, "hi": 18.0, "sizes": 4, "leaf": 16, "group": 32},
        # a burst of requests to the server, a few block steps each
        {"name": "serve_12", "kind": "serve", "count": 12, "lo": 12.0, "hi": 17.0, "sizes": 5, "steps": 6},
        # the allocation-free sort near its largest size, for callers inside another memory budget
        {"name": "sort_1m_odd", "kind": "sort", "n": 1000001, "bits": 63},
    ]


def _log_size(rng, lo, hi):
    """A size spread over the logarithm of [2^lo, 2^hi]; mostly odd or ragged, now and then a power of two."""
    x = rng.uniform(lo, hi)
    return 1 << round(x) if rng.random() < 0.2 else max(2, int(2.0 ** x))


def draw(rng):
    kind = rng.choice(["force", "force", "tree", "tree", "walk", "walk", "walk", "steps", "steps", "integrate",
                       "batch", "serve", "sort"])
    model = rng.choice(["plummer", "nfw", "galaxy"])
    leaf = rng.choice([8, 16, 16, 20, 24, 32, 32])
    group = rng.choice([16, 32, 32, 64, 64])
    mac = rng.choice(["acceleration"] * 4 + ["angle", "multipole"])
    curve = rng.choice(["morton"] * 4 + ["hilbert"])
    if kind == "force":
        return {"kind": kind, "model": model, "n": _log_size(rng, 10, 18), "leaf": leaf, "group": group, "mac": mac,
                "curve": curve}
    if kind == "tree":
        return {"kind": kind, "model": model, "n": _log_size(rng, 12, 23), "leaf": leaf, "curve": curve}
    if kind == "walk":
        return {"kind": kind, "model": model, "n": _log_size(rng, 14, 21.5), "leaf": leaf, "group": group, "mac": mac,
                "curve": curve, "active": round(10.0 ** rng.uniform(-2.5, 0.0), 4)}
    if kind == "steps":
        return {"kind": kind, "model": model, "n": _log_size(rng, 12, 21), "leaf": leaf, "group": group,
                "rebuild": rng.choice([0, 4]), "steps": rng.randint(1, 3)}
    if kind == "integrate":
        return {"kind": kind, "model": model, "n": _log_size(rng, 14, 23), "active": round(10.0 ** rng.uniform(-2.5, 0.0), 4)}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(4, 64), "lo": 11.0, "hi": round(rng.uniform(13.0, 17.0), 2),
                "sizes": rng.randrange(1 << 20), "leaf": leaf, "group": rng.choice([16, 32])}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(2, 12), "lo": 11.0, "hi": round(rng.uniform(12.0, 16.0), 2),
                "sizes": rng.randrange(1 << 20), "steps": rng.randint(2, 6)}
    return {"kind": "sort", "n": _log_size(rng, 10, 20), "bits": rng.choice([24, 45, 63, 63])}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _uniform(gen, n, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)


def _isotropic(gen, n):
    cth, phi = _uniform(gen, n, -1.0, 1.0), _uniform(gen, n, 0.0, 2.0 * math.pi)
    sth = torch.sqrt(torch.clamp(1.0 - cth * cth, min=0.0))
    return torch.stack([sth * torch.cos(phi), sth * torch.sin(phi), cth], 1)


def _interp(x, xp, fp):
    xp, fp = torch.as_tensor(xp, device="cuda"), torch.as_tensor(fp, device="cuda")
    k = torch.clamp(torch.searchsorted(xp, x.contiguous()), 1, xp.numel() - 1)
    w = torch.clamp((x - xp[k - 1]) / (xp[k] - xp[k - 1]), 0.0, 1.0)
    return fp[k - 1] + w * (fp[k] - fp[k - 1])


def _nfw_mass(rs, rt):
    """(r, M(<r)/M) of an NFW halo tapered exponentially beyond rt."""
    r = np.geomspace(1e-5 * rs, rt + 16.0 * rs, 1 << 14)
    rho = 1.0 / ((r / rs) * (1.0 + r / rs) ** 2) * np.where(r > rt, np.exp(-(r - rt) / rs), 1.0)
    shell = 4.0 * math.pi * r * r * rho
    m = np.concatenate([[0.0], np.cumsum(0.5 * (shell[1:] + shell[:-1]) * np.diff(r))])
    m += 2.0 * math.pi * rs * r[0] ** 2
    m[0] = 0.0
    return r, m / m[-1]


def _sample(model, n, seed):
    """Positions (n x 3, FP32 values in FP64), velocities, masses and analytic |a| of one system, in random order."""
    gen = _gen(seed)
    if model == "plummer":
        u = _uniform(gen, n, 1e-10, 1.0 - 1e-10)
        r = torch.clamp(1.0 / torch.sqrt(u ** (-2.0 / 3.0) - 1.0), max=100.0)
        pos = r[:, None] * _isotropic(gen, n)
        enclosed = lambda q: (q * q / (1.0 + q * q)) ** 1.5  # noqa: E731
        spin = None
    elif model == "nfw":
        tr, tm = _nfw_mass(1.0, 10.0)
        r = _interp(_uniform(gen, n), tm, tr)
        pos = r[:, None] * _isotropic(gen, n)
        enclosed = lambda q: _interp(q, tr, tm)  # noqa: E731
        spin = None
    else:  # Hernquist bulge 3 %, exponential disk 5 %, NFW halo 92 %
        nb, nd = round(0.03 * n), round(0.05 * n)
        nh = n - nb - nd
        tr, tm = _nfw_mass(7.6, 200.0)
        s = torch.sqrt(_uniform(gen, nb) * (200.0 / 200.6) ** 2)
        bulge = (0.6 * s / (1.0 - s))[:, None] * _isotropic(gen, nb)
        rad = torch.clamp(-5.4 * torch.log(_uniform(gen, nd, 1e-12) * _uniform(gen, nd, 1e-12)), max=200.0)
        phi = _uniform(gen, nd, 0.0, 2.0 * math.pi)
        z = 0.6 * torch.atanh(torch.clamp(2.0 * _uniform(gen, nd) - 1.0, -0.999999, 0.999999))
        disk = torch.stack([rad * torch.cos(phi), rad * torch.sin(phi), z], 1)
        halo = _interp(_uniform(gen, nh), tm, tr)[:, None] * _isotropic(gen, nh)
        pos = torch.cat([bulge, disk, halo])
        spin = (nb, nd, phi)

        def enclosed(q):
            return (0.03 * (q / (q + 0.6)) ** 2 + 0.05 * (1.0 - (1.0 + q / 5.4) * torch.exp(-q / 5.4))
                    + 0.92 * _interp(q, tr, tm))
    pos = (pos - pos.mean(0)).float().double().contiguous()
    q = torch.linalg.vector_norm(pos, dim=1)
    mass_in = enclosed(q)
    speed = torch.sqrt(mass_in / torch.clamp(q, min=1e-6))
    vel = (speed / math.sqrt(3.0))[:, None] * torch.randn((n, 3), generator=gen, device="cuda", dtype=torch.float64)
    if spin is not None:
        nb, nd, phi = spin
        d = slice(nb, nb + nd)
        vel[d] *= 0.15
        vel[d, 0] -= speed[d] * torch.sin(phi)
        vel[d, 1] += speed[d] * torch.cos(phi)
    eps = EPS[model]
    aold = (mass_in * q / (q * q + eps * eps) ** 1.5 + 1e-12).float()
    mass = torch.full((n,), 1.0 / n, dtype=torch.float32, device="cuda")
    return pos, vel.contiguous(), mass, aold.contiguous()


def _params(case, **more):
    p = g.gt_default_params()
    p.eps = EPS[case.get("model", "plummer")]
    p.leaf_max = case.get("leaf", 16)
    p.group_max = case.get("group", 64)
    p.group_mode = g.GT_GROUP_CELLS  # one size for all: the sizes tuned on line depend on the run's times
    p.mac = MACS[case.get("mac", "acceleration")]
    if p.mac == g.GT_MAC_MULTIPOLE:
        p.delta_acc = 2.0 ** -8  # Delta_mul
    p.key_curve = CURVES[case.get("curve", "morton")]
    p.levels = LEVELS
    for k, v in more.items():
        setattr(p, k, v)
    return p


def _empty(shape, dtype):
    return torch.empty(shape, dtype=dtype, device="cuda")


def _ids(s):
    ids = _empty(s.n, torch.int32)
    s.get_state({"id": ids})
    return ids.long()


def _key_order(pos, vel, mass, aold):
    """The arrays of a system in key order: a checkpoint is written in that order."""
    k = torch.sort(_keys64(pos, "morton"), stable=True)[1]
    return pos[k].contiguous(), vel[k].contiguous(), mass[k].contiguous(), aold[k].contiguous()


def _levels(aold, eps, eta):
    """(dt_max, level, t0) of particles with these |a|, as a run at tick T_RESTART holds them."""
    dt = torch.sqrt(2.0 * eta * eps / aold.double())
    dt_max = 2.0 ** math.floor(math.log2(float(dt.max())))
    level = torch.clamp(torch.ceil(torch.log2(dt_max / dt)), 0, LEVELS - 1).long()
    span = 2 ** (LEVELS - 1 - level)
    t0 = T_RESTART - T_RESTART % span
    return dt_max, level.to(torch.uint8).contiguous(), t0.contiguous()


def _chosen(aold, share):
    """The share of the particles with the largest |a| (the finest levels), as a rising list of indices."""
    n = aold.numel()
    k = max(1, min(n, round(share * n)))
    on = torch.zeros(n, dtype=torch.bool, device="cuda")
    on[torch.topk(aold, k).indices] = True
    return torch.nonzero(on).flatten().int().contiguous()


def _sort_keys(case, seed):
    keys = torch.randint(0, 1 << 62, (case["n"],), generator=_gen(seed), device="cuda", dtype=torch.int64)
    keys = (keys << 1 | keys >> 61 & 1) & ((1 << 63) - 1)
    return (keys >> (63 - case["bits"])).contiguous()


def _own_forces(case, pos, aold):
    """A caller's active list and its own (central, analytic) forces on it."""
    active = _chosen(aold, case["active"])
    rows = active.long()
    r = torch.linalg.vector_norm(pos[rows], dim=1, keepdim=True)
    acc = torch.cat([-pos[rows] / torch.clamp(r, min=1e-6) * aold[rows, None], -1.0 / (1.0 + r)], 1)
    return active, acc.float().contiguous()


def _sizes(case):
    rng = np.random.default_rng(case["sizes"])
    n = np.rint(2.0 ** rng.uniform(case["lo"], case["hi"], case["count"])).astype(int)
    return [int(v) for v in n], ["plummer" if c < 0.5 else "nfw" for c in rng.uniform(0.0, 1.0, case["count"])]


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("force", "tree", "walk"):
        n = case["n"]
        pos, vel, mass, aold = _sample(case["model"], n, seed)
        s = g.System(n, _params(case))
        s.set_state(pos, vel, mass)
        st["s"] = s
        if kind == "tree":
            cap = n + 2048  # of the caller's cell arrays, zeroed behind the last cell
            st.update(keys=_empty(n, torch.int64), order=_empty(n, torch.int32), cap=cap,
                      jpos=torch.zeros((cap, 4), dtype=torch.float32, device="cuda"))
        else:
            s.build_tree()
            st["aold"] = aold[_ids(s)].contiguous()
            st["active"] = None if case.get("active", 1.0) >= 1.0 else _chosen(st["aold"], case["active"])
            st["acc"] = _empty((n if st["active"] is None else st["active"].numel(), 4), torch.float32)
    elif kind == "steps":
        n = case["n"]
        pos, vel, mass, aold = _key_order(*_sample(case["model"], n, seed))
        p = _params(case, rebuild_every=case["rebuild"])
        dt_max, level, t0 = _levels(aold, p.eps, p.eta)
        st.update(s=g.System(n, p), pos=pos, vel=vel, mass=mass, aold=aold, level=level, t0=t0, dt_max=dt_max,
                  out={"pos": _empty((n, 3), torch.float64), "vel": _empty((n, 3), torch.float64),
                       "acc": _empty((n, 4), torch.float32), "aold": _empty(n, torch.float32),
                       "id": _empty(n, torch.int32)})
    elif kind == "integrate":
        n = case["n"]
        pos, vel, mass, aold = _key_order(*_sample(case["model"], n, seed))
        p = _params(case)
        dt_max, level, t0 = _levels(aold, p.eps, p.eta)
        s = g.System(n, p)
        s.set_state(pos, vel, mass)
        s.set_integrator_state(level, t0, aold, None, dt_max, T_RESTART)
        active, acc = _own_forces(case, pos, aold)
        st.update(s=s, active=active, acc=acc, T=T_RESTART,
                  posm=_empty((n, 4), torch.float32),
                  out={"pos": _empty((n, 3), torch.float64), "vel": _empty((n, 3), torch.float64),
                       "aold": _empty(n, torch.float32), "level": _empty(n, torch.uint8),
                       "t0": _empty(n, torch.int64)})
    elif kind == "batch":
        ns, models = _sizes(case)
        b = g.Batch(ns, [_params({**case, "model": m}) for m in models])
        keep = []
        for k, (n, m) in enumerate(zip(ns, models)):
            pos, vel, mass, aold = _sample(m, n, seed * 1000 + k)
            dt_max, level, t0 = _levels(aold, EPS[m], b.params[k].eta)
            torch.cuda.synchronize()  # the members run on the batch's own stream
            b.systems[k].set_state(pos, vel, mass)
            b.systems[k].set_integrator_state(level, t0, aold, None, dt_max, T_RESTART)
            keep.append((pos, vel, mass, aold, level, t0))
        b.sync()
        b.capture()
        b.launch()  # the members' particles take their key order
        b.sync()
        st.update(b=b, acc=[_empty((n, 4), torch.float32) for n in ns], ids=[_empty(n, torch.int32) for n in ns])
    elif kind == "serve":
        ns, models = _sizes(case)
        st["srv"] = g.Server(40 * 10**9, max_slots=16, walk_queue=8192)
        st["req"] = []
        for k, (n, m) in enumerate(zip(ns, models)):
            pos, vel, mass, _ = _sample(m, n, seed * 1000 + k)
            p = _params({"model": m, "group": 32}, rebuild_every=4, walk_queue=8192)
            st["req"].append((pos.cpu().numpy(), vel.cpu().numpy(), mass.cpu().numpy(), p,
                              np.empty((n, 3)), np.empty((n, 3))))
    else:
        n = case["n"]
        st.update(src=_sort_keys(case, seed), keys=_empty(n, torch.int64), vals=_empty(n, torch.int32),
                  index=torch.arange(n, dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    kind = st["case"]["kind"]
    if kind in ("force", "walk"):
        if kind == "force":
            st["s"].build_tree()
        st["s"].accel_active(st["active"], st["aold"], st["acc"])
        return {"acc": st["acc"]}
    if kind == "tree":
        s = st["s"]
        s.build_tree()
        nn = ctypes.c_int64(st["cap"])
        rc = g.load().gt_get_tree(s._h, st["keys"].data_ptr(), st["order"].data_ptr(), None, st["jpos"].data_ptr(),
                                  None, ctypes.byref(nn), torch.cuda.current_stream().cuda_stream)
        if rc != g.GT_OK:
            raise g.GothicError(rc, "gt_get_tree")
        return {"keys": st["keys"], "order": st["order"], "jpos": st["jpos"]}
    if kind == "steps":
        s = st["s"]
        s.set_state(st["pos"], st["vel"], st["mass"])
        s.set_integrator_state(st["level"], st["t0"], st["aold"], None, st["dt_max"], T_RESTART)
        for _ in range(st["case"]["steps"]):
            s.block_step()
        o = s.get_state(st["out"])
        # snapshots hold FP32, as N-body snapshot formats do
        return {"pos": o["pos"].float(), "vel": o["vel"].float(), "acc": o["acc"], "aold": o["aold"], "id": o["id"]}
    if kind == "integrate":
        s = st["s"]
        st["T"] += 1 << (LEVELS - 1)
        s.predict(st["T"], st["posm"])
        s.correct(st["active"], st["acc"], st["T"])
        return {"posm": st["posm"], **s.get_state(st["out"])}
    if kind == "batch":
        b = st["b"]
        b.launch()
        for k, (acc, ids) in enumerate(zip(st["acc"], st["ids"])):
            b.get_acc(k, acc, ids)
        return {"acc": torch.cat(st["acc"]), "id": torch.cat(st["ids"])}
    if kind == "serve":
        srv, todo = st["srv"], {}
        waiting = list(range(len(st["req"])))
        while waiting or todo:
            while waiting:
                pos, vel, mass, p, _, _ = st["req"][waiting[0]]
                t = srv.submit(pos, vel, mass, p, st["case"]["steps"])
                if t is None:
                    break
                todo[t] = waiting.pop(0)
            for t in list(todo):
                if srv.poll(t, *st["req"][todo[t]][4:]):
                    del todo[t]
        return {"pos": np.concatenate([r[4] for r in st["req"]]).astype(np.float32),
                "vel": np.concatenate([r[5] for r in st["req"]]).astype(np.float32)}
    st["keys"].copy_(st["src"])
    st["vals"].copy_(st["index"])
    g.gt_sort_pairs_noalloc(st["keys"], st["vals"], st["case"]["n"])
    return {"keys": st["keys"], "vals": st["vals"]}


# ------------------------------------------------------------------ the work of a pass
def _walk_work(n, na):
    """20 operations for each of ~34 log2(n) interactions of a particle (what the acceleration criterion at
    Delta_acc = 2^-7 needs on these models)."""
    return 20.0 * 34.0 * math.log2(max(n, 2)) * na


def work(case):
    kind = case["kind"]
    n = case.get("n", 0)
    tree = 16.0 * n + 85.0 * n * 2 + 12.0 * n + 48.0 * n / 8  # positions, the state in and out, keys and order, cells
    if kind == "tree":
        return {"bytes": tree, "flops": 0.0}
    if kind == "force":
        return {"bytes": tree + 20.0 * n, "flops": _walk_work(n, n)}
    if kind == "walk":
        na = case["active"] * n
        return {"bytes": 16.0 * n + 32.0 * n / 8 + 40.0 * na, "flops": _walk_work(n, na)}
    if kind == "steps":
        due = {1: 0.04, 2: 0.05, 3: 0.08, 4: 0.09}[case["steps"]] * n  # i-particles of the steps together
        load = 2 * (52.0 + 13.0) * n + 2 * 84.0 * n
        return {"bytes": load + tree + 76.0 * n * case["steps"] + 110.0 * due, "flops": _walk_work(n, due)}
    if kind == "integrate":
        return {"bytes": 76.0 * n + 61.0 * n + 150.0 * case["active"] * n, "flops": 6.0 * n + 40.0 * case["active"] * n}
    if kind in ("batch", "serve"):
        ns = _sizes(case)[0]
        evals = 1 if kind == "batch" else 2 + 0.1 * case["steps"]
        io = 20 if kind == "batch" else 100
        return {"bytes": sum(250.0 * v * evals + io * v for v in ns), "flops": evals * sum(_walk_work(v, v) for v in ns)}
    return {"bytes": 2 * 24.0 * n, "flops": 0.0}


# ------------------------------------------------------------------ the same in 64 bits
def _direct(pos, mass, eps, rows):
    """Eq. (1) in 64 bits for the given rows: acceleration and potential, j = i left out of the potential."""
    out = _empty((rows.numel(), 4), torch.float64)
    m = mass.double()
    step = max(1, (1 << 25) // pos.shape[0])
    for a in range(0, rows.numel(), step):
        x = pos[rows[a:a + step]]
        r2 = torch.full((x.shape[0], pos.shape[0]), eps * eps, dtype=torch.float64, device="cuda")
        for c in range(3):
            r2 += (pos[None, :, c] - x[:, None, c]) ** 2
        r2.rsqrt_()
        out[a:a + step, 3] = m[rows[a:a + step]] / eps - r2 @ m
        w = r2 * r2 * r2 * m[None, :]
        out[a:a + step, :3] = w @ pos - x * w.sum(1, keepdim=True)
    return out


def _keys64(pos, curve):
    lo = pos.min(0).values
    side = (pos.max(0).values - lo).max()
    q = torch.clamp(torch.floor((pos - lo) * (float(1 << 21) / side)), max=float((1 << 21) - 1)).long()
    x = [q[:, c].clone() for c in range(3)]
    if curve == "hilbert":  # Skilling's transpose
        for b in range(20, 0, -1):
            p = (1 << b) - 1
            for c in range(3):
                on = (x[c] >> b & 1).bool()
                t = torch.where(on, torch.zeros_like(x[0]), (x[0] ^ x[c]) & p)
                if c == 0:
                    x[0] = torch.where(on, x[0] ^ p, x[0])
                else:
                    x[0] = torch.where(on, x[0] ^ p, x[0] ^ t)
                    x[c] = x[c] ^ t
        x[1] ^= x[0]
        x[2] ^= x[1]
        t = torch.zeros_like(x[0])
        for b in range(20, 0, -1):
            t = torch.where((x[2] >> b & 1).bool(), t ^ ((1 << b) - 1), t)
        x = [v ^ t for v in x]
    key = torch.zeros_like(x[0])
    for b in range(21):
        for c in range(3):
            key |= (x[c] >> b & 1) << (3 * b + 2 - c)
    return key


def _exact_tree(case, seed):
    pos, _, mass, _ = _sample(case["model"], case["n"], seed)
    keys, order = torch.sort(_keys64(pos, case["curve"]), stable=True)
    x, m = pos[order], mass[order].double()
    terms = torch.cat([m[:, None], m[:, None] * x], 1)
    cells, above = [], None
    for level in range(22):
        prefix = keys >> (3 * (21 - level))
        new = torch.ones_like(keys, dtype=torch.bool)
        new[1:] = prefix[1:] != prefix[:-1]
        cell = torch.cumsum(new, 0) - 1
        count = torch.bincount(cell)
        keep = torch.ones_like(count, dtype=torch.bool) if above is None else above[new] > case["leaf"]
        sums = torch.zeros((count.numel(), 4), dtype=torch.float64, device="cuda").index_add_(0, cell, terms)[keep]
        cells.append(torch.cat([sums[:, 1:] / sums[:, :1], sums[:, :1]], 1))
        above = count[cell]
        if not bool((above > case["leaf"]).any()):
            break
    jpos = torch.zeros((case["n"] + 2048, 4), dtype=torch.float64, device="cuda")
    cells = torch.cat(cells)
    jpos[:cells.shape[0]] = cells
    return {"keys": keys, "order": order.int(), "jpos": jpos}


def _exact_integrate(case, seed):
    pos, vel, mass, aold = _key_order(*_sample(case["model"], case["n"], seed))
    p = _params(case)
    dt_max, level, t0 = _levels(aold, p.eps, p.eta)
    level = level.long()
    T, tick = T_RESTART + (1 << (LEVELS - 1)), dt_max * 2.0 ** -(LEVELS - 1)
    dt = ((T - t0).double() * tick)[:, None]
    posm = torch.cat([pos + dt * vel, mass.double()[:, None]], 1)
    active, acc = _own_forces(case, pos, aold)
    rows, a = active.long(), acc[:, :3].double()
    a2 = (a * a).sum(1)
    pos, vel, aold, t0 = pos.clone(), vel.clone(), aold.double(), t0.clone()
    pos[rows] += dt[rows] * vel[rows]
    vel[rows] += (dt_max * 2.0 ** -(level[rows] + 1).double())[:, None] * a
    want = torch.clamp(torch.ceil(torch.log2(dt_max / torch.sqrt(2.0 * p.eta * p.eps / torch.sqrt(a2)))), 0, LEVELS - 1).long()
    old = level[rows]
    longer = (want < old) & (T % (2 ** (LEVELS - old)) == 0)
    now = torch.where(want > old, want, torch.where(longer, old - 1, old))
    vel[rows] += (dt_max * 2.0 ** -(now + 1).double())[:, None] * a
    level[rows], t0[rows], aold[rows] = now, T, torch.sqrt(a2)
    return {"posm": posm, "pos": pos, "vel": vel, "aold": aold, "level": level, "t0": t0}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("force", "walk"):
        share = case.get("active", 1.0)
        if case["n"] * max(1.0, share * case["n"]) > DIRECT_PAIRS:
            return None
        pos, _, mass, aold = _sample(case["model"], case["n"], seed)
        order = torch.sort(_keys64(pos, case["curve"]), stable=True)[1]
        pos, aold = pos[order].contiguous(), aold[order].contiguous()
        rows = torch.arange(case["n"], device="cuda") if share >= 1.0 else _chosen(aold, share).long()
        return {"acc": _direct(pos, mass, EPS[case["model"]], rows)}
    if kind == "tree":
        return _exact_tree(case, seed)
    if kind == "integrate":
        return _exact_integrate(case, seed)
    if kind == "batch":
        ns, models = _sizes(case)
        if sum(n * n for n in ns) > DIRECT_PAIRS:
            return None
        acc, ids = [], []
        for k, (n, m) in enumerate(zip(ns, models)):
            pos, _, mass, _ = _sample(m, n, seed * 1000 + k)
            order = torch.sort(_keys64(pos, "morton"), stable=True)[1]
            acc.append(_direct(pos[order].contiguous(), mass, EPS[m], torch.arange(n, device="cuda")))
            ids.append(order.int())
        return {"acc": torch.cat(acc), "id": torch.cat(ids)}
    if kind == "sort":
        keys, order = torch.sort(_sort_keys(case, seed), stable=True)
        return {"keys": keys, "vals": order.int()}
    return None  # the truth of block steps through a tree has no direct sum that small
