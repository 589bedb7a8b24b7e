"""Performance cases of the DEM library: what its users run, through its public calls.

Scenes are stepped through ``Scene.step``, read back with ``get_state_into``, ``stats`` and
``contacts``, batched as sub-scenes, or sent to ``Server``; bare configurations go through
``find_pairs``.  Sizes are those of the repository's workloads (1000-sphere deposition, 500 to
50,000-sphere sweeps, 300,000- and million-sphere compactions, triaxial loading).

Sphere packings are made here, without the library: a small periodic cell is relaxed by
descending the overlap energy, tiled to the size asked for, disturbed a little, and numbered at
random, so that neighbours in space have unrelated ids (as spheres of a random placement do).
``exact`` restates a scene's steps in plain FP64 torch.
"""
import math

import numpy as np
import torch

import paper_2301_00611_gb300 as dem
from paper_2301_00611_gb300.dem import find_pairs

RHO, YOUNG, NU, DT_FACTOR = 2600.0, 5e7, 0.25, 0.5


def listed():
    base = {"precision": "fp64", "law": "linear", "phi": 0.64, "radii": "uniform", "speed": 0.02,
            "damping": 0.2, "friction": 0.5, "shear": False, "servo": False, "tstep": False}
    return [
        # the contact set of a small assembly, asked for by an analysis script
        {"name": "pairs_3k", "kind": "pairs", "n": 3001, "phi": 0.62, "radii": "uniform", "margin": 0.0},
        # the same of a million spheres: a packing's contact network, or another code's collider
        {"name": "pairs_1m", "kind": "pairs", "n": 1000000, "phi": 0.62, "radii": "lognormal", "margin": 0.0},
        # a script that looks at the statistics after every step of a 20,000-sphere scene
        dict(base, name="monitor_20k", kind="monitor", n=20000, steps=1),
        # the tutorial's deposition: 1000 spheres in a walled box, 100 steps between two looks
        dict(base, name="deposition_1k", kind="box", n=1000, steps=100, phi=0.3, radii="coarse", speed=0.5),
        # the headline job in its dense part: a million spheres, FP64
        dict(base, name="dense_1m_fp64", kind="periodic", n=1000000, steps=100, radii="lognormal", phi=0.63),
        # the same job in mixed precision
        dict(base, name="dense_1m_mixed", kind="periodic", n=1000000, steps=400, radii="lognormal", phi=0.63,
             precision="mixed"),
        # triaxial loading under the stress servo, the largest scene
        dict(base, name="triax_2m_mixed", kind="periodic", n=2000000, steps=300, precision="mixed", servo=True),
        # simple shear of a Hertz-Mindlin packing with the stiffness time stepper
        dict(base, name="shear_hertz_100k", kind="periodic", n=100003, steps=50, law="hertz", shear=True, tstep=True),
        # a parameter sweep: 64 walled depositions of 500 to 50,000 spheres advanced together
        dict(base, name="batch_64_mixed", kind="batch", n=64, steps=100, nmin=500, nmax=50000, phi=0.3,
             radii="coarse", speed=0.5, precision="mixed"),
        # fast, loose granular flow: the collider runs every few tens of steps
        dict(base, name="flow_300k", kind="periodic", n=300000, steps=100, phi=0.3, speed=2.0, damping=0.0,
             friction=0.1),
        # a checkpoint of a running job: one step, then the state and every contact with its history
        dict(base, name="checkpoint_100k", kind="checkpoint", n=100000, steps=1),
        # requests of several users served together (FP64), each submitted whole and read back whole
        dict(base, name="served_16", kind="served", n=16, steps=200, nmin=1000, nmax=10000, phi=0.3,
             radii="coarse", speed=0.5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pairs", "monitor", "box", "box", "periodic", "periodic", "periodic", "batch", "checkpoint",
                       "served"])
    if kind == "pairs":
        return {"kind": kind, "n": _log(rng, 1000, 1000000), "phi": rng.choice([0.3, 0.62]),
                "radii": rng.choice(["uniform", "lognormal"]), "margin": rng.choice([0.0, 1e-4])}
    c = {"kind": kind, "precision": rng.choice(["fp64", "mixed"]), "law": rng.choice(["linear", "linear", "hertz"]),
         "phi": rng.choice([0.3, 0.63]), "radii": rng.choice(["uniform", "lognormal"]),
         "damping": rng.choice([0.2, 0.4]), "friction": rng.uniform(0.2, 0.7), "shear": False, "servo": False,
         "tstep": False}
    c["speed"] = rng.choice([0.02, 0.2] if c["phi"] > 0.5 else [0.2, 2.0])
    if kind in ("batch", "served"):
        c.update(n=rng.randrange(4, 65) if kind == "batch" else rng.randrange(2, 17), steps=rng.randrange(40, 101),
                 nmin=500, nmax=rng.choice([5000, 20000]), phi=0.3, radii="coarse", speed=0.5, law="linear")
        if kind == "served":
            c["precision"] = "fp64"
    elif kind == "box":
        c.update(n=_log(rng, 500, 200000), steps=rng.randrange(20, 101), radii="coarse",
                 phi=0.3, speed=0.5, tstep=rng.random() < 0.2)
    elif kind in ("monitor", "checkpoint"):
        c.update(n=_log(rng, 1000, 100000), steps=1, phi=0.63, speed=0.02)
    else:
        c.update(n=_log(rng, 3000, 1000000), steps=rng.randrange(20, 101), shear=rng.random() < 0.3,
                 tstep=rng.random() < 0.2)
        c["servo"] = not c["shear"] and c["phi"] > 0.5 and rng.random() < 0.3
    return c


# ------------------------------------------------------------------ inputs
def _radii(kind, n, rng):
    if kind == "lognormal":   # the compaction's grading
        return np.clip(rng.lognormal(math.log(1e-3), 0.25, n), 0.5e-3, 2e-3)
    lo, hi = (9e-3, 11e-3) if kind == "coarse" else (0.8e-3, 1.2e-3)
    return rng.uniform(lo, hi, n)


def _cell(n, phi, radii, rng):
    """n spheres in a periodic cube at solid fraction phi, relaxed down the energy of linear
    contacts: (positions, radii, edge).  Dense: a jammed network; loose: no overlaps."""
    r = _radii(radii, n, rng)
    L = float((np.sum(4 / 3 * np.pi * r ** 3) / phi) ** (1 / 3))
    x = torch.from_numpy(rng.uniform(0, 1, (n, 3))).float().cuda()
    rr = torch.from_numpy(r / L).float().cuda()
    R = rr[:, None] + rr[None, :]
    K = rr[:, None] * rr[None, :] / R * (2.0 / rr.mean())
    K.fill_diagonal_(0.0)
    for _ in range(400 if phi > 0.5 else 80):
        d = [x[:, None, k] - x[None, :, k] for k in range(3)]
        d = [q - torch.round(q) for q in d]
        l = torch.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]).clamp_min_(1e-9)
        f = K * (R - l).clamp_min_(0.0) / l
        x = x + 0.3 * torch.stack([(f * q).sum(1) for q in d], 1)
    return np.mod(x.double().cpu().numpy(), 1.0) * L, r, L


def _tile(cell, n, k, rng):
    """The cell repeated k[0] x k[1] x k[2] times, cut to n spheres, disturbed and renumbered."""
    x, r, L = cell
    off = np.stack(np.meshgrid(*[np.arange(q) for q in k], indexing="ij"), -1).reshape(-1, 3) * L
    X = (x[None] + off[:, None]).reshape(-1, 3)
    R = np.broadcast_to(r, (len(off), len(r))).reshape(-1)
    at = rng.permutation(len(R))[:n]
    X, R = X[at], R[at]
    return X + rng.uniform(-1e-3, 1e-3, X.shape) * R[:, None], R.copy(), np.asarray(k) * L


class Spheres:
    """A scene's input as the library's classes take it (the fields of a workload)."""

    class Mat:
        def __init__(self, friction, young):
            self.density, self.young, self.poisson, self.friction = RHO, young, NU, friction

    def __init__(self, pos, radius, edge, periodic, case, rng, young=YOUNG, friction=None):
        n = len(radius)
        self.pos, self.radius, self.periodic, self.n = pos, radius, periodic, n
        self.mat_id = np.zeros(n, np.int32)
        self.materials = [self.Mat(case["friction"] if friction is None else friction, young)]
        self.cell, self.damping, self.gravity = np.diag(edge), case["damping"], np.zeros(3)
        self.box_lo, self.box_hi, self.wall_mask = np.zeros(3), np.asarray(edge, float), 0
        self.vel = rng.normal(0, case["speed"] / 2, (n, 3))
        self.angvel = rng.normal(0, 0.2 * case["speed"] / radius.mean(), (n, 3))
        self.velgrad = np.zeros((3, 3))
        self.dt = DT_FACTOR * radius.min() * math.sqrt(RHO / young)
        if periodic:
            # loading at constant volume, so that passes go on meeting the same kind of packing
            self.velgrad = np.diag([1.0, 1.0, -2.0])
        else:   # walls just touching the outermost spheres; the cloud falls onto the floor
            self.box_lo = -0.995 * radius.max() * np.ones(3)
            self.box_hi = np.asarray(edge, float) + 0.995 * radius.max()
            self.wall_mask, self.gravity = 0x3F, np.array([0, 0, -9.81])
            self.vel[:, 2] -= case["speed"]


def _sizes(case):
    """Sphere counts of a batch: log-uniform, of the case alone."""
    rng = np.random.default_rng([case["n"], case["nmin"], case["nmax"]])
    return np.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["n"])).astype(int).tolist()


def _inputs(case, seed):
    """The scenes of a case: one, or a list for batched and served ones."""
    rng = np.random.default_rng([seed, 77])
    n = case["n"]
    periodic = case["kind"] in ("periodic", "monitor", "checkpoint", "pairs")
    if case["kind"] in ("batch", "served"):
        cell = _cell(500, case["phi"], case["radii"], rng)
        out = []
        for m in _sizes(case):
            k = max(1, math.ceil((m / 1000) ** (1 / 3)))
            k = (k, k, math.ceil(m / (500 * k * k)))
            out.append(Spheres(*_tile(cell, m, k, rng), False, case, rng, young=10 ** rng.uniform(6, 8),
                               friction=rng.uniform(0.2, 0.7)))
        return out
    k = max(1, math.ceil((n / 2200) ** (1 / 3)))
    if case["kind"] in ("pairs", "checkpoint"):
        # as many contacts whatever the seed: one packing, moved about its periodic cell, its
        # axes exchanged, its spheres numbered anew
        fixed = np.random.default_rng([n, 78])
        X, R, edge = _tile(_cell(math.ceil(n / k ** 3), case["phi"], case["radii"], fixed), n, (k, k, k), fixed)
        at = rng.permutation(n)
        X, R = np.mod(X + rng.uniform(0, 1, 3) * edge, edge)[at][:, rng.permutation(3)].copy(), R[at]
    else:
        X, R, edge = _tile(_cell(math.ceil(n / k ** 3), case["phi"], case["radii"], rng), n, (k, k, k), rng)
    if case["kind"] == "pairs":
        return X, R, edge
    w = Spheres(X, R, edge, periodic, case, rng)
    if case["shear"]:   # the tiled lattice again, described by a sheared cell
        w.cell[0, 1] = edge[0] / k
        w.velgrad = np.array([[0.0, 4.0, 0], [0, 0, 0], [0, 0, 0]])
    return w


def _scene(w, case):
    mixed = case["precision"] == "mixed"
    s = dem.Scene.from_workload(w, dt=w.dt, precision=dem.DEM_MIXED if mixed else dem.DEM_FP64)
    if case["law"] == "hertz":
        s.set_law(dem.DEM_LAW_HERTZ_MINDLIN)
    if case["tstep"]:
        s.set_timestepper(safety=0.5, interval=1)
    if case["servo"]:
        s.set_triax(SERVO["goal"], SERVO["mask"], SERVO["rate"], SERVO["grow"], SERVO["every"])
    return s


SERVO = {"goal": (-1e5, -1e5, -2.0), "mask": 3, "rate": (10.0, 10.0, 10.0), "grow": 0.25, "every": 5}


def prepare(case, seed):
    w = _inputs(case, seed)
    kind = case["kind"]
    if kind == "pairs":
        X, R, edge = w
        return {"kind": kind, "pos": torch.from_numpy(X).cuda(), "radius": torch.from_numpy(R).cuda(),
                "cell": np.diag(edge), "margin": case["margin"]}
    st = {"kind": kind, "steps": case["steps"]}
    if kind == "served":
        st["server"] = dem.Server(precision=dem.DEM_FP64, tick_steps=100)
        st["work"] = w
        return st
    if kind == "batch":
        mixed = case["precision"] == "mixed"
        s = dem.Scene(precision=dem.DEM_MIXED if mixed else dem.DEM_FP64, capacity_bodies=sum(q.n for q in w))
        for k, q in enumerate(w):
            s.add_workload(q, k, dt=q.dt)
    else:
        s = _scene(w, case)
    st["scene"] = s
    n = s.n
    st["out"] = {"pos": np.empty((n, 3)), "vel": np.empty((n, 3)), "angvel": np.empty((n, 3)), "ori": np.empty((n, 4))}
    return st


STATS = ("kinetic_energy", "unbalanced_force", "coordination", "packing_fraction", "stress")


def run(st):
    kind = st["kind"]
    if kind == "pairs":
        return find_pairs(st["pos"], st["radius"], periodic=True, cell=st["cell"], margin=st["margin"])
    if kind == "served":
        srv = st["server"]
        tickets = [srv.submit(w, st["steps"], keep_state=True, dt=w.dt) for w in st["work"]]
        out = {k: [] for k in ("pos", "vel", "angvel", "ori")}
        for t in tickets:
            srv.wait(t)
            state = srv.result(t, state=True)["state"]
            srv.release(t)
            for k in out:
                out[k].append(state[k])
        return {k: np.concatenate(v) for k, v in out.items()}
    s = st["scene"]
    s.step(st["steps"])
    if kind == "monitor":
        stats = s.stats()
        return {k: stats[k] for k in STATS + ("n_contacts",)}
    if kind == "checkpoint":
        return {"state": s.state(force=False), "contacts": s.contacts()}
    s.get_state_into(**st["out"])
    return st["out"]


# ------------------------------------------------------------------ floors
def work(case):
    """Every step reads and writes the state once, with the history of the contacts it finds; a
    query reads its inputs and writes its outputs."""
    n = case["n"]
    if case["kind"] in ("batch", "served"):
        n = sum(_sizes(case))
    c = n * (2.7 if case["phi"] > 0.5 else 0.1)
    if case["kind"] == "pairs":
        return {"bytes": 32 * n + 20 * c, "flops": 10 * c}
    mixed = case["precision"] == "mixed"
    # state (x, v, w, q) twice and (r, m, I, id); contacts: (Fs, n) twice, (kn, ks, tan phi), ids
    body = 13 * 8 * 2 + 28
    row = (2 * 24 + 2 * 12 + 12 + 12) if mixed else (4 * 24 + 24 + 12)
    out = {"bytes": case["steps"] * (body * n + row * c) + 104 * n,
           "flops": case["steps"] * (131.0 * n + 132.0 * c)}
    if case["kind"] == "monitor":
        out["bytes"] -= 104 * n
    if case["kind"] == "checkpoint":
        out["bytes"] += c * (8 + 12 + 16 * 8)
    return out


# ------------------------------------------------------------------ the method in plain FP64 torch
def _neighbours(x, r, H, periodic, cut):
    """All pairs i < j whose centres are within r_i + r_j + cut, with the cell shift of j."""
    n, dev = len(r), x.device
    reach = 2 * float(r.max()) + cut
    if periodic:
        Hi = torch.linalg.inv(H)
        s = x @ Hi.T
        img = torch.floor(s)
        s = s - img
        width = 1.0 / torch.linalg.norm(Hi, dim=1)
        nc = [max(1, int(q / reach)) for q in width.tolist()]
    else:
        lo, hi = x.min(0).values, x.max(0).values
        nc = [max(1, int(q / reach)) for q in (hi - lo).tolist()]
        s = (x - lo) / (hi - lo).clamp_min(1e-30)
        img = torch.zeros_like(x)
    ni = torch.tensor(nc, device=dev)
    ci = torch.minimum((s * ni).long().clamp_min(0), ni - 1)
    key = (ci[:, 2] * nc[1] + ci[:, 1]) * nc[0] + ci[:, 0]
    ks, order = torch.sort(key, stable=True)
    count = torch.bincount(ks, minlength=nc[0] * nc[1] * nc[2])
    occ = int(count.max())
    member = torch.full((len(count), occ), -1, dtype=torch.long, device=dev)
    member[ks, torch.arange(n, device=dev) - (torch.cumsum(count, 0) - count)[ks]] = order
    me = torch.arange(n, device=dev)
    span = [(-1, 0, 1) if q >= 3 or not periodic else (-1, 0)[2 - q:] for q in nc]
    found = []
    for o in ((a, b, c) for a in span[0] for b in span[1] for c in span[2]):
        cj = ci + torch.tensor(o, device=dev)
        wrap = torch.div(cj, ni, rounding_mode="floor")
        ok = torch.ones(n, dtype=torch.bool, device=dev) if periodic else (wrap == 0).all(1)
        cj = cj - wrap * ni
        kj = (cj[:, 2] * nc[1] + cj[:, 1]) * nc[0] + cj[:, 0]
        for q in range(occ):
            j = member[kj, q]
            sel = torch.nonzero(ok & (j > me)).squeeze(1)
            jj = j[sel]
            c = (wrap[sel].double() + img[sel] - img[jj]) if periodic else torch.zeros(len(sel), 3, device=dev).double()
            d = x[jj] + (c @ H.T if periodic else 0) - x[sel]
            if periodic and min(nc) < 3:   # few cells: the nearest image decides
                c = c - torch.round(d @ Hi.T)
                d = x[jj] + c @ H.T - x[sel]
            near = (d * d).sum(1) < (r[sel] + r[jj] + cut) ** 2
            found.append((sel[near], jj[near], c[near]))
    return [torch.cat([f[q] for f in found]) for q in range(3)]


def _cross(a, b):
    return torch.linalg.cross(a, b)


def _dot(a, b):
    return (a * b).sum(1, keepdim=True)


def _law(n, pen, kn, ks, tanphi, fs, n0, w12, u, dt, hertz):
    """Shear transport and increment, normal force, Coulomb cap: (force on body 2, shear force)."""
    b = _cross(n0, n) + 0.5 * dt * _dot(n, w12) * n
    fs = fs - _cross(fs, b)
    sq = torch.sqrt(pen) if hertz else 1.0
    fs = fs - ks * sq * dt * (u - _dot(n, u) * n)
    fn = kn * pen * sq
    big = torch.linalg.norm(fs, dim=1, keepdim=True)
    fs = torch.where(big > fn * tanphi, fs * (fn * tanphi / big.clamp_min(1e-300)), fs)
    return fn * n + fs, fs


def _simulate(w, case, steps):
    """`steps` steps of the scene w: state and the last step's contacts, in FP64."""
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    x, v, om, r = T(w.pos), T(w.vel), T(w.angvel), T(w.radius)[:, None]
    N, dt, hertz = len(r), w.dt, case["law"] == "hertz"
    q = torch.zeros(N, 4, dtype=torch.float64, device="cuda")
    q[:, 0] = 1
    E, tanphi = w.materials[0].young, math.tan(w.materials[0].friction)
    m = RHO * 4 / 3 * math.pi * r ** 3
    inertia = 0.4 * m * r * r
    G = E / (2 * (1 + NU))
    I3 = torch.eye(3, dtype=torch.float64, device="cuda")
    H, L = T(w.cell), T(w.velgrad)
    Hp, Lp = H.clone(), torch.zeros_like(L)
    g = T(w.gravity)
    i = None
    def stiffness(ra, rb, wall):
        if hertz:
            sR = torch.sqrt(ra if wall else ra * rb / (ra + rb))
            return 4 / 3 * sR / (2 * (1 - NU * NU) / E), 8 * sR / (2 * (2 - NU) / G)
        return 2 * E * ra * rb / (ra + rb), 2 * E * NU * ra * rb / (ra + rb)

    wfs = torch.zeros(6, N, 3, dtype=torch.float64, device="cuda")
    knw, ksw = stiffness(r, r, True)
    for step in range(steps):
        law_dt = dt
        if i is None or step == again:   # candidates near enough for the next steps; history carried over
            speed = float(torch.linalg.norm(v, dim=1).max()) + 0.5
            span = max(1, min(steps, int(float(r.max()) / (2.2 * speed * 1.2 * dt))))
            old, again = None if i is None else (i * N + j, fs, n0, was), step + span
            i, j, c = _neighbours(x, r[:, 0], H, w.periodic, 2.2 * speed * 1.2 * dt * span + 0.02 * float(r.min()))
            at = torch.argsort(i * N + j)
            i, j, c = i[at], j[at], c[at]
            r1, r2 = r[i], r[j]
            kn, ks = stiffness(r1, r2, False)
            fs, n0 = torch.zeros(2, len(i), 3, dtype=torch.float64, device="cuda")
            was = torch.zeros(len(i), 1, dtype=torch.bool, device="cuda")
            if old is not None:
                k = torch.nonzero(old[3][:, 0]).squeeze(1)
                at = torch.searchsorted(i * N + j, old[0][k])
                fs[at], n0[at], was[at] = old[1][k], old[2][k], True
        d = x[j] + c @ H.T - x[i] if w.periodic else x[j] - x[i]
        l2 = (d * d).sum(1, keepdim=True)
        real = l2 < (r1 + r2) ** 2
        l = torch.sqrt(l2)
        n = d / l
        pen = (r1 + r2 - l).clamp_min(0.0)
        n0 = torch.where(was, n0, n)
        v2 = v[j] + c @ (Lp @ Hp).T if w.periodic else v[j]
        u = (r1 + r2) / l * (v2 - v[i]) - _cross(r2 * om[j] + r1 * om[i], n)
        F, f2 = _law(n, pen, kn, ks, tanphi, torch.where(was, fs, torch.zeros_like(fs)), n0, om[i] + om[j], u, law_dt, hertz)
        F, fs = torch.where(real, F, torch.zeros_like(F)), torch.where(real, f2, torch.zeros_like(f2))
        n0, was = n, real
        d1, d2 = r1 - 0.5 * pen, r2 - 0.5 * pen
        M = -_cross(n, F)
        force = torch.zeros_like(x).index_add_(0, j, F).index_add_(0, i, -F)
        torque = torch.zeros_like(x).index_add_(0, j, d2 * M).index_add_(0, i, d1 * M)
        if case["tstep"]:
            tangent = lambda k_, s_, p: (1.5 * k_ * torch.sqrt(p), s_ * torch.sqrt(p)) if hertz else (k_, s_)  # noqa: E731
            tn, ts = tangent(kn, ks, pen)
            n2 = n * n
            zero = torch.zeros_like(n2)
            kt = torch.where(real, (tn - ts) * n2 + ts, zero)
            Kt = torch.zeros_like(x).index_add_(0, i, kt).index_add_(0, j, kt)
            Kr = torch.zeros_like(x)
            for who, arm in ((i, d1), (j, d2)):
                Kr.index_add_(0, who, torch.where(real, ts * arm * arm * (1 - n2), zero))
        for a in range(6):
            if not w.wall_mask:
                break
            ax = a >> 1
            dist = x[:, ax:ax + 1] - float(w.box_hi[ax] if a & 1 else w.box_lo[ax])
            hit = dist.abs() < r
            nw = torch.zeros_like(x)
            nw[:, ax:ax + 1] = torch.where(dist >= 0, 1.0, -1.0).double()
            pw = (r - dist.abs()).clamp_min(0.0)
            uw = 2 * r / (2 * r - pw) * v - _cross(r * om, nw)
            Fw, f2 = _law(nw, pw, knw, ksw, tanphi, wfs[a], nw, om, uw, law_dt, hertz)
            if case["tstep"]:
                tn, ts = tangent(knw, ksw, pw)
                n2, arm = nw * nw, r - 0.5 * pw
                Kt += torch.where(hit, (tn - ts) * n2 + ts, torch.zeros_like(n2))
                Kr += torch.where(hit, ts * arm * arm * (1 - n2), torch.zeros_like(n2))
            Fw, wfs[a] = torch.where(hit, Fw, torch.zeros_like(Fw)), torch.where(hit, f2, torch.zeros_like(f2))
            force += Fw
            torque += _cross(-(r - 0.5 * pw) * nw, Fw)
        if case["tstep"]:
            big = max(float((Kt / m).max()), float((Kr / inertia).max()))
            dt = 0.5 * math.sqrt(2.0 / big) if big > 0 else 0.5 * float(r.min()) * math.sqrt(RHO / E)
        total = force + m * g
        acc, aacc = total / m, torque / inertia
        vref = v - x @ Lp.T if w.periodic else v
        vn = v + dt * acc * (1 - w.damping * torch.sign(total * (vref + 0.5 * dt * acc)))
        om = om + dt * aacc * (1 - w.damping * torch.sign(torque * (om + 0.5 * dt * aacc)))
        if w.periodic:
            vn = vn + x @ (L - Lp).T + dt * (v @ L.T)
        x, v = x + dt * vn, vn
        half = 0.5 * dt * om
        ang = torch.linalg.norm(half, dim=1, keepdim=True)
        e = half * torch.where(ang > 0, torch.sin(ang) / ang.clamp_min(1e-300), torch.ones_like(ang))
        q = torch.cat([torch.cos(ang) * q[:, :1] - _dot(e, q[:, 1:]),
                       torch.cos(ang) * q[:, 1:] + q[:, :1] * e + _cross(e, q[:, 1:])], 1)
        if w.periodic:
            L2 = L.clone()
            if case["servo"] and (step + 1) % SERVO["every"] == 0:
                V, lc = torch.det(H), l * n
                for a in range(3):
                    L2[a, a] = SERVO["goal"][a]
                    if SERVO["mask"] >> a & 1:
                        sig = -(F[:, a] * lc[:, a]).sum() / V
                        K = (torch.where(real, kn, torch.zeros_like(kn))[:, 0] * lc[:, a] ** 2).sum() / V
                        rate = (1 - SERVO["grow"]) * (SERVO["goal"][a] - sig) / (K * dt * SERVO["every"])
                        L2[a, a] = rate.clamp(-SERVO["rate"][a], SERVO["rate"][a])
            Hp, H = H, (I3 + L * dt) @ H
            Lp, L = L, L2
    return {"x": x, "v": v, "om": om, "q": q, "i": i, "j": j, "c": c, "real": real[:, 0], "F": F, "fs": fs, "n": n, "l": l,
            "pen": pen, "kn": kn, "ks": ks, "d1": d1, "tan": tanphi, "force": force, "m": m, "I": inertia, "H": H, "r": r}


def exact(case, seed):
    if case["kind"] == "pairs":   # whole numbers
        return None
    w = _inputs(case, seed)
    if case["kind"] in ("batch", "served"):
        got = [_simulate(q, case, case["steps"]) for q in w]
        return {o: torch.cat([s[k] for s in got]) for o, k in (("pos", "x"), ("vel", "v"), ("angvel", "om"), ("ori", "q"))}
    s = _simulate(w, case, case["steps"])
    state = {"pos": s["x"], "vel": s["v"], "angvel": s["om"], "ori": s["q"]}
    if case["kind"] == "checkpoint":
        k = torch.nonzero(s["real"]).squeeze(1)
        k = k[torch.argsort(s["i"][k] * len(s["m"]) + s["j"][k])]
        phys = torch.cat([s["kn"], s["ks"], torch.full_like(s["kn"], s["tan"])], 1)
        return {"state": state, "contacts": {
            "id1": None, "id2": None, "c": None, "fn": (s["F"] - s["fs"])[k], "fs": s["fs"][k], "normal": s["n"][k],
            "cpoint": (s["x"][s["i"]] + s["d1"] * s["n"])[k], "phys": phys[k], "pen": s["pen"][k, 0]}}
    if case["kind"] == "monitor":
        V, F = float(torch.det(s["H"])), s["F"][s["real"]]
        ke = 0.5 * (s["m"] * s["v"] ** 2).sum() + 0.5 * (s["I"] * s["om"] ** 2).sum()
        return {"kinetic_energy": float(ke), "coordination": 2.0 * len(F) / len(s["m"]), "n_contacts": None,
                "unbalanced_force": float(torch.linalg.norm(s["force"], dim=1).mean() / torch.linalg.norm(F, dim=1).mean()),
                "packing_fraction": float((4 / 3 * math.pi * s["r"] ** 3).sum()) / V,
                "stress": -(s["F"].T @ (s["l"] * s["n"])) / V}
    return state
