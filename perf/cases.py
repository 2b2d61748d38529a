"""Performance cases: the work that users of this package have it do, through its public calls.

The cases are time stepping of scenes (one frame = a number of steps and a
read of the state), first-step forces on caller-owned device buffers, and the
learned surrogate's two calls (graph + forward of one stride, one training
step), over the package's range of sizes, precisions and options.  Beds are
settled by a short run before they are measured, as the benchmark does.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  what a program holds before the call
    run(state)           one pass, and its outputs
    work(case)           bytes and operations of one pass that cannot be left out
    exact(case, seed)    the outputs in plain 64-bit torch
"""
import math

import numpy as np
import torch

from paper_2507_12610_gb300 import batch, dem, scenes, surrogate

PRECISIONS = {"fp64": dem.DEM_FP64, "mixed": dem.DEM_MIXED, "mixed64": dem.DEM_MIXED64}


def listed():
    return [
        # the pouring box workload (1,000 spheres, 12 triangles): a small scene resumed
        # from its checkpoint, where launches and latency count
        dict(name="box_mixed_1k", kind="box", n=1000, precision="mixed", steps=500, forces=False),
        # the same in double precision with contact forces read, as a reference run takes it
        dict(name="box_fp64_1k", kind="box", n=1000, precision="fp64", steps=200, forces=True),
        # the angle-of-repose heap while its stream still falls: spawning, plates, 20,000 rows
        dict(name="heap_mixed_20k", kind="heap", n=20_000, precision="mixed", steps=300,
             forces=False),
        # the rotating drum at the size of its statistics runs
        dict(name="drum_mixed_20k", kind="drum", n=20_000, precision="mixed", steps=200,
             forces=False),
        # the headline: the 1,000,000-sphere rotating drum, a frame every 100 steps
        dict(name="drum_mixed_1m", kind="drum", n=1_000_000, precision="mixed", steps=100,
             forces=False),
        # the double-precision step, bound by the FP64 pipe
        dict(name="drum_fp64_200k", kind="drum", n=200_000, precision="fp64", steps=20,
             forces=False),
        # the granular column collapse (log-normal radii, wide floor), FP32 law on FP64 state
        dict(name="column_mixed64_200k", kind="column", n=200_000, precision="mixed64", steps=50,
             forces=False),
        # a batched ensemble of hoppers with a material each
        dict(name="hoppers_mixed_64", kind="hoppers", n=64, precision="mixed", steps=100,
             forces=False),
        # first-step forces on caller-owned buffers, no allocation
        dict(name="forces_fp64_100k", kind="forces", n=100_000),
        # one stride of the surrogate (neighbour graph + network) on the 100,000-sphere drum
        dict(name="stride_100k", kind="stride", n=100_000),
        # the same on a small drum
        dict(name="stride_3k", kind="stride", n=3_000),
        # one training step of the surrogate on hopper scenes
        dict(name="train_12", kind="train", n=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["box", "heap", "drum", "drum", "drum", "column", "hoppers", "forces",
                       "stride", "stride", "train"])
    if kind in ("forces", "stride"):
        return dict(kind=kind, n=_log_int(rng, 2_000, 100_000))
    if kind == "train":
        return dict(kind=kind, n=rng.randint(2, 12))
    precision = rng.choice(["fp64", "mixed", "mixed", "mixed64"])
    lo, hi = {"box": (300, 1500), "heap": (5_000, 40_000), "drum": (2_000, 400_000),
              "column": (2_000, 200_000), "hoppers": (3, 64)}[kind]
    if precision == "fp64" and kind in ("drum", "column"):
        hi = 120_000
    steps = rng.randint(10, 20) if precision == "fp64" else rng.randint(40, 100)
    return dict(kind=kind, n=_log_int(rng, lo, hi), precision=precision, steps=steps,
                forces=kind == "box" and rng.random() < 0.5)


# ---- inputs ------------------------------------------------------------------

def _scene(case, seed):
    """The scene as the package's workloads define it, before it settles."""
    kind, n = case["kind"], case["n"]
    if kind == "box":
        f = (n / 1000.0) ** (1.0 / 3.0)
        return scenes.box_scene(n=n, seed=seed, speed=0.3, size=(0.020 * f, 0.020 * f, 0.060 * f))
    if kind == "column":
        return scenes.column_scene(n=n, seed=seed, spacing=2.2e-3)
    if kind in ("hoppers", "train"):
        # the batched workload's ranges; the sizes are the case's, the rest the seed's
        top = 8_000 if kind == "hoppers" else 3_000
        sizes = np.exp(np.random.default_rng(n).uniform(math.log(500), math.log(top), n))
        mu = np.random.default_rng(seed).uniform((0.2, 0.0, 0.0), (0.8, 0.2, 0.2), (n, 3))
        return batch.combine([batch.hopper_scene(int(k), seed * 1009 + i, tuple(mu[i]))
                              for i, k in enumerate(sizes)])
    if kind == "heap":
        # the heap scene with half of its grains already piled between the plates
        s = scenes.repose_scene(n=n, seed=seed)
        r, half = s["spawn"]["r_min"], 0.5 * s["gap"]
        rng = np.random.default_rng(seed)
        ny = int((2 * half - 2.2 * r) / (2.02 * r)) + 1
        nx = max(4, int(math.sqrt(n / 2 / ny)) * 2)
        k = np.arange(n // 2)
        x = np.stack([(k % nx - 0.5 * (nx - 1)) * 2.02 * r,
                      (k // nx % ny - 0.5 * (ny - 1)) * 2.02 * r,
                      1.01 * r + k // (nx * ny) * 2.02 * r], axis=1)
        x += rng.uniform(-0.008 * r, 0.008 * r, size=x.shape)
        s.update(R=np.full(len(x), r), x=x)
        return s
    radius = scenes.drum_geometry(n)[0] + 0.006 if n < 20_000 else None
    theta, rings = (128, 15) if n >= 400_000 else (64, 8)
    return scenes.drum_scene(n=n, seed=seed, n_theta=theta, n_rings=rings, nn_dist=2.15e-3,
                             speed=0.02, radius=radius)


SETTLE = {"box": 3000, "heap": 500, "drum": 2500, "column": 2000, "hoppers": 1000, "train": 1000,
          "forces": 2500, "stride": 2500}


def _settled(case, seed):
    """The scene with its particles where they are after a settling run."""
    s = _scene(case, seed)
    sc = dem.Scene.from_dict(s, precision=dem.DEM_MIXED)
    sc.step(SETTLE[case["kind"]])
    st = sc.state()
    a, R = sc.active, sc.radii()
    sc.close()
    keep = {k: v[:a] for k, v in st.items()}
    s = dict(s, R=R[:a], **keep)
    if s.get("material") is not None:
        s["material"] = s["material"][:a]
    return s


def _pinned(n, width):
    return torch.empty((n, width), dtype=torch.float64, pin_memory=True).numpy()


def _weights(seed):
    """Network weights (inputs incl. the constant block, outputs) per layer."""
    rng = np.random.default_rng(seed)
    out = {}
    for name, (kin, nout) in surrogate.LAYERS.items():
        w = np.zeros((kin, nout), np.float32)
        used = 7 if kin == 16 else kin - 16
        cols = 6 if name == "dec" else nout
        w[:used, :cols] = rng.normal(scale=math.sqrt(2.0 / used), size=(used, cols))
        w[used, :cols] = 0.1
        out[name] = w
    return out


def _targets(s, seed):
    """Scaled mean accelerations [n][6] to train on: gravity and contact scatter."""
    rng = np.random.default_rng(seed + 1)
    t = rng.normal(scale=0.5, size=(len(s["R"]), 6))
    t[:, 2] -= 0.981
    return t


def prepare(case, seed):
    kind = case["kind"]
    s = _settled(case, seed)
    if kind == "forces":
        dev = {k: torch.as_tensor(s[k], device="cuda") for k in ("R", "x", "v", "w")}
        F, T = torch.empty_like(dev["x"]), torch.empty_like(dev["x"])
        rmax = float(s["R"].max())
        box = (s["x"].min(axis=0) - rmax, s["x"].max(axis=0) + rmax)
        return dict(kind=kind, params=s["params"], rmax=rmax, box=box, F=F, T=T, **dev)
    if kind == "stride":
        return dict(kind=kind, bed=s, rmax=float(s["R"].max()),
                    model=surrogate.MPNN(weights=_weights(seed)))
    if kind == "train":
        g = surrogate.make_graph(s["x"], s["v"], s["w"], s["R"], float(s["R"].max()))
        return dict(kind=kind, graph=g, model=surrogate.MPNN(weights=_weights(seed)),
                    target=surrogate.target_buffer(_targets(s, seed), g.npad))
    kw = dict(skin=0.3 * float(s["R"].max()), step_warps=8) if kind == "hoppers" else {}
    sc = dem.Scene.from_dict(s, precision=PRECISIONS[case["precision"]],
                             record_forces=case["forces"], **kw)
    frame = {k: _pinned(sc.n, w) for k, w in (("x", 3), ("v", 3), ("w", 3), ("q", 4))}
    # the small box resumes from its checkpoint in every pass; the others run on
    return dict(kind=kind, scene=sc, steps=case["steps"], forces=case["forces"], frame=frame,
                blob=sc.save() if kind == "box" else None)


# ---- one pass ----------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "forces":
        rc = dem.contact_forces_noalloc(
            state["params"], len(state["R"]), state["rmax"], state["R"].data_ptr(),
            state["x"].data_ptr(), state["v"].data_ptr(), state["w"].data_ptr(),
            state["F"].data_ptr(), state["T"].data_ptr(), state["box"])
        if rc != dem.DEM_OK:
            raise dem.DemError(rc, "contact_forces_noalloc")
        return dict(F=state["F"], T=state["T"])
    if kind == "stride":
        b = state["bed"]
        g = surrogate.make_graph(b["x"], b["v"], b["w"], b["R"], state["rmax"])
        y = state["model"].forward(g, keep=False)
        return dict(y=y[:g.n, :surrogate.OUT], off=g.off)
    if kind == "train":
        m = state["model"]
        loss = m.loss_and_grad(state["graph"], state["target"])
        m.adam(1e-3)
        return dict(loss=np.float32(loss), **{f"G_{k}": v for k, v in m.G.items()})
    sc, f = state["scene"], state["frame"]
    if state["blob"] is not None:
        sc.load(state["blob"])
    sc.step(state["steps"])
    rc = sc.read_state_into(f["x"], f["v"], f["w"], f["q"])
    if rc != dem.DEM_OK:
        raise dem.DemError(rc, "step")
    out = dict(f)
    if state["forces"]:
        out["F"], out["T"] = sc.forces()
    return out


# ---- what a pass cannot do without ---------------------------------------------

PAIRS = {"box": 1.5, "heap": 2.0, "drum": 2.6, "column": 1.5, "hoppers": 1.5, "forces": 2.6}
ENTRIES = 9.0   # list entries per particle
EDGES = 11.0    # directed graph edges per particle (cutoff 2.2 R_max)


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "hoppers":
        n = int(n * 7500 / math.log(16.0))   # mean of the log-uniform sizes
    if kind == "train":
        n = int(n * 2500 / math.log(6.0))
    if kind == "forces":
        return {"bytes": n * (10 + 6) * 8.0, "flops": n * 275.0 * PAIRS[kind]}
    if kind in ("stride", "train"):
        E, H = EDGES * n, 128
        fwd = 2.0 * (n * 16 * H + E * 16 * H + 3 * (E * 400 * H + n * 272 * H) + n * 144 * 6)
        weights = sum(a * b for a, b in surrogate.LAYERS.values())
        if kind == "stride":
            return {"bytes": n * 10 * 4.0 + weights * 2.0 + n * 6 * 4.0, "flops": fwd}
        return {"bytes": (n + E) * 32.0 + n * 6 * 4.0 + weights * 4.0 * 7, "flops": 3.0 * fwd}
    fp64 = case["precision"] == "fp64"
    spring = 56 if fp64 else 28
    pairs = PAIRS[kind]
    # state read and written once (x, v, omega, q; R read; 8 bytes a value in every
    # precision), the list, the springs and keys
    per = 27 * 8 + 4 * ENTRIES + pairs * (2 * spring + 8)
    flops = 275.0 * pairs + 190.0
    return {"bytes": n * per * case["steps"] + n * 13 * 8.0, "flops": n * flops * case["steps"]}


# ---- the same in plain 64-bit torch ----------------------------------------------

def _dev(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device="cuda")


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def _cross(a, b):
    a, b = torch.broadcast_tensors(a, b)
    return torch.linalg.cross(a, b, dim=-1)


def _near_pairs(x, R, reach):
    """Index pairs i < j with |x_i - x_j| < R_i + R_j + reach (cell search)."""
    h = 2.0 * float(R.max()) + reach
    c = ((x - x.min(0).values) / h).floor().long() + 1
    nc = c.max(0).values + 2
    key = (c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0]
    skey, order = torch.sort(key)
    found = []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            row = key + (dz * nc[1] + dy) * nc[0]
            a = torch.searchsorted(skey, row - 1)
            m = torch.searchsorted(skey, row + 1, right=True) - a
            i = torch.repeat_interleave(torch.arange(len(R), device=x.device), m)
            first = torch.cumsum(m, 0) - m
            j = order[a[i] + torch.arange(len(i), device=x.device) - first[i]]
            keep = j > i
            i, j = i[keep], j[keep]
            near = (x[i] - x[j]).norm(dim=1) < R[i] + R[j] + reach
            found.append(i[near] * len(R) + j[near])
    return torch.sort(torch.cat(found)).values


def _closest(q, E, four):
    """Closest points of triangles (vertices 0-2) and rectangles (`four`) to q."""
    a, b, c, d = E[..., 0, :], E[..., 1, :], E[..., 2, :], E[..., 3, :]
    u, w = b - a, torch.where(four, d - a, c - a)
    s, t = _dot(q - a, u) / _dot(u, u), _dot(q - a, w) / _dot(w, w)
    rect = a + s.clamp(0, 1) * u + t.clamp(0, 1) * w
    nrm = _cross(u, w)
    plane = q - _dot(q - a, nrm) / _dot(nrm, nrm) * nrm
    inside, best, dist = None, None, None
    for p0, p1 in ((a, b), (b, c), (c, a)):
        e = p1 - p0
        side = _dot(_cross(e, plane - p0), nrm) >= 0
        inside = side if inside is None else inside & side
        foot = p0 + (_dot(q - p0, e) / _dot(e, e)).clamp(0, 1) * e
        d2 = _dot(q - foot, q - foot)
        best = foot if best is None else torch.where(d2 < dist, foot, best)
        dist = d2 if dist is None else torch.minimum(d2, dist)
    return torch.where(four, rect, torch.where(inside, plane, best))


def _spring(u, n, v, k, c, lim, dt):
    """Sliding or rolling spring: force and the spring after the step."""
    ut = u - _dot(u, n) * n
    a, b = _dot(u, u), _dot(ut, ut)
    u = torch.where((a > 0) & (b > 0), (a / b.where(b > 0, torch.ones_like(b))).sqrt() * ut,
                    torch.zeros_like(u))
    f = -k * u - c * v
    size = f.norm(dim=-1, keepdim=True)
    stay = size <= lim
    clip = lim / size.where(size > 0, torch.ones_like(size)) * f
    return torch.where(stay, f, clip), torch.where(stay, u + dt * v, -(clip + c * v) / k)


class _Plain:
    """The time step of the paper, pairs and mesh contacts, written out in
    64-bit torch (no drag, no spawning; triangles and rectangles)."""

    def __init__(self, s):
        p = self.p = s["params"]
        self.R, self.x, self.v, self.w, self.q = (_dev(s[k]) for k in ("R", "x", "v", "w", "q"))
        self.n = len(self.R)
        self.m = 4.0 / 3.0 * math.pi * p["rho"] * self.R ** 3
        mu = torch.tensor([[p["mu_s"], p["mu_r"], p["mu_t"]]], dtype=torch.float64, device="cuda")
        self.mu = mu.expand(self.n, 3)
        if s.get("material") is not None:
            self.mu = _dev(s["material_mu"])[torch.as_tensor(s["material"], device="cuda").long()]
        V, El, _ = scenes.all_elements(s)
        self.four = torch.as_tensor(El[:, 3] >= 0, device="cuda")
        self.E0 = _dev(V)[torch.as_tensor(np.where(El < 0, El[:, :1], El), device="cuda").long()]
        self.om, self.ctr = _dev(p["mesh_omega"]), _dev(p["mesh_center"])
        self.step_no, self.reach = 0, 0.4 * float(self.R.max())
        self.pk = torch.empty(0, dtype=torch.long, device="cuda")
        self.mk, self.ph, self.mh = self.pk, self._hist(0), self._hist(0)
        self.x_ref = None

    def _hist(self, k):
        return torch.zeros((k, 7), dtype=torch.float64, device="cuda")

    def elements(self, idx=None):
        """Vertices at the present pose of the mesh."""
        E = self.E0 if idx is None else self.E0[idx]
        wn = float(self.om.norm())
        if wn == 0:
            return E
        th, ax, r = wn * self.step_no * self.p["dt"], self.om / wn, E - self.ctr
        turn = _cross(ax, r)
        return self.ctr + math.cos(th) * r + math.sin(th) * turn \
            + (1 - math.cos(th)) * _dot(ax, r) * ax

    def _search(self):
        if self.x_ref is not None:
            far = float((self.x - self.x_ref).norm(dim=1).max())
            arm = float((self.E0 - self.ctr).norm(dim=-1).max()) if len(self.E0) else 0.0
            far += arm * float(self.om.norm()) * self.p["dt"] * (self.step_no - self.at)
            if far < 0.49 * self.reach:
                return
        self.x_ref, self.at = self.x.clone(), self.step_no
        keys = _near_pairs(self.x, self.R, self.reach)
        self.ph, self.pk = self._carry(self.pk, self.ph, keys), keys
        found, E, M = [], self.elements(), len(self.E0)
        rows = max(1, 8_000_000 // max(M, 1))
        for a in range(0, self.n, rows):
            q = self.x[a:a + rows, None]
            d = (q - _closest(q, E, self.four[:, None])).norm(dim=-1)
            i, k = torch.nonzero(d < self.R[a:a + rows, None] + self.reach, as_tuple=True)
            found.append((i + a) * M + k)
        keys = torch.cat(found)
        self.mh, self.mk = self._carry(self.mk, self.mh, keys), keys

    def _carry(self, old, hist, new):
        out = self._hist(len(new))
        if len(old) and len(new):
            at = torch.searchsorted(old, new).clamp(max=len(old) - 1)
            same = old[at] == new
            out[same] = hist[at[same]]
        return out

    def _law(self, h, n, delta, Es, Gs, Rs, ms, ri, rj, reff, dv, rw, om, mu):
        """Force on i, torques on i and j (springs in h are updated)."""
        p = self.p
        ln = math.log(p["e_n"])
        beta = 1.0 / math.sqrt(1.0 + (math.pi / ln) ** 2)
        a = (Rs * delta).sqrt()
        kn, ks = 4.0 / 3.0 * Es * a, 8.0 * Gs * a
        cn, cs = (5.0 * ms * kn).sqrt() * beta, (ms * ks / 6.0).sqrt() * beta
        v = dv + _cross(n, rw)
        vn = _dot(v, n) * n
        fn = kn * delta * n - cn * vn
        size = fn.norm(dim=-1, keepdim=True)
        fs, us = _spring(h[:, 0:3], n, v - vn, ks, cs, mu[:, 0:1] * size, p["dt"])
        fr, ur = _spring(h[:, 3:6], n, reff * _cross(om, n), kn, cn,
                         mu[:, 1:2] * size, p["dt"])
        vt, ut, lim = Rs * _dot(om, n), h[:, 6:7], mu[:, 2:3] * size
        ft = -ks * ut - cs * vt
        stay = ft.abs() <= lim
        ft = torch.where(stay, ft, torch.where(ft > 0, lim, -lim))
        ut = torch.where(stay, ut + p["dt"] * vt, -(ft + cs * vt) / ks)
        side, tr, tt = _cross(fs, n), Rs * _cross(n, fr), ft * Rs * n
        return fn + fs, ri * side + tr + tt, rj * side - tr - tt, torch.cat([us, ur, ut], 1)

    def step(self):
        p, R, x, v, w = self.p, self.R[:, None], self.x, self.v, self.w
        G = p["E"] / (2.0 * (1.0 + p["nu"]))
        Es, Gs = p["E"] / (1.0 - p["nu"] ** 2), G / (2.0 - p["nu"])
        self._search()
        F, T = torch.zeros_like(x), torch.zeros_like(x)
        i, j = self.pk // self.n, self.pk % self.n
        d = x[i] - x[j]
        dist = d.norm(dim=1, keepdim=True)
        delta = R[i] + R[j] - dist
        on = (delta >= 0)[:, 0] & (dist > 0)[:, 0]
        h = self._hist(len(i))
        i, j, d, dist, delta, old = i[on], j[on], d[on], dist[on], delta[on], self.ph[on]
        ri, rj = R[i] - 0.5 * delta, R[j] - 0.5 * delta
        m = self.m[:, None]
        f, ti, tj, h[on] = self._law(
            old, d / dist, delta, 0.5 * Es, 0.5 * Gs, 1.0 / (1.0 / R[i] + 1.0 / R[j]),
            1.0 / (1.0 / m[i] + 1.0 / m[j]), ri, rj, 1.0 / (1.0 / ri + 1.0 / rj), v[i] - v[j],
            ri * w[i] + rj * w[j], w[i] - w[j], 0.5 * (self.mu[i] + self.mu[j]))
        self.ph = h
        for t, a, b in ((F, f, -f), (T, ti, tj)):
            t.index_add_(0, i, a)
            t.index_add_(0, j, b)
        if len(self.mk):
            M = len(self.E0)
            i, k = self.mk // M, self.mk % M
            d = x[i] - _closest(x[i], self.elements(k), self.four[k, None])
            dist = d.norm(dim=1, keepdim=True)
            delta = R[i] - dist
            on = (delta >= 0)[:, 0] & (dist > 0)[:, 0]
            h = self._hist(len(i))
            i, d, dist, delta, old = i[on], d[on], dist[on], delta[on], self.mh[on]
            n, ri = d / dist, R[i] - 0.5 * delta
            om = self.om.expand(n.shape)
            wall = _cross(om, x[i] - ri * n - self.ctr)
            f, ti, _, h[on] = self._law(old, n, delta, Es, Gs, R[i], m[i], ri, 0.0 * ri, ri,
                                        v[i] - wall, ri * w[i], w[i] - om, self.mu[i])
            self.mh = h
            F.index_add_(0, i, f)
            T.index_add_(0, i, ti)
        self.F, self.T = F, T
        dt = p["dt"]
        acc, alp = F / m + _dev(p["g"]), T / (0.4 * m * R * R)
        self.v = v + dt * acc
        self.x = x + dt * self.v
        self.q = self._turn(self._turn(self.q, w, 0.5 * dt), alp, (0.5 * dt) ** 2)
        self.w = w + dt * alp
        self.step_no += 1

    @staticmethod
    def _turn(q, a, h):
        """q times (cos h|a|, sin h|a| a / |a|)."""
        size = a.norm(dim=1, keepdim=True)
        s, c = torch.sin(h * size) / size.where(size > 0, torch.ones_like(size)), torch.cos(h * size)
        b, q0, qv = s * a, q[:, :1], q[:, 1:]
        return torch.cat([q0 * c - _dot(qv, b), q0 * b + c * qv + _cross(qv, b)], 1)


def _network(s, weights):
    """Graph (receiver, sender; ascending) and the network in 64 bits."""
    f32 = lambda a: _dev(np.asarray(a, dtype=np.float32))  # noqa: E731
    x, v, w, R = f32(s["x"]), f32(s["v"]), f32(s["w"]), f32(s["R"])
    n, vs, Rs = len(R), surrogate.SCALES["vs"], surrogate.SCALES["Rs"]
    cut = 2.2 * float(s["R"].max())
    keys = _near_pairs(x, torch.zeros_like(R), cut)
    i, j = keys // n, keys % n
    dst, src = torch.cat([i, j]), torch.cat([j, i])
    order = torch.sort(dst * n + src).indices
    dst, src = dst[order], src[order]
    z = lambda k: torch.zeros((k, 16), dtype=torch.float64, device="cuda")  # noqa: E731
    nf, ef, one_n, one_e = z(n), z(len(dst)), z(n), z(len(dst))
    nf[:, 0:3], nf[:, 3:6], nf[:, 6], nf[:, 7] = v / vs, R[:, None] * w / vs, R / Rs - 1.0, 1.0
    d = x[src] - x[dst]
    ef[:, 0:3], ef[:, 3] = d / Rs, (d.norm(dim=1) - R[dst] - R[src]) / Rs
    ef[:, 4:7], ef[:, 7] = (v[src] - v[dst]) / vs, 1.0
    one_n[:, 0], one_e[:, 0] = 1.0, 1.0
    h, e = torch.relu(nf @ weights["node"]), torch.relu(ef @ weights["edge"])
    for r in range(surrogate.ROUNDS):
        m = torch.relu(torch.cat([h[dst], h[src], e, one_e], 1) @ weights[f"msg{r}"])
        M = torch.zeros_like(h).index_add(0, dst, m)
        h = h + torch.relu(torch.cat([h, M, one_n], 1) @ weights[f"upd{r}"])
    return torch.cat([h, one_n], 1) @ weights["dec"]


def exact(case, seed):
    kind = case["kind"]
    if kind == "heap":
        return None   # spawning: the stream of kept grains has no plain counterpart here
    s = _settled(case, seed)
    if kind in ("stride", "train"):
        W = {k: _dev(v).requires_grad_(kind == "train") for k, v in _weights(seed).items()}
        if kind == "stride":
            return dict(y=_network(s, W)[:, :surrogate.OUT], off=None)
        y = _network(s, W)[:, :surrogate.OUT]
        loss = ((y - _dev(_targets(s, seed).astype(np.float32))) ** 2).mean()
        loss.backward()
        out = dict(loss=float(loss.detach()))
        for k, t in W.items():   # rows up to a multiple of 64, as the gradients are kept
            g = torch.zeros((surrogate.pad64(t.shape[0]), t.shape[1]), dtype=torch.float64)
            g[:t.shape[0]] = t.grad.cpu()
            out[f"G_{k}"] = g
        return out
    if kind == "forces":
        s = dict(s, verts=np.zeros((0, 3)), tris=np.zeros((0, 3), np.int32), elems=None)
    ref = _Plain(s)
    for _ in range(1 if kind == "forces" else case["steps"]):
        ref.step()
    if kind == "forces":
        return dict(F=ref.F, T=ref.T)
    out = {k: getattr(ref, k) for k in ("x", "v", "w", "q")}
    if case["forces"]:
        out["F"], out["T"] = ref.F, ref.T
    return out
