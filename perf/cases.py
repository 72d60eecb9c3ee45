"""Workloads whose time is measured, and what their results should be.

Each case is one call sequence a user of the library makes through its public entry points: stepping an
atmosphere (mixed precision and float64, small grids and the benchmark's, the paper's Held-Suarez and
hot-Jupiter set-ups, the approximation switches), an ensemble, an exchange of the fields with the host
every large step, the learned closure's rollout, and the training of its network.

A stepping pass ends with a checkpoint into a device buffer, whose stored fields (deviations from the
reference column, planes [level][column]) are the outputs. The flow of every state is drawn from the
seed: jets, planetary waves of wind and temperature, hydrostatically balanced columns, small noise.

`exact` computes the same in float64 with plain torch: the grid, the operators, the split-explicit step,
the physics, the zonal means and the network are written out again below from the paper's equations."""

import math

import numpy as np
import torch

import paper_1607_05535_gb300 as thor
import workloads as wls

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
SPRING = (1.15, 1.0, 1.0, 0.01, 0.0, 10)      # beta, alpha, k, dt, tol, iterations (the workloads' grids)
FORCING = {"none": 0, "held_suarez": 1, "hot_jupiter": 2}


def listed():
    return [
        # the benchmark: Held-Suarez Earth, mixed precision
        dict(name="hs_g6_l32_mixed", kind="step", planet="earth", glevel=6, nv=32, precision="mixed", dt=600.0,
             n_small=8, n_large=2),
        # the paper's hot Jupiter (1 bar at the bottom) at the benchmark's resolution
        dict(name="hj_g6_l32_mixed", kind="step", planet="hot_jupiter", glevel=6, nv=32, precision="mixed", dt=300.0,
             n_small=6, n_large=2),
        # the paper's long Held-Suarez run: an odd level count, zonal statistics of every sample
        dict(name="hs_g5_l37_mixed_climate", kind="step", planet="earth", glevel=5, nv=37, precision="mixed", dt=1000.0,
             n_small=6, n_large=8, z_top=32.0e3, profile=1, nlat=36),
        # the float64 arm of the benchmark
        dict(name="hs_g6_l32_fp64", kind="step", planet="earth", glevel=6, nv=32, precision="fp64", dt=600.0,
             n_small=8, n_large=1),
        # the plain float64 method at the small standard resolution
        dict(name="hs_g4_l20_fp64", kind="step", planet="earth", glevel=4, nv=20, precision="fp64", dt=1800.0,
             n_small=6, n_large=10),
        # float64 state exchanged with the host every large step (coupling, assimilation)
        dict(name="hs_g5_l32_fp64_host", kind="host", planet="earth", glevel=5, nv=32, precision="fp64", dt=1000.0,
             n_small=6, n_large=1),
        # one large step of a tiny model (the tests' size): launches and latency
        dict(name="hs_g3_l12_mixed", kind="step", planet="earth", glevel=3, nv=12, precision="mixed", dt=1800.0,
             n_small=6, n_large=1),
        # the approximation switches and third-order vertical interpolation, an odd level count
        dict(name="hs_g5_l33_mixed_switches", kind="step", planet="earth", glevel=5, nv=33, precision="mixed",
             dt=1000.0, n_small=6, n_large=4, shallow=1, hydrostatic=1, vorder=3),
        # 64 atmospheres of uneven size stepped together
        dict(name="ensemble_64_l32_mixed", kind="ensemble", members=64, nv=32, precision="mixed", n_small=8, n_large=2),
        # the learned closure online: coarse graining, features, a window of coarse steps corrected by the network
        dict(name="closure_g6_g5_l32", kind="closure", planet="earth", glevel=6, nv=32, precision="mixed", dt=600.0,
             n_small=8, n_large=4),
        # training the closure's network (16 minibatches)
        dict(name="mlp_train_l32_b1024", kind="train", nv=32, hidden=256, batch=1024, steps=16),
        # outputs and gradients of a network for 37 levels: widths that are no multiple of 8, a ragged batch
        dict(name="mlp_grad_l37_b1000", kind="grad", nv=37, hidden=256, batch=1000),
    ]


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["host", "ensemble", "closure", "train", "grad"])
    nv = rng.randint(8, 40)
    if kind == "train" or kind == "grad":
        b = int(round(math.exp(rng.uniform(math.log(64), math.log(8192)))))
        c = dict(kind=kind, nv=nv, hidden=rng.choice([64, 128, 250, 256]), batch=b)
        if kind == "train":
            c["steps"] = rng.randint(2, 16)
        return c
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(2, 24), nv=nv, precision=rng.choice(["mixed", "mixed", "fp64"]),
                    n_small=rng.choice([6, 8]), n_large=1)
    glevel = rng.randint(2, 6)
    hj = rng.random() < 0.25
    dt = {2: 1800.0, 3: 1800.0, 4: 1800.0, 5: 1000.0, 6: 600.0}[glevel] * rng.uniform(0.7, 1.0)
    if hj:
        dt, nv = min(0.5 * dt, 600.0), max(nv, 20)      # layers of at most half a scale height
    c = dict(kind=kind, planet="hot_jupiter" if hj else "earth", glevel=glevel, nv=nv,
             precision=rng.choice(["mixed", "mixed", "mixed", "fp64"]), dt=dt, n_small=rng.choice([6, 8]))
    if kind == "closure":
        c.update(planet="earth", glevel=rng.randint(3, 5), precision="mixed", dt=min(dt, 1000.0), n_large=4)
        return c
    if c["precision"] == "fp64" and glevel == 6:
        c["nv"] = nv = min(nv, 24)
    if kind == "host":
        c.update(precision="fp64", n_large=1, glevel=min(glevel, 5))
        return c
    c["n_large"] = (2 if c["precision"] == "mixed" else 1) if glevel == 6 else rng.randint(1, 4) + hj
    if rng.random() < 0.3:
        c.update(shallow=rng.randint(0, 1), hydrostatic=rng.randint(0, 1), vorder=rng.choice([1, 2, 3]))
    if rng.random() < 0.3:
        c["nlat"] = rng.choice([18, 36, 90])
    return c


# ------------------------------------------------------------------ what a case is made of

class Setup:
    """One atmosphere's parameters."""

    def __init__(self, planet, glevel, nv, z_top, T0, p_surf, forcing, dt, n_small, profile=0, shallow=0,
                 hydrostatic=0, vorder=1, hj_dT=300.0):
        self.planet, self.glevel, self.nv, self.z_top, self.T0, self.p_surf = planet, glevel, nv, z_top, T0, p_surf
        self.forcing, self.dt, self.n_small, self.profile, self.shallow = forcing, dt, n_small, profile, shallow
        self.hydrostatic, self.vorder, self.hj_dT = hydrostatic, vorder, hj_dT
        self.ncol = 10 * 4 ** glevel + 2
        self.gamma = planet.cp / (planet.cp - planet.Rd)
        zi = np.linspace(0.0, z_top, nv + 1)
        self.zi, self.zc = zi, 0.5 * (zi[1:] + zi[:-1])
        self.big = forcing == "hot_jupiter"

    def column(self, T):
        """Pressures of columns with the layer temperatures T ([..., nv]) in the discrete hydrostatic balance."""
        P, zc, zi = self.planet, self.zc, self.zi
        p = [self.p_surf * torch.exp(-P.gravity * zc[0] / (P.Rd * T[..., 0]))]
        for i in range(1, self.nv):
            dz = zc[i] - zc[i - 1]
            w0, w1 = (zc[i] - zi[i]) / dz, (zi[i] - zc[i - 1]) / dz
            p.append(p[-1] * (1.0 - P.gravity * dz * w0 / (P.Rd * T[..., i - 1]))
                     / (1.0 + P.gravity * dz * w1 / (P.Rd * T[..., i])))
        return torch.stack(p, -1)

    def reference(self):
        """(T, rho, rho theta) of the resting column the stored deviations refer to."""
        P = self.planet
        T = torch.full((self.nv,), float(self.T0), dtype=F64)
        if self.profile:
            T[:] = 315.0
            for _ in range(400):
                s = self.column(T) / 1.0e5
                T = torch.clamp((315.0 - 10.0 * torch.log(s)) * s ** (P.Rd / P.cp), min=200.0)
        p = self.column(T)
        return T, p / (P.Rd * T), P.p_ref / P.Rd * (p / P.p_ref) ** (1.0 / self.gamma)

    def fields(self, points, seed):
        """A flow in motion at the points: (rho, mom, W, rho theta), [column][level], float64 on DEV."""
        g = torch.Generator().manual_seed(int(seed))
        rnd = lambda *s: torch.rand(*s, generator=g, dtype=F64).to(DEV) * 2.0 - 1.0
        x = torch.as_tensor(points, dtype=F64, device=DEV)
        zc = torch.as_tensor(self.zc / self.z_top, device=DEV)
        zi = torch.as_tensor(self.zi / self.z_top, device=DEV)
        Tr = self.reference()[0].to(DEV)
        scale = torch.sin(math.pi * torch.clamp(0.15 + 0.6 * zc, max=1.0))

        def wave():          # a smooth planetary-scale function on the sphere, about 1 in size
            q = rnd(3, 3)
            return (x @ q * x).sum(1) + 0.5 * torch.sin(5.0 * (x @ rnd(3))) + 0.3 * torch.sin(9.0 * (x @ rnd(3)))

        T = Tr + (8.0 if self.big else 1.0) * scale * (10.0 * (1.0 / 3.0 - x[:, 2:] ** 2) + 1.5 * wave()[:, None])
        T += 0.1 * torch.rand(T.shape, generator=torch.Generator(DEV).manual_seed(int(seed)), device=DEV, dtype=F64)
        p = self.column(T)
        rho = p / (self.planet.Rd * T)
        th = self.planet.p_ref / self.planet.Rd * (p / self.planet.p_ref) ** (1.0 / self.gamma)
        u0 = 400.0 if self.big else 25.0
        vel = torch.zeros(self.ncol, self.nv, 3, device=DEV, dtype=F64)
        for a, f in ((torch.tensor([0.0, 0.0, 1.0], device=DEV, dtype=F64), 4.0 * x[:, 2] ** 2 * (1.0 - x[:, 2] ** 2)),
                     (rnd(3), 0.3 * wave()), (rnd(3), 0.1 * wave())):
            vel += (u0 * f)[:, None, None] * scale[:, None] * torch.linalg.cross(a.expand_as(x), x)[:, None, :]
        a = rnd(3)           # a divergent part, as in gravity waves and storms
        a = (a - (x @ a)[:, None] * x) * torch.sin(12.0 * (x @ rnd(3)) + 1.0)[:, None]
        vel += (1.0 if self.big else 0.3) * u0 * a[:, None, :] * torch.cos(math.pi * zc)[:, None]
        mom = rho[..., None] * vel
        ri = torch.cat([rho[:, :1], 0.5 * (rho[:, 1:] + rho[:, :-1]), rho[:, -1:]], 1)
        w = (2.0 if self.big else 0.02) * ri * torch.sin(math.pi * zi) * wave()[:, None]
        w[:, 0] = w[:, -1] = 0.0
        return rho, mom, w, th


def setup_of(case, glevel=None):
    c = case
    common = dict(profile=c.get("profile", 0), shallow=c.get("shallow", 0), hydrostatic=c.get("hydrostatic", 0),
                  vorder=c.get("vorder", 1))
    g = c["glevel"] if glevel is None else glevel
    if c["planet"] == "hot_jupiter":
        return Setup(wls.HOT_JUPITER_TABLE1, g, c["nv"], 4875.0e3, 1600.0, 1.0e5, "hot_jupiter", c["dt"],
                     c["n_small"], hj_dT=300.0, **common)
    return Setup(wls.EARTH, g, c["nv"], c.get("z_top", 36.0e3), 300.0, 1.0e5, "held_suarez", c["dt"], c["n_small"],
                 **common)


def members_of(case):
    return [Setup(m.planet, m.glevel, case["nv"], wls.ENSEMBLE_Z_TOP, 300.0, 1.0e5, "held_suarez", m.dt, m.n_small)
            for m in wls.ensemble_members(case["members"], n_small=case["n_small"])]


_grids = {}


def grid_of(s):
    """A program builds the grid of a resolution once and makes its states from it."""
    key = (s.glevel, s.nv, s.planet.radius, s.z_top)
    if key not in _grids:
        _grids[key] = thor.thor_grid_create(s.glevel, s.nv, s.planet.radius, s.z_top, thor.thor_spring(*SPRING))
    return _grids[key]


class Atmosphere:
    """A library state on a stream of its own, with a device buffer for its checkpoints."""

    def __init__(self, s, precision, seed, stream=None):
        P = s.planet
        self.s, self.grid = s, grid_of(s)
        self.stream = stream or torch.cuda.Stream()
        init = thor.thor_init(s.T0, s.p_surf, 0.0, 1234, FORCING[s.forcing], s.hj_dT,
                              thor.THOR_FP64 if precision == "fp64" else thor.THOR_MIXED, 1, 1, s.shallow,
                              s.hydrostatic, s.profile, s.vorder)
        self.dtype = torch.float64 if precision == "fp64" else torch.float32
        self.h = thor.thor_state_init(self.grid, thor.thor_planet(P.radius, P.omega, P.gravity, P.Rd, P.cp, P.p_ref,
                                                                  P.diff_D), init, self.stream.cuda_stream)
        self.start = [f.cpu().contiguous() for f in s.fields(thor.thor_grid_points(self.grid), seed)]
        thor.thor_state_set_all(self.h, *self.start)
        self.buf = torch.empty(thor.thor_checkpoint_bytes(self.h), dtype=torch.uint8, device=DEV)

    def checkpoint(self):
        """The stored fields rho', M_x, M_y, M_z, (rho theta)', W as [level][column] views of the checkpoint."""
        thor.thor_checkpoint_save(self.h, self.buf)
        nv, v = self.s.nv, self.buf[64:].view(self.dtype)
        planes = (6 * nv + 1) * (1 if self.dtype == torch.float64 else 2)    # mixed: the low parts follow
        v = v.view(planes, -1)[:, :self.s.ncol]
        return [v[i * nv:(i + 1) * nv] for i in range(5)] + [v[5 * nv:6 * nv + 1]]

    def __del__(self):
        if getattr(self, "h", None) is not None:
            thor.thor_state_destroy(self.h)
            self.h = None


def net_sizes(case):
    return [10 * case["nv"], case["hidden"], case["hidden"], case["hidden"], 5 * case["nv"]]


def net_params(sizes, seed):
    """He-uniform weights and small biases, flat: W_0, b_0, W_1, b_1, ..."""
    g = np.random.default_rng(int(seed))
    out = []
    for k, n in zip(sizes[:-1], sizes[1:]):
        out += [g.uniform(-1, 1, k * n) * math.sqrt(6.0 / k), 0.05 * g.standard_normal(n)]
    return np.concatenate(out).astype(np.float32)


def net_data(sizes, batches, batch, seed):
    """Normalised features and a target that depends on them smoothly."""
    g = torch.Generator(DEV).manual_seed(int(seed))
    x = torch.randn(batches, batch, sizes[0], generator=g, device=DEV)
    a = torch.randn(sizes[0], sizes[-1], generator=g, device=DEV) / math.sqrt(sizes[0])
    return x, torch.tanh(x @ a) + 0.1 * torch.randn(batches, batch, sizes[-1], generator=g, device=DEV)


class Network:
    def __init__(self, sizes, batch, params, stream=None):
        self.sizes, self.params = sizes, params
        self.h = thor.thor_mlp_create(sizes, batch, 1, stream)
        thor.thor_mlp_set_params(self.h, params)

    def __del__(self):
        if getattr(self, "h", None) is not None:
            thor.thor_mlp_destroy(self.h)
            self.h = None


def closure_norm(s, fields):
    """Per-feature and per-output scales from the fine flow: every field's deviation by level, a twentieth of it
    for the neighbour anomalies; the network's correction over a window is a hundredth of the deviation."""
    _, rb, tb = s.reference()
    rho, mom, _, th = (f.to(DEV) for f in fields)
    rms = lambda f: f.square().mean(0).sqrt() + 1e-12
    sc = torch.cat([rms(rho - rb.to(DEV)), rms(mom[..., 0]), rms(mom[..., 1]), rms(mom[..., 2]), rms(th - tb.to(DEV))])
    f32 = lambda t: t.to(torch.float32).contiguous()
    zero = torch.zeros_like
    return [f32(t) for t in (zero(torch.cat([sc, sc])), torch.cat([sc, 0.05 * sc]), zero(sc), 0.01 / (4 * s.dt) * sc)]


# ------------------------------------------------------------------ the measured calls

class Prepared:
    def __init__(self, case):
        self.case = case


def prepare(case, seed):
    q = Prepared(case)
    kind = case["kind"]
    if kind in ("step", "host"):
        q.a = Atmosphere(setup_of(case), case["precision"], seed)
        if kind == "host":
            q.inp = [f.pin_memory() for f in q.a.start]
            q.out = [torch.empty_like(f).pin_memory() for f in q.a.start]
    elif kind == "ensemble":
        q.stream = torch.cuda.Stream()
        q.a = [Atmosphere(s, case["precision"], seed + 7919 * i, q.stream) for i, s in enumerate(members_of(case))]
        q.h = thor.thor_ensemble_create([a.h for a in q.a], q.stream.cuda_stream)
        q.steps, q.dts = [a.s.n_small for a in q.a], [a.s.dt for a in q.a]
        q.close = EnsembleHandle(q.h)
    elif kind == "closure":
        q.fine = Atmosphere(setup_of(case), case["precision"], seed)
        q.a = Atmosphere(setup_of(case, case["glevel"] - 1), case["precision"], seed)
        q.map = thor.thor_grid_coarse_map(q.fine.grid, q.a.grid)
        sizes = [10 * case["nv"], 256, 256, 256, 5 * case["nv"]]
        q.net = Network(sizes, 1024, net_params(sizes, seed), q.a.stream.cuda_stream)
        q.norm = closure_norm(q.fine.s, q.fine.start)
        q.x = torch.empty(q.a.s.ncol, sizes[0], device=DEV)
        torch.cuda.synchronize()
        thor.thor_closure_attach(q.a.h, q.net.h, *q.norm, period=case["n_large"])
    else:
        sizes = net_sizes(case)
        q.net = Network(sizes, case["batch"], net_params(sizes, seed), torch.cuda.current_stream().cuda_stream)
        q.x, q.t = net_data(sizes, case.get("steps", 1), case["batch"], seed)
        q.loss = torch.zeros(1, device=DEV)
        q.y, q.g = torch.empty_like(q.t[0]), torch.empty(thor.thor_mlp_info(q.net.h), device=DEV)
    return q


class EnsembleHandle:
    def __init__(self, h):
        self.h = h

    def __del__(self):
        thor.thor_ensemble_destroy(self.h)


def run(q):
    c = q.case
    if c["kind"] == "step":
        thor.thor_step(q.a.h, c["n_large"], c["n_small"], c["dt"])
        if not c.get("nlat"):
            return q.a.checkpoint()
        thor.thor_zonal_accumulate(q.a.h, c["nlat"])
        out = q.a.checkpoint()
        z = thor.thor_zonal_read(q.a.h, c["nlat"], c["nv"], reset=True)[0]
        # the statistics are written in the precision the state has
        return out + [z[..., j].astype(np.float64 if c["precision"] == "fp64" else np.float32) for j in range(9)]
    if c["kind"] == "host":
        thor.thor_state_set_all(q.a.h, *q.inp)
        thor.thor_step(q.a.h, c["n_large"], c["n_small"], c["dt"])
        return list(thor.thor_state_get_all(q.a.h, q.a.s.ncol, c["nv"], q.out))
    if c["kind"] == "ensemble":
        thor.thor_ensemble_step(q.h, c["n_large"], q.steps, q.dts)
        for a in q.a:
            thor.thor_checkpoint_save(a.h, a.buf)
        # one tensor per member: all its fields, [plane][column], the mixed states' low parts left out
        return [a.buf[64:].view(a.dtype).view((6 * a.s.nv + 1) * (8 // a.dtype.itemsize), -1)[:6 * a.s.nv + 1, :a.s.ncol]
                for a in q.a]
    if c["kind"] == "closure":
        thor.thor_coarse_grain(q.fine.h, q.a.h, q.map)
        thor.thor_closure_features(q.a.h, q.norm[0], q.norm[1], q.x)
        thor.thor_step(q.a.h, c["n_large"], c["n_small"], c["dt"])
        return [q.x] + q.a.checkpoint()
    if c["kind"] == "train":
        for i in range(c["steps"]):
            thor.thor_mlp_train_step(q.net.h, q.x[i], q.t[i], 1e-3, q.loss)
        return [thor.thor_mlp_get_params(q.net.h), q.loss]
    thor.thor_mlp_forward(q.net.h, q.x[0], q.y)
    thor.thor_mlp_backward(q.net.h, q.t[0], q.g)
    return [q.y, q.g]


def work(case):
    """The words the method reads and writes per cell: 13 per slow-term evaluation, 27 per small step, 9 for the
    physics; and its arithmetic, about 250, 160 and 60 operations."""
    c = case
    if c["kind"] in ("train", "grad"):
        z = net_sizes(c)
        w = sum(a * b for a, b in zip(z[:-1], z[1:]))
        per = c["batch"] * (6 * w - 2 * z[0] * z[1])
        io = c["batch"] * (z[0] + z[-1]) * 4
        if c["kind"] == "train":
            return {"bytes": c["steps"] * (io + 7 * 4 * w), "flops": c["steps"] * per}
        return {"bytes": io + c["batch"] * z[-1] * 4 + 8 * w, "flops": per}
    word = 8 if c["precision"] == "fp64" else 4

    def steps(s):
        cells, n = s.ncol * s.nv, 1 + s.n_small // 2 + s.n_small
        return (c["n_large"] * cells * word * (3 * 13 + 27 * n + 9), c["n_large"] * cells * (3 * 250 + 160 * n + 60))

    if c["kind"] == "ensemble":
        b, f = (sum(v) for v in zip(*(steps(s) for s in members_of(c))))
        return {"bytes": b, "flops": f}
    s = setup_of(c, c["glevel"] - 1 if c["kind"] == "closure" else None)
    b, f = steps(s)
    if c["kind"] == "closure":
        z = [10 * c["nv"], 256, 256, 256, 5 * c["nv"]]
        f += 2 * s.ncol * sum(p * q for p, q in zip(z[:-1], z[1:]))
        b += s.ncol * s.nv * 4 * (4 * 6 + 3 * 10)
    if c["kind"] == "host":
        b += 2 * 8 * s.ncol * (6 * s.nv + 1)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in float64, plain torch

def unit(v):
    return v / np.linalg.norm(v, axis=-1, keepdims=True)


def arc(a, b):
    return np.arctan2(np.linalg.norm(np.cross(a, b), axis=-1), (a * b).sum(-1))


def tri_area(a, b, c):
    num = np.abs((a * np.cross(b, c)).sum(-1))
    return 2.0 * np.arctan2(num, 1.0 + (a * b).sum(-1) + (b * c).sum(-1) + (c * a).sum(-1))


def centroid(v):
    """Centroids of spherical polygons v [..., corner, 3]."""
    w = np.roll(v, -1, axis=-2)
    cr = np.cross(v, w)
    s = np.linalg.norm(cr, axis=-1, keepdims=True)
    return unit((np.arctan2(s, (v * w).sum(-1, keepdims=True)) * cr / s).sum(-2))


class Mesh:
    """The spring-smoothed icosahedral grid (Sec. 2) in the column order of `points`, and its operators as sparse
    matrices on the unit sphere: D[d] (divergence of component d), G[d] (projected gradient), L (Laplacian)."""

    def __init__(self, glevel, points):
        lat, fifth = math.atan(0.5), 2.0 * math.pi / 5.0
        ring = lambda z, off: [(math.cos(lat) * math.cos(k * fifth + off), math.cos(lat) * math.sin(k * fifth + off), z)
                               for k in range(5)]
        P = np.array([(0, 0, 1.0)] + ring(math.sin(lat), 0.0) + ring(-math.sin(lat), fifth / 2) + [(0, 0, -1.0)])
        T = []
        for k in range(5):
            u, v, m, n = 1 + k, 1 + (k + 1) % 5, 6 + k, 6 + (k + 1) % 5
            T += [(0, u, v), (u, m, v), (m, n, v), (11, n, m)]
        T = np.array(T)
        for _ in range(glevel):
            e = np.sort(np.concatenate([T[:, [0, 1]], T[:, [1, 2]], T[:, [2, 0]]]), 1)
            _, first, back = np.unique(e[:, 0] * len(P) + e[:, 1], return_index=True, return_inverse=True)
            ab, bc, ca = (len(P) + back.reshape(3, -1))
            a, b, c = T.T
            P = np.concatenate([P, unit(P[e[first, 0]] + P[e[first, 1]])])
            T = np.concatenate([np.stack(t, 1) for t in ((a, ab, ca), (ab, b, bc), (ca, bc, c), (ab, bc, ca))])
        flip = (np.cross(P[T[:, 1]] - P[T[:, 0]], P[T[:, 2]] - P[T[:, 0]]) * P[T].sum(1)).sum(1) < 0
        T[flip] = T[flip][:, [0, 2, 1]]
        N = len(P)
        # triangles and neighbours around every point, counter-clockwise
        v, a = T.T.reshape(-1), T[:, [1, 2, 0]].T.reshape(-1)
        e1 = unit(np.cross(P, np.where(np.abs(P[:, 2:]) < 0.9, [[0, 0, 1.0]], [[1.0, 0, 0]])))
        ang = np.arctan2((P[a] * np.cross(P, e1)[v]).sum(1), (P[a] * e1[v]).sum(1))
        order = np.lexsort((ang, v))
        nn = np.bincount(v, minlength=N)
        pos = np.arange(3 * len(T)) - np.repeat(np.cumsum(nn) - nn, nn)
        rf, nb = np.zeros((N, 6), int), np.tile(np.arange(N)[:, None], (1, 6))
        rf[v[order], pos] = np.tile(np.arange(len(T)), 3)[order]
        nb[v[order], pos] = a[order]
        five = nn == 5
        if glevel > 0:
            P = self.springs(P, nb, five, glevel)
        C = centroid(P[T])
        P = P.copy()
        P[~five], P[five] = centroid(C[rf[~five]]), centroid(C[rf[five][:, :5]])
        # the library's column order: nearest points
        lib, own = torch.as_tensor(points, device=DEV), torch.as_tensor(P, device=DEV)
        perm = torch.cat([(q @ own.T).argmax(1) for q in lib.split(2048)]).cpu().numpy()
        assert np.abs(P[perm] - points).max() < 1e-9
        inv = np.empty(N, int)
        inv[perm] = np.arange(N)
        P, T, rf, nn, self.nb = P[perm], inv[T], rf[perm], nn[perm], inv[nb[perm]]
        self.nn = torch.as_tensor(nn, device=DEV)
        # edge lengths times outward normals over areas, and what each corner contributes to them
        k = np.arange(6)
        valid = k < nn[:, None]
        c0, c1 = C[rf], C[np.take_along_axis(rf, np.where(k + 1 < nn[:, None], k + 1, 0), 1)]
        n = np.cross(c0, c1)
        n = n / np.maximum(np.linalg.norm(n, axis=-1, keepdims=True), 1e-300)
        n *= np.where((n * P[:, None]).sum(-1) > 0, -1.0, 1.0)[..., None]
        self.area = np.where(valid, tri_area(P[:, None], c0, c1), 0.0).sum(1)
        ln = np.where(valid, arc(c0, c1), 0.0)[..., None] * n / self.area[:, None, None]
        prev = np.take_along_axis(ln, np.where(k > 0, k - 1, nn[:, None] - 1)[..., None], 1)
        E = np.where(valid[..., None], 0.5 * (ln + prev), 0.0)                     # (N, 6, 3)
        x = P[T]
        wt = np.stack([tri_area(x[:, (i + 1) % 3], x[:, (i + 2) % 3], C) for i in range(3)], 1)
        wt /= wt.sum(1, keepdims=True)
        te = np.stack([unit(np.cross(x[:, i], x[:, (i + 1) % 3])) for i in range(3)], 1)
        te *= np.where((te * np.roll(x, -2, axis=1)).sum(-1) > 0, -1.0, 1.0)[..., None]
        te *= np.stack([arc(x[:, i], x[:, (i + 1) % 3]) for i in range(3)], 1)[..., None]
        grad = 0.5 * (te + np.roll(te, 1, axis=1)) - wt[..., None] * te.sum(1)[:, None]
        grad /= tri_area(x[:, 0], x[:, 1], x[:, 2])[:, None, None]                 # (F, 3 vertices, 3)
        row = np.repeat(np.arange(N), 18)
        col = T[rf].reshape(-1)

        def matrix(val, diag=None):
            r, c, u = row, col, val.reshape(-1)
            if diag is not None:
                r, c, u = np.append(r, np.arange(N)), np.append(c, np.arange(N)), np.append(u, diag)
            m = torch.sparse_coo_tensor(torch.as_tensor(np.stack([r, c])), torch.as_tensor(u), (N, N), device=DEV)
            return m.coalesce().to_sparse_csr()

        dv = E[:, :, None, :] * wt[rf][..., None]                                  # (N, 6, 3 vertices, 3)
        self.D = [matrix(dv[..., d]) for d in range(3)]
        pj = lambda f: f - (f * P.reshape((N,) + (1,) * (f.ndim - 2) + (3,))).sum(-1, keepdims=True) \
            * P.reshape((N,) + (1,) * (f.ndim - 2) + (3,))
        gv, gd = pj(dv), pj(-ln.sum(1))
        self.G = [matrix(gv[..., d], gd[:, d]) for d in range(3)]
        self.L = matrix((E[:, :, None, :] * grad[rf]).sum(-1))
        self.P, self.points = torch.as_tensor(P, device=DEV), P

    @staticmethod
    def springs(P, nb, five, glevel):
        beta, alpha, k, dt, _, iters = SPRING
        rest = beta * 2.0 * math.pi / (10.0 * 2.0 ** (glevel - 1))
        v = np.zeros_like(P)
        for _ in range(iters):
            Q = P[nb]
            dot = (P[:, None] * Q).sum(-1)
            t = Q - dot[..., None] * P[:, None]
            size = np.linalg.norm(t, axis=-1, keepdims=True)
            F = (k * (arc(P[:, None], Q) - rest)[..., None] * t / np.where(size > 0, size, 1.0)).sum(1)
            v += dt * (F - alpha * v)
            v[five] = 0.0
            new = unit(P + dt * v)
            new[five] = P[five]
            v -= (v * new).sum(1, keepdims=True) * new
            P = new
        return P


_meshes = {}


def mesh_of(s):
    if s.glevel not in _meshes:
        _meshes[s.glevel] = Mesh(s.glevel, thor.thor_grid_points(grid_of(s)))
    return _meshes[s.glevel]


def lagrange(nodes, targets, first, k):
    """Interpolation matrix (targets x nodes) of order k from the k + 1 nodes nearest each target; first: the
    index of the first node above each target."""
    A = np.zeros((len(targets), len(nodes)))
    for i, (z, f) in enumerate(zip(targets, first)):
        j0 = min(max(f - (k + 2) // 2, 0), len(nodes) - k - 1)
        for j in range(j0, j0 + k + 1):
            A[i, j] = np.prod([(z - nodes[m]) / (nodes[j] - nodes[m]) for m in range(j0, j0 + k + 1) if m != j])
    return torch.as_tensor(A.T.copy(), device=DEV)


class Core:
    """The split-explicit dynamical core (Sec. 3-5); fields are [column][level] float64 tensors, vectors lists of three."""

    def __init__(self, s, mesh):
        t = lambda a: torch.as_tensor(np.asarray(a), device=DEV)
        self.s, self.m = s, mesh
        nv, A = s.nv, s.planet.radius
        deep = 0.0 if s.shallow else 1.0
        self.rc, self.ri = t(A + deep * s.zc), t(A + deep * s.zi)
        self.dz, self.dzc = t(np.diff(s.zi)), t(np.diff(s.zc))
        inner = range(1, nv)
        self.I1 = lagrange(s.zc, s.zi[1:-1], inner, 1)
        self.Ik = lagrange(s.zc, s.zi[1:-1], inner, max(s.vorder, 1))
        self.Ck = lagrange(s.zi, s.zc, range(1, nv + 1), max(s.vorder, 1))
        self.r = [mesh.P[:, d:d + 1] for d in range(3)]
        dbar = math.sqrt(2.0 * math.pi / 5.0) * A / 2.0 ** s.glevel
        self.Kd = s.planet.diff_D * dbar ** 4 / s.dt
        self.ends = lambda x: torch.nn.functional.pad(x, (1, 1))

    def div(self, F):
        return sum(D @ f for D, f in zip(self.m.D, F)) / self.rc

    def grad(self, f):
        return [G @ f / self.rc for G in self.m.G]

    def lap(self, f, r=None):
        return self.m.L @ f / (self.rc if r is None else r) ** 2

    def div_v(self, w):
        f = self.ri ** 2 * w
        return (f[:, 1:] - f[:, :-1]) / (self.rc ** 2 * self.dz)

    def proj(self, F):
        d = sum(f * r for f, r in zip(F, self.r))
        return [f - d * r for f, r in zip(F, self.r)]

    def pressure(self, th):
        P = self.s.planet
        return P.p_ref * (P.Rd * th / P.p_ref) ** self.s.gamma

    def slow(self, rho, M, W, th):
        s, P, r, ends = self.s, self.s.planet, self.r, self.ends
        p = self.pressure(th)
        Wc = W @ self.Ck
        up = lambda x: ends(x @ self.Ik)
        full = [m + Wc * q for m, q in zip(M, r)]
        v = [(m if s.shallow else f) / rho for m, f in zip(M, full)]
        adv = lambda a: self.div([m * a for m in M]) + self.div_v(W * up(a))
        A = [adv(a) for a in v]
        if s.shallow:
            f = 2.0 * P.omega * r[2]
            C = [f * (r[1] * M[2] - r[2] * M[1]), f * (r[2] * M[0] - r[0] * M[2]), f * (r[0] * M[1] - r[1] * M[0])]
            Ar = up(adv(Wc / rho))
        else:
            C = [-2.0 * P.omega * full[1], 2.0 * P.omega * full[0], 0.0]
            Ar = up(sum((a + c) * q for a, c, q in zip(A, C, r)))
        AC = self.proj([a + c for a, c in zip(A, C)])
        # hyperdiffusion
        Kd, rho_k, rho_1 = self.Kd, rho @ self.Ik, rho @ self.I1
        F_rho = -self.lap(Kd * self.lap(rho))
        F_M = self.proj([-self.lap(rho * Kd * self.lap(m / rho)) for m in M])
        ri = self.ri[1:-1]
        F_W = ends(-self.lap(rho_k * Kd * self.lap(W[:, 1:-1] / rho_k, ri), ri))
        F_th = th / (s.gamma * p) * -P.Rd * self.lap(rho * Kd * self.lap(p / (rho * P.Rd)))
        S_M = self.proj([-g - a + f for g, a, f in zip(self.grad(p), AC, F_M)])
        S_W = ends(-(p[:, 1:] - p[:, :-1]) / self.dzc - P.gravity * rho_1)
        if not s.hydrostatic:
            S_W = S_W - Ar + F_W
        return dict(p=p, S_M=S_M, S_W=S_W, S_rho=-self.div(M) - self.div_v(W) + F_rho, S_th=F_th, theta=th / rho,
                    thi=ends(th / rho @ self.I1), Pi=s.gamma * p / th)

    def solve(self, dt, W, S_W, a, b, c, thi, Pi):
        """The implicit vertical momentum: Eqs. dens2 and pt2 substituted into Eq. momr2, one tridiagonal per column."""
        g, delta = self.s.planet.gravity, 0.0 if self.s.hydrostatic else 1.0
        lo, hi = self.ri[:-1] ** 2 / (self.rc ** 2 * self.dz), self.ri[1:] ** 2 / (self.rc ** 2 * self.dz)
        wl, wh = (torch.diagonal(self.I1).clone(), torch.diagonal(self.I1, -1).clone())
        th, dzc = thi[:, 1:-1], self.dzc
        pl, ph = Pi[:, :-1], Pi[:, 1:]
        d2 = dt * dt
        diag = delta + d2 / dzc * th * (ph * lo[1:] + pl * hi[:-1]) - d2 * g * (wl * hi[:-1] - wh * lo[1:])
        low = -d2 / dzc * pl * lo[:-1] * thi[:, :-2] + d2 * g * wl * lo[:-1]
        upp = -d2 / dzc * ph * hi[1:] * thi[:, 2:] - d2 * g * wh * hi[1:]
        rhs = delta * W[:, 1:-1] + dt * S_W[:, 1:-1] - dt * (c[:, 1:] - c[:, :-1]) / dzc - dt * g * (a @ self.I1)
        cp, dp = [upp[:, 0] / diag[:, 0]], [rhs[:, 0] / diag[:, 0]]
        for m in range(1, self.s.nv - 1):
            q = 1.0 / (diag[:, m] - low[:, m] * cp[-1])
            dp.append((rhs[:, m] - low[:, m] * dp[-1]) * q)
            cp.append(upp[:, m] * q)
        x = [dp[-1]]
        for m in range(self.s.nv - 3, -1, -1):
            x.append(dp[m] - cp[m] * x[-1])
        return self.ends(torch.stack(x[::-1], 1))

    def stage(self, Xt, X, dt, steps):
        rho, M, W, th = X
        co = self.slow(*X)
        r, m, w, t = Xt[0] - rho, [a - b for a, b in zip(Xt[1], M)], Xt[2] - W, Xt[3]
        p = self.pressure(t) - co["p"]
        for _ in range(steps):
            D = self.div([a + b for a, b in zip(M, m)]) + self.div_v(W + w)
            DD = self.grad(self.lap(D))
            m = self.proj([a + dt * (-g - self.Kd * d + q) for a, g, d, q in zip(m, self.grad(p), DD, co["S_M"])])
            a = r + dt * (co["S_rho"] - self.div(m))
            b = t + dt * (co["S_th"] - self.div([co["theta"] * (u + v) for u, v in zip(M, m)])
                          - self.div_v(co["thi"] * W))
            w = self.solve(dt, w, co["S_W"], a, b, p + co["Pi"] * (b - t), co["thi"], co["Pi"])
            r, t = a - dt * self.div_v(w), b - dt * self.div_v(co["thi"] * w)
            p = self.pressure(t) - co["p"]
        return rho + r, [u + v for u, v in zip(M, m)], W + w, t

    def physics(self, rho, M, W, th):
        s, P = self.s, self.s.planet
        p = self.pressure(th)
        T = p / (rho * P.Rd)
        ps = p[:, :1] * torch.exp(P.gravity * s.zc[0] / (P.Rd * T[:, :1]))
        sig, sl = p / ps, self.r[2]
        if s.forcing == "held_suarez":
            day, c2 = 86400.0, 1.0 - sl * sl
            ramp = torch.clamp((sig - 0.7) / 0.3, min=0.0)
            Kv = ramp / day
            KT = 1.0 / (40 * day) + (1.0 / (4 * day) - 1.0 / (40 * day)) * ramp * c2 * c2
            q = p / 1.0e5
            Te = torch.clamp((315.0 - 60.0 * sl * sl - 10.0 * torch.log(q) * c2) * q ** (P.Rd / P.cp), min=200.0)
        else:
            z = torch.as_tensor(s.zc, device=DEV)
            zs, G, dT = 2.0e6, 2.0e-4, 10.0
            Tv = torch.where(z <= zs, 1600.0 - G * (zs + (z - zs) / 2) + torch.sqrt((G * (z - zs) / 2) ** 2 + dT * dT),
                             1600.0 - G * zs + dT)
            bt = torch.where(z <= zs, torch.sin(math.pi * (sig - 0.12) / (2.0 * 0.88)), 0.0 * sig)
            Kv, KT, Te = 0.0, 1.0 / 1.5e5, Tv + bt * s.hj_dT * self.r[0]
        T = (T + KT * s.dt * Te) / (1.0 + KT * s.dt)
        th = P.p_ref / P.Rd * (rho * P.Rd * T / P.p_ref) ** (1.0 / s.gamma)
        return rho, [m / (1.0 + Kv * s.dt) for m in M], W, th

    def step(self, X):
        X = (X[0], [X[1][..., d] for d in range(3)], X[2], X[3]) if torch.is_tensor(X[1]) else X
        Xs, n, dt = X, self.s.n_small, self.s.dt
        for d, k in ((dt / 3.0, 1), (dt / n, n // 2), (dt / n, n)):
            Xs = self.stage(X, Xs, d, k)
        return self.physics(*Xs)

    def stored(self, X):
        """rho', M_x, M_y, M_z, (rho theta)', W as [level][column]."""
        _, rb, tb = (q.to(DEV) for q in self.s.reference())
        return [q.T.contiguous() for q in (X[0] - rb, *X[1], X[3] - tb, X[2])]

    def zonal(self, X, nlat):
        """Band weights, means of u, v, T, p and the covariances u'v', v'T', u'u', v'v', each [level][band]."""
        P, x = self.s.planet, self.m.points
        lon, lat = np.arctan2(x[:, 1], x[:, 0]), np.arcsin(np.clip(x[:, 2], -1, 1))
        b = torch.as_tensor(np.minimum(np.floor((lat + math.pi / 2 + 1e-9) / math.pi * nlat).astype(int), nlat - 1), device=DEV)
        on = np.hypot(x[:, 0], x[:, 1]) >= 1e-9
        t = lambda q: torch.as_tensor(q * on, device=DEV)[:, None]
        rho, M, _, th = X
        vx, vy, vz = (m / rho for m in M)
        u = vy * t(np.cos(lon)) - vx * t(np.sin(lon))
        v = vz * t(np.cos(lat)) - t(np.sin(lat)) * (vx * t(np.cos(lon)) + vy * t(np.sin(lon)))
        p = self.pressure(th)
        T = p / (rho * P.Rd)
        w = torch.as_tensor(self.m.area, device=DEV)[:, None] * self.rc ** 2 * self.dz
        band = lambda q: torch.zeros(nlat, q.shape[1], dtype=F64, device=DEV).index_add_(0, b, q)
        W = band(w)
        mean = lambda q: torch.where(W > 0, band(w * q) / torch.where(W > 0, W, 1.0), 0.0)
        mu, mv, mT = mean(u), mean(v), mean(T)
        cov = lambda f, g, mf, mg: mean(f * g) - mf * mg
        return [q.T.contiguous() for q in (W, mu, mv, mT, mean(p), cov(u, v, mu, mv), cov(v, T, mv, mT),
                                           cov(u, u, mu, mu), cov(v, v, mv, mv))]


def forward(sizes, flat, x):
    """Layer inputs (x, hidden activations) and the output of the network."""
    h, o = [x], 0
    for l, (k, n) in enumerate(zip(sizes[:-1], sizes[1:])):
        z = h[-1] @ flat[o:o + k * n].view(k, n) + flat[o + k * n:o + k * n + n]
        o += k * n + n
        if l + 2 == len(sizes):
            return h, z
        h.append(torch.relu(z))


def gradient(sizes, flat, h, g):
    """Gradient of sum(y * g) with respect to every parameter, in the flat order."""
    out, o = [], len(flat)
    for l in range(len(sizes) - 2, -1, -1):
        k, n = sizes[l], sizes[l + 1]
        o -= k * n + n
        out.insert(0, torch.cat([(h[l].T @ g).reshape(-1), g.sum(0)]))
        g = (g @ flat[o:o + k * n].view(k, n).T) * (h[l] > 0)
    return torch.cat(out)


def exact(case, seed):
    c = case
    if c["kind"] in ("train", "grad"):
        sizes = net_sizes(c)
        p = torch.as_tensor(net_params(sizes, seed), device=DEV).double()
        x, t = (q.double() for q in net_data(sizes, c.get("steps", 1), c["batch"], seed))
        if c["kind"] == "grad":
            h, y = forward(sizes, p, x[0])
            return [y, gradient(sizes, p, h, t[0])]
        m = v = torch.zeros_like(p)
        for i in range(c["steps"]):
            h, y = forward(sizes, p, x[i])
            loss = (y - t[i]).square().mean()
            g = gradient(sizes, p, h, 2.0 * (y - t[i]) / y.numel())
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 1e-3 * (m / (1 - 0.9 ** (i + 1))) / ((v / (1 - 0.999 ** (i + 1))).sqrt() + 1e-8)
        return [p, loss.reshape(1)]
    if c["kind"] == "ensemble":
        out = []
        for i, s in enumerate(members_of(c)):
            core = Core(s, mesh_of(s))
            X = s.fields(thor.thor_grid_points(grid_of(s)), seed + 7919 * i)
            for _ in range(c["n_large"]):
                X = core.step(X)
            out.append(torch.cat(core.stored(X)))
        return out
    s = setup_of(c)
    X = s.fields(thor.thor_grid_points(grid_of(s)), seed)
    if c["kind"] == "closure":
        return exact_closure(c, s, X, seed)
    core = Core(s, mesh_of(s))
    for _ in range(c["n_large"]):
        X = core.step(X)
    if c["kind"] == "host":
        return [X[0], torch.stack(X[1], -1), X[2], X[3]]
    return core.stored(X) + (core.zonal(X, c["nlat"]) if c.get("nlat") else [])


def exact_closure(c, fine, X, seed):
    s = setup_of(c, c["glevel"] - 1)
    mf, mc = mesh_of(fine), mesh_of(s)
    near = thor.thor_grid_coarse_map(grid_of(fine), grid_of(s))       # the map the call is given
    near = torch.as_tensor(near, device=DEV).long()
    area = torch.as_tensor(mf.area, device=DEV)
    total = torch.zeros(s.ncol, dtype=F64, device=DEV).index_add_(0, near, area)

    def mean(f):
        q = f.reshape(f.shape[0], -1) * (area / total[near])[:, None]
        return torch.zeros(s.ncol, q.shape[1], dtype=F64, device=DEV).index_add_(0, near, q).reshape((s.ncol,) + f.shape[1:])

    core = Core(s, mc)
    rho, mom, w, th = (mean(f) for f in X)
    Y = (rho, core.proj([mom[..., d] for d in range(3)]), w, th)
    inm, ins, outm, outs = (q.double() for q in closure_norm(fine, X))
    _, rb, tb = (q.to(DEV) for q in s.reference())
    f = torch.cat([Y[0] - rb, *Y[1], Y[3] - tb], 1)
    nb = torch.as_tensor(mc.nb, device=DEV)
    ring = sum(f[nb[:, j]] * (mc.nn > j)[:, None] for j in range(6)) / mc.nn[:, None]
    x = (torch.cat([f, ring - f], 1) - inm) / ins
    sizes = [10 * s.nv, 256, 256, 256, 5 * s.nv]
    tau = forward(sizes, torch.as_tensor(net_params(sizes, seed), device=DEV).double(), x)[1] * outs + outm
    for _ in range(c["n_large"]):
        Y = core.step(Y)
    t = (c["n_large"] * s.dt * tau).split(s.nv, 1)
    m = core.proj(list(t[1:4]))
    return [x] + core.stored((Y[0] + t[0], [a + b for a, b in zip(Y[1], m)], Y[2], Y[3] + t[4]))
