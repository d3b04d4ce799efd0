"""The work that users of the library have it do, as measurable cases.

A case is one call pattern of the public interface on one mesh size:

* ``se``, ``sesm``, ``visc``: a model hands over its state and the frozen forcing as device arrays,
  advances ``steps`` baroclinic steps of M substeps and takes eta, U and <<U>> back (``extra`` adds
  the freshwater flux and the step-mean elevation);
* ``host``: the same for a model that lives on the host: pinned host arrays in, host arrays and the
  FP64 volume and energy out;
* ``batch``: an ensemble of closed basins of uneven size in one context;
* ``train``: loss and weight gradient of one sample of the learned surrogate;
* ``rollout``: surrogate steps from a given state.

Meshes are the repository's recipes (rectangular basin, jittered Delaunay channel and basins,
icosahedral sphere with land); states, forcings, weights and samples come from the seed.
"""
import functools
import math

import numpy as np
import torch

from paper_2311_08241_gb300 import inputs as I
from paper_2311_08241_gb300 import sesw as S

DEV = "cuda"
G, THETA = I.G_DEFAULT, I.THETA_DEFAULT
HID, LAYERS = 64, 3
ACCEPT_ALL = 1e30


def listed():
    return [
        # the small closed basin of the verification runs (101 x 51 vertices, M = 30): a step is all latency
        {"name": "basin_small", "kind": "se", "mesh": "rect", "nx": 101, "ny": 51, "M": 30, "steps": 10, "extra": False},
        # a regional channel of ragged size with every optional per-vertex term (freshwater, step mean)
        {"name": "channel_extra", "kind": "se", "mesh": "channel", "nx": 253, "ny": 147, "M": 33, "steps": 4,
         "extra": True},
        # the wind-driven channel benchmark (199,920 vertices, M = 40)
        {"name": "channel", "kind": "se", "mesh": "channel", "nx": 588, "ny": 340, "M": 40, "steps": 4, "extra": False},
        # the same channel driven from a host model, one step per exchange, with the diagnostics
        {"name": "channel_host", "kind": "host", "mesh": "channel", "nx": 588, "ny": 340, "M": 40, "steps": 1,
         "extra": False},
        # the global mesh: icosahedral sphere level 8 with 30 % land (458,683 wet vertices, M = 50)
        {"name": "sphere", "kind": "se", "mesh": "sphere", "level": 8, "M": 50, "steps": 4, "extra": False},
        # an ensemble of basins of 20k to 400k vertices, the shape of the default benchmark at a third of its size
        {"name": "ensemble", "kind": "batch", "basins": 24, "vmin": 20000, "vmax": 400000, "M": 40, "steps": 2},
        # the AB3-AM4 scheme on the channel, and on a mesh whose state does not stay on chip
        {"name": "channel_sesm", "kind": "sesm", "mesh": "channel", "nx": 588, "ny": 340, "M": 40, "steps": 4,
         "extra": False},
        {"name": "large_sesm", "kind": "sesm", "mesh": "channel", "nx": 841, "ny": 485, "M": 40, "steps": 2,
         "extra": False},
        # the barotropic viscosity with the freshwater flux on the channel
        {"name": "channel_visc", "kind": "visc", "mesh": "channel", "nx": 588, "ny": 340, "M": 40, "steps": 2,
         "extra": True},
        # surrogate training, one sample: the level-6 sphere of the small training run, the level-8 one of the large
        {"name": "train_small", "kind": "train", "mesh": "sphere", "level": 6},
        {"name": "train_large", "kind": "train", "mesh": "sphere", "level": 8},
        # surrogate inference, steps taken without the fallback
        {"name": "rollout", "kind": "rollout", "mesh": "sphere", "level": 7, "M": 50, "steps": 2},
    ]


def _channel_size(rng, vlo, vhi):
    nv = math.exp(rng.uniform(math.log(vlo), math.log(vhi)))
    nx = max(12, int(math.sqrt(nv * 1.73 * rng.uniform(0.6, 1.6))))
    return {"mesh": "channel", "nx": nx, "ny": max(9, int(nv / nx))}


def draw(rng):
    kind = rng.choice(["se", "se", "se", "host", "batch", "sesm", "sesm", "visc", "visc", "train", "rollout"])
    if kind == "batch":
        vmin = int(math.exp(rng.uniform(math.log(500), math.log(20000))))
        return {"kind": kind, "basins": rng.randint(2, 20), "vmin": vmin, "vmax": vmin * rng.randint(2, 18),
                "M": rng.randint(20, 50), "steps": rng.randint(1, 3)}
    if kind in ("train", "rollout"):
        c = {"mesh": "sphere", "level": rng.randint(4, 7)} if rng.random() < 0.4 else _channel_size(rng, 2000, 200000)
        c["kind"] = kind
        if kind == "rollout":
            c.update(M=rng.randint(20, 50), steps=rng.randint(1, 3))
        return c
    if kind in ("se", "visc") and rng.random() < 0.3:
        c = {"mesh": "sphere", "level": rng.randint(4, 7)}
    elif kind in ("se", "host") and rng.random() < 0.3:
        c = {"mesh": "rect", "nx": rng.randint(12, 301), "ny": rng.randint(12, 201)}
    else:
        c = _channel_size(rng, 500, {"se": 400000, "host": 200000, "sesm": 400000, "visc": 200000}[kind])
    c.update(kind=kind, M=rng.randint(15, 50), steps=1 if kind == "host" else rng.randint(1, 4),
             extra=kind != "host" and rng.random() < 0.4)
    return c


# ------------------------------------------------------------------------------ meshes

_KEEP = {}


def _kept(key, make):
    """The last few meshes made (a mesh depends on the case alone, the fields on the seed)."""
    if key not in _KEEP:
        while len(_KEEP) >= 3:
            _KEEP.pop(next(iter(_KEEP)))
        _KEEP[key] = make()
    return _KEEP[key]


@functools.lru_cache(maxsize=2)
def _sphere(level):
    return I.sphere_mesh(level)


def _mesh(case):
    """(mesh, vertex spacing, stable substep) of a single-mesh case."""
    if case["mesh"] == "sphere":
        m = _sphere(case["level"])
        return m, 28e3 * 2.0 ** (8 - case["level"]), 36.0
    if case["mesh"] == "rect":
        return _kept(("rect", case["nx"], case["ny"]), lambda: (
            I.basin_case(nx=case["nx"], ny=case["ny"], dx=10e3).mesh, 10e3, 20.0))

    def make():
        nx, ny = case["nx"], case["ny"]
        h = 4000e3 / nx
        Ly = (ny - 1) * h * math.sqrt(3.0) / 2.0
        m = I.channel_case(nx=nx, ny=ny, Ly=Ly).mesh
        return m, h, 12.0 * h / 6803.0
    return _kept(("channel", case["nx"], case["ny"]), make)


def _basins(case):
    def make():
        cs = I.ensemble_cases(case["basins"], vmin=case["vmin"], vmax=case["vmax"], M=case["M"])
        return [c.mesh for c in cs], [c.params for c in cs]
    return _kept(("batch", case["basins"], case["vmin"], case["vmax"], case["M"]), make)


def _params(case, h, dt):
    M = case.get("M", 50)
    visc = None
    if case["kind"] == "visc":
        # a background viscosity well inside the explicit limit (the sphere's shallow coasts tighten it)
        visc = ((0.002 if case["mesh"] == "sphere" else 0.05) * h * h / (24.0 * dt), 0.02)
    sesm = case["kind"] == "sesm"
    return I.Params(tau=M * dt * (0.9 if sesm else 1.0), M=M, scheme=1 if sesm else 0, visc=visc)


# ------------------------------------------------------------------------------ fields

def _waves(X, rng, n=6, kmax=9.0):
    """A smooth field on points X [N][3] of unit extent, about 1 in size: a few random plane waves."""
    out = torch.zeros(X.shape[0], dtype=torch.float64, device=DEV)
    for _ in range(n):
        k = torch.tensor(rng.normal(size=3) * rng.uniform(1.0, kmax), device=DEV)
        out += float(rng.normal()) * torch.cos(X @ k + float(rng.uniform(0, 6.3)))
    return out / math.sqrt(n / 2.0)


def _points(meshes):
    xs, cs = [], []
    for m in meshes:
        p = torch.from_numpy(np.asarray(m.pos, dtype=np.float64)).to(DEV)
        p = (p - p.mean(0)) / float((p.max(0).values - p.min(0).values).max())
        t = torch.from_numpy(np.asarray(m.tri)).to(DEV).long()
        # a triangle takes the point of its first corner (periodic meshes wrap)
        xs.append(p)
        cs.append(p[t[:, 0]])
    return torch.cat(xs), torch.cat(cs)


def _fields(meshes, seed):
    """State and forcing: an elevation of some decimetres, transports of some m^2/s, a wind-sized forcing."""
    rng = np.random.default_rng(seed)
    X, C = _points(meshes)
    f = {"eta": 0.05 + 0.2 * _waves(X, rng),
         "U": torch.stack([4.0 * _waves(C, rng), 4.0 * _waves(C, rng)], dim=1).contiguous(),
         "R": torch.stack([1e-4 * _waves(C, rng), 1e-4 * _waves(C, rng)], dim=1).contiguous()}
    # a shallow coast (10 m on the sphere) keeps small elevations
    H = torch.from_numpy(np.concatenate([m.depth for m in meshes])).to(DEV)
    f["eta"] = f["eta"] * torch.clamp(H / 400.0, max=1.0)
    He = torch.cat([torch.from_numpy(m.depth[m.tri].mean(axis=1)).to(DEV) for m in meshes])
    f["U"] = (f["U"] * torch.clamp(He / 400.0, max=1.0)[:, None]).contiguous()
    f["R"] = (f["R"] * torch.clamp(He / 400.0, max=1.0)[:, None]).contiguous()
    w = torch.from_numpy(rng.normal(size=X.shape[0]) * 2e-6).to(DEV)
    f["W"] = w - w.mean()
    return f


# ------------------------------------------------------------------------------ surrogate inputs

def _shapes():
    s = [(2, HID), (6, HID)] + [(3 * HID, HID), (2 * HID, HID)] * LAYERS + [(HID, 4), (HID, 1)]
    return s


def _weights(rng):
    parts = []
    for k, c in _shapes():
        a = math.sqrt(6.0 / (k + c))
        parts += [rng.uniform(-a, a, k * c), rng.normal(size=c) * 0.05]
    return np.concatenate(parts).astype(np.float32)


def _scales(mesh, h):
    He = mesh.depth[mesh.tri].mean(axis=1)
    # eta, H, U, R, f, length, increments of the transports, increment of the mean elevation
    return np.array([0.2, float(He.max()), 4.0, 1e-4, max(1e-12, float(np.abs(mesh.coriolis).max())), h, 0.8, 0.02])


def _targets(mesh, rng):
    X, C = _points([mesh])
    return [torch.stack([0.8 * _waves(C, rng), 0.8 * _waves(C, rng)], dim=1).contiguous(),
            torch.stack([0.8 * _waves(C, rng), 0.8 * _waves(C, rng)], dim=1).contiguous(), 0.02 * _waves(X, rng)]


def _surrogate_inputs(case, seed):
    mesh, h, dt = _mesh(case)
    rng = np.random.default_rng(seed + 7)
    return mesh, h, dt, _fields([mesh], seed), _weights(rng), _scales(mesh, h), _targets(mesh, rng)


# ------------------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    kind = case["kind"]
    sim = S.Subcycle()
    if kind == "batch":
        meshes, params = _basins(case)
        sim.sesw_mesh_upload_batch(meshes)
        sim.sesw_set_params_batch(params)
        f = _fields(meshes, seed)
    elif kind in ("train", "rollout"):
        mesh, h, dt, f, w, sc, tg = _surrogate_inputs(case, seed)
        sim.sesw_mesh_upload(mesh)
        sim.sesw_set_params(_params(case, h, dt))
        sim.sesw_surrogate_init(1)
        sim.sesw_surrogate_weights(set=w)
        sim.sesw_surrogate_scales(set=sc)
        if kind == "train":
            sim.sesw_surrogate_set_sample(0, f["eta"], f["U"], f["R"], *tg)
    else:
        mesh, h, dt = _mesh(case)
        if kind == "visc":
            sim.sesw_set_mode(S.SESW_MODE_GRAPH)
        sim.sesw_mesh_upload(mesh)
        sim.sesw_set_params(_params(case, h, dt))
        f = _fields([mesh], seed)
        if case["extra"] and kind == "se":
            sim.sesw_set_eta_mean(True)
    st = {"case": case, "sim": sim, "f": f}
    if kind == "host":
        st["f"] = {k: f[k].cpu().pin_memory() for k in ("eta", "U", "R")}
        st["out"] = [torch.empty(n, dtype=torch.float64).pin_memory() for n in
                     ((sim.nv,), (sim.ne, 2), (sim.ne, 2))]
    elif kind != "train":
        st["out"] = [torch.empty(n, dtype=torch.float64, device=DEV) for n in ((sim.nv,), (sim.ne, 2), (sim.ne, 2))]
        st["mean"] = torch.empty(sim.nv, dtype=torch.float64, device=DEV)
    return st


def run(st):
    case, sim, f = st["case"], st["sim"], st["f"]
    kind = case["kind"]
    if kind == "train":
        loss, grad = sim.sesw_surrogate_gradient(0)
        return {"loss": loss, "grad": grad}
    eta, U, Um = st["out"]
    sim.sesw_set_state(f["eta"], f["U"])
    sim.sesw_set_forcing(f["R"])
    if kind == "rollout":
        _, resid = sim.sesw_surrogate_advance(case["steps"], ACCEPT_ALL)
        sim.sesw_get_state(eta, U, Um)
        return {"eta": eta, "U": U, "Umean": Um, "resid": resid}
    if case.get("extra"):
        sim.sesw_set_freshwater(f["W"])
    sim.sesw_advance(case["steps"])
    sim.sesw_get_state(eta, U, Um)
    out = {"eta": eta, "U": U, "Umean": Um}
    if case.get("extra") and kind == "se":
        sim.sesw_get_eta_mean(st["mean"])
        out["eta_mean"] = st["mean"]
    if kind == "host":
        out["volume"], out["energy"] = sim.sesw_diagnostics()
    return out


# ------------------------------------------------------------------------------ work

def _size(case):
    if case["kind"] == "batch":
        ms = _basins(case)[0]
        return sum(m.nv for m in ms), sum(m.ne for m in ms)
    m = _mesh(case)[0]
    return m.nv, m.ne


def work(case):
    """State, forcing and mesh read once, results written once; the operations of every substep or layer."""
    V, E = _size(case)
    kind = case["kind"]
    mesh = 44 * E + 4 * V       # corners, gradients, area, depth, Coriolis; 1 / dual area
    if kind in ("train", "rollout"):
        layers = sum(2 * k * c * (E if i % 2 else V) for i, (k, c) in enumerate(_shapes()[:2 + 2 * LAYERS])
                     if i < 2) + LAYERS * 2 * HID * HID * (3 * E + 2 * V) + 2 * HID * (4 * E + V)
        if kind == "train":
            return {"bytes": mesh + 4 * (2 * V + 8 * E), "flops": 3 * layers}
        return {"bytes": case["steps"] * (mesh + 8 * (2 * V + 8 * E)), "flops": case["steps"] * layers}
    per_e = {"se": 46, "host": 46, "batch": 46, "sesm": 54, "visc": 110}[kind]
    return {"bytes": mesh + 8 * (2 * V + 8 * E) + (16 * V if case.get("extra") else 0),
            "flops": case["steps"] * case["M"] * (per_e * E + 8 * V)}


# ------------------------------------------------------------------------------ the same in 64 bits

class _Geo:
    """A mesh's discrete operators in 64 bits: P1 gradients, areas, median-dual divergence."""

    def __init__(self, meshes):
        off, tri = 0, []
        for m in meshes:
            tri.append(torch.from_numpy(np.asarray(m.tri)).to(DEV).long() + off)
            off += m.nv
        cat = lambda a: torch.from_numpy(np.concatenate(a)).to(DEV)   # noqa: E731
        self.t = torch.cat(tri)
        self.V, self.E = off, self.t.shape[0]
        xy = cat([m.xy for m in meshes])
        self.xy = xy
        a, b, c = xy[:, 0], xy[:, 1], xy[:, 2]
        self.A = 0.5 * ((b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1]) - (c[:, 0] - a[:, 0]) * (b[:, 1] - a[:, 1]))
        self.g = []
        for k in range(3):
            d = xy[:, (k + 2) % 3] - xy[:, (k + 1) % 3]
            self.g.append(torch.stack([-d[:, 1], d[:, 0]], 1) / (2 * self.A)[:, None])
        self.f = cat([m.coriolis for m in meshes])
        H = cat([m.depth for m in meshes])
        self.Hv = H
        self.H0 = (H[self.t[:, 0]] + H[self.t[:, 1]] + H[self.t[:, 2]]) / 3.0
        self.Asum = self.to_vertices([self.A] * 3)
        self.Av = self.Asum / 3.0

    def to_vertices(self, per_corner):
        out = torch.zeros((self.V,) + per_corner[0].shape[1:], dtype=torch.float64, device=DEV)
        for k in range(3):
            out.index_add_(0, self.t[:, k], per_corner[k])
        return out

    def corner_mean(self, x):
        return (x[self.t[:, 0]] + x[self.t[:, 1]] + x[self.t[:, 2]]) / 3.0

    def grad(self, x):
        return sum(x[self.t[:, k]][:, None] * self.g[k] for k in range(3))

    def inflow(self, F):
        """Net flux into each vertex's cell over its area: -div F."""
        w = self.A[:, None] * F
        return self.to_vertices([(w * self.g[k]).sum(1) for k in range(3)]) / self.Av


class _Visc:
    """The two-point flux of the barotropic viscosity, edge by edge (derived here)."""

    def __init__(self, geo, bg, flow):
        self.geo, self.bg, self.flow = geo, bg, flow
        t, xy, E = geo.t, geo.xy, geo.E
        lo = torch.cat([torch.minimum(t[:, k], t[:, (k + 1) % 3]) for k in range(3)])
        hi = torch.cat([torch.maximum(t[:, k], t[:, (k + 1) % 3]) for k in range(3)])
        key = lo * geo.V + hi
        order = torch.argsort(key, stable=True)
        ks = key[order]
        first = torch.nonzero(ks[1:] == ks[:-1])[:, 0]
        i, j = order[first], order[first + 1]
        self.e, self.n = i % E, j % E                    # the two triangles of each interior edge
        ke, kn = i // E, j // E
        # positions: corner k of e joins corner k + 1; in the neighbour the same edge runs backwards
        a1, b1, c1 = (xy[self.e, (ke + q) % 3] for q in range(3))
        b2, a2, c2 = (xy[self.n, (kn + q) % 3] for q in range(3))
        self.va, self.vb = t[self.e, ke], t[self.e, (ke + 1) % 3]
        self.vc1, self.vc2 = t[self.e, (ke + 2) % 3], t[self.n, (kn + 2) % 3]
        d1, d2 = b1 - a1, b2 - a2
        l1, l2 = d1.norm(dim=1), d2.norm(dim=1)
        self.L = 0.5 * (l1 + l2)
        u1, u2 = d1 / l1[:, None], d2 / l2[:, None]
        self.cs = (u1 * u2).sum(1)
        self.sn = u2[:, 0] * u1[:, 1] - u2[:, 1] * u1[:, 0]      # turns the neighbour's frame into e's
        m1, m2 = (a1 + b1 + c1) / 3, (a2 + b2 + c2) / 3
        r = m2 - 0.5 * (a2 + b2)
        r = torch.stack([self.cs * r[:, 0] - self.sn * r[:, 1], self.sn * r[:, 0] + self.cs * r[:, 1]], 1)
        self.d = (0.5 * (a1 + b1) + r - m1).norm(dim=1)

    def __call__(self, U, eta):
        geo = self.geo
        H = geo.H0 + geo.corner_mean(eta)
        u = U / H[:, None]
        un, ue = u[self.n], u[self.e]
        rot = torch.stack([self.cs * un[:, 0] - self.sn * un[:, 1], self.sn * un[:, 0] + self.cs * un[:, 1]], 1)
        du = rot - ue
        He = 0.5 * (H[self.e] + H[self.n])
        A = self.bg + self.flow * du.norm(dim=1) * self.L
        fl = (He * A * self.L / self.d)[:, None] * du
        back = torch.stack([self.cs * fl[:, 0] + self.sn * fl[:, 1], -self.sn * fl[:, 0] + self.cs * fl[:, 1]], 1)
        out = torch.zeros_like(U)
        out.index_add_(0, self.e, fl)
        out.index_add_(0, self.n, -back)
        return out / geo.A[:, None]


def _se_step(geo, eta, U, R, W, dt_e, dt_v, M, visc):
    S_, esum = torch.zeros_like(U), torch.zeros_like(eta)
    a = (0.5 * geo.f * dt_e)[:, None]
    dte = dt_e[:, None]
    sw = torch.tensor([1.0, -1.0], dtype=torch.float64, device=DEV)
    V0 = visc(U, eta) if visc else None
    for m in range(M):
        r = R + (visc(U, eta) - V0) if visc and m else R
        H = geo.H0 + geo.corner_mean(eta)
        rhs = U + a * U.flip(1) * sw + dte * (r - (G * H)[:, None] * geo.grad(eta))
        Un = (rhs + a * rhs.flip(1) * sw) / (1 + a * a)
        F = (1 + THETA) * Un - THETA * U
        S_ += F
        esum += eta
        eta = eta + geo.inflow(dte * F) - dt_v * W
        U = Un
    return eta, U, S_ / M, esum / M


def _sesm_step(geo, eta, U, R, W, dt_e, dt_v, M):
    chi, beta = 0.5 * THETA, 0.281105
    gam, zeta = 0.083 - 0.514 * chi, 0.010 - 0.135 * chi
    delta = 2 * chi + gam + 2 * zeta + 0.5
    ab, am = (1.5 + beta, -(0.5 + 2 * beta), beta), (delta, 1 - delta - gam - zeta, gam, zeta)
    Us, es, S_ = [U] * 3, [eta] * 4, torch.zeros_like(U)
    sw = torch.tensor([1.0, -1.0], dtype=torch.float64, device=DEV)
    dte = dt_e[:, None]
    ab3 = lambda: sum(ab[q] * Us[q] for q in range(3))   # noqa: E731
    for m in range(M):
        F = ab3()
        S_ += F
        es = [es[0] + geo.inflow(dte * F) - dt_v * W] + es[:3]
        ea = sum(am[q] * es[q] for q in range(4))
        H = geo.H0 + geo.corner_mean(ea)
        Un = Us[0] + dte * (geo.f[:, None] * F.flip(1) * sw - (G * H)[:, None] * geo.grad(ea) + R)
        Us = [Un] + Us[:2]
    return es[0], Us[0], S_ / M


def _net(geo, w, sc, eta, U, R):
    """The network's outputs in 64 bits, weights as bfloat16 holds them (biases as they are)."""
    p, o = [], 0
    for k, c in _shapes():
        p.append((w[o:o + k * c].reshape(k, c), w[o + k * c:o + k * c + c]))
        o += k * c + c
    lin = lambda x, q: x @ q[0] + q[1]   # noqa: E731
    hv = torch.tanh(lin(torch.stack([eta / sc[0], geo.Hv / sc[1]], 1), p[0]))
    he = torch.tanh(lin(torch.cat([U / sc[2], R / sc[3], (geo.f / sc[4])[:, None], (geo.H0 / sc[1])[:, None]], 1), p[1]))
    for l in range(LAYERS):
        gx = sc[5] * sum(geo.g[k][:, 0:1] * hv[geo.t[:, k]] for k in range(3))
        gy = sc[5] * sum(geo.g[k][:, 1:2] * hv[geo.t[:, k]] for k in range(3))
        he = he + torch.tanh(lin(torch.cat([he, gx, gy], 1), p[2 + 2 * l]))
        mean = geo.to_vertices([geo.A[:, None] * he] * 3) / geo.Asum[:, None]
        hv = hv + torch.tanh(lin(torch.cat([hv, mean], 1), p[3 + 2 * l]))
    return lin(he, p[2 + 2 * LAYERS]), lin(hv, p[3 + 2 * LAYERS])[:, 0]


def _held(w):
    """The weight vector with its matrices rounded to bfloat16, in 64 bits."""
    x, o = torch.from_numpy(w.copy()), 0
    for k, c in _shapes():
        x[o:o + k * c] = x[o:o + k * c].bfloat16().float()
        o += k * c + c
    return x.double().to(DEV)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "rollout"):
        mesh, h, dt, f, w, sc, tg = _surrogate_inputs(case, seed)
        geo, w = _Geo([mesh]), _held(w)
        if kind == "train":
            w.requires_grad_(True)
            oe, ov = _net(geo, w, sc, f["eta"], f["U"], f["R"])
            te = torch.cat([tg[0], tg[1]], 1) / sc[6]
            loss = (oe - te).square().mean() + (ov - tg[2] / sc[7]).square().mean()
            loss.backward()
            return {"loss": float(loss.detach()), "grad": w.grad.detach()}
        p = _params(case, h, dt)
        eta, U = f["eta"], f["U"]
        for _ in range(case["steps"]):
            oe, ov = _net(geo, w, sc, eta, U, f["R"])
            Um, Un, eb = U + sc[6] * oe[:, 0:2], U + sc[6] * oe[:, 2:4], eta + sc[7] * ov
            dU = Un - U
            sp = Um - (THETA / p.M) * dU - dU / (2 * p.M)
            H = geo.H0 + geo.corner_mean(eb)
            cor = torch.stack([-geo.f * sp[:, 1], geo.f * sp[:, 0]], 1)
            r = dU + p.tau * (cor + (G * H)[:, None] * geo.grad(eb) - f["R"])
            resid = float(((geo.A[:, None] * r * r).sum() / (geo.A[:, None] * dU * dU).sum()).sqrt())
            eta, U = eta + p.tau * geo.inflow(Um), Un
        return {"eta": eta, "U": U, "Umean": Um, "resid": resid}
    if kind == "batch":
        meshes, params = _basins(case)
        dts = [p.tau / p.M for p in params]
    else:
        mesh, h, dt = _mesh(case)
        p = _params(case, h, dt)
        meshes, dts = [mesh], [p.tau / p.M]
    geo = _Geo(meshes)
    f = _fields(meshes, seed)
    dt_e = torch.cat([torch.full((m.ne,), d, dtype=torch.float64, device=DEV) for m, d in zip(meshes, dts)])
    dt_v = torch.cat([torch.full((m.nv,), d, dtype=torch.float64, device=DEV) for m, d in zip(meshes, dts)])
    W = f["W"] if case.get("extra") else torch.zeros(geo.V, dtype=torch.float64, device=DEV)
    visc = _Visc(geo, *p.visc) if kind == "visc" else None
    eta, U, mean = f["eta"], f["U"], None
    for _ in range(case["steps"]):
        if kind == "sesm":
            eta, U, Um = _sesm_step(geo, eta, U, f["R"], W, dt_e, dt_v, case["M"])
        else:
            eta, U, Um, mean = _se_step(geo, eta, U, f["R"], W, dt_e, dt_v, case["M"], visc)
    out = {"eta": eta, "U": U, "Umean": Um}
    if case.get("extra") and kind == "se":
        out["eta_mean"] = mean
    if kind == "host":
        H = geo.H0 + geo.corner_mean(eta)
        out["volume"] = float((geo.Av * eta).sum())
        out["energy"] = float((0.5 * G * geo.Av * eta * eta).sum() + (geo.A * (U * U).sum(1) / (2 * H)).sum())
    return out
