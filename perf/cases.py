"""The work a user of the library has it do, as measurable cases.

Every case goes through the public entry points (``Lattice``, ``Ensemble``,
``MLP``) on the workloads of the benchmark, the tests and the warm-start
study: vessel lattices stepped between two outputs, in each population
storage, alone, batched and monitored; and the warm-start network's forward
pass, training and use.  Fields are returned in the precision the populations
are held in (the library writes them as doubles whatever the storage).

``listed()`` names the cases, ``draw(rng)`` gives others of the same ranges,
``prepare`` / ``run`` set one up and run one pass, ``work`` counts the bytes
and operations a pass cannot do without, and ``exact`` restates a pass in
FP64 with plain torch.
"""
import math

import numpy as np
import torch

import lbm_inputs as I

DEVICE = "cuda"
BYTES = {"f64": 8, "f32": 4, "f16s": 2, "bf16s": 2}
FIELD = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16,
         "bf16s": torch.bfloat16}
F_WALL = 0.85      # wall velocity ratio of every workload of the repository
N_GLOBAL = 5       # run-level features of the warm-start network
FLOP_SITE = 260    # one site update: moments, 19 equilibria, relaxation


def listed():
    return [
        # the short rigid-vs-elastic validation tube, FP64: too small to fill
        # the chip, so what counts is the time from one step to the next
        {"name": "short_tube_f64", "kind": "tube", "storage": "f64", "radius": 8.0, "length": 64,
         "tau": 0.8, "wall": "elastic", "steps": 100},
        # a small tube with an output every 25 steps (an odd number)
        {"name": "short_tube_f32", "kind": "tube", "storage": "f32", "radius": 12.0, "length": 159,
         "tau": 0.8, "wall": "elastic", "steps": 25},
        # the benchmark's long pulsatile tube, FP32 and half-precision storage
        {"name": "long_tube_f32", "kind": "tube", "storage": "f32", "radius": 40.0, "length": 1024,
         "tau": 0.6, "wall": "elastic", "steps": 40},
        {"name": "long_tube_f16s", "kind": "tube", "storage": "f16s", "radius": 40.0,
         "length": 1024, "tau": 0.6, "wall": "elastic", "steps": 40},
        # the same tube with the mass and the inlet and outlet fluxes of every
        # step read back to the host: a run under supervision
        {"name": "monitored_tube_f32", "kind": "monitored", "storage": "f32", "radius": 40.0,
         "length": 1024, "tau": 0.6, "wall": "elastic", "steps": 40},
        # bifurcating vessel trees: oblique vessels, many walls, many outlets
        {"name": "tree_f32", "kind": "tree", "storage": "f32", "depth": 6, "radius": 48.0,
         "tau": 0.6, "wall": "elastic", "steps": 40},
        {"name": "tree_bf16s", "kind": "tree", "storage": "bf16s", "depth": 6, "radius": 40.0,
         "tau": 0.6, "wall": "elastic", "steps": 40},
        # a batch of uneven tubes with their own stiffness, inflow and
        # relaxation time, stepped together between two looks at their fields
        {"name": "ensemble_f16s", "kind": "ensemble", "storage": "f16s", "members": 48,
         "family": 0, "steps": 100},
        {"name": "ensemble_f32", "kind": "ensemble", "storage": "f32", "members": 48,
         "family": 0, "steps": 100},
        # the warm-start network: minibatches of training as the study runs
        # them, one large forward pass, and the start of a tube it proposes
        {"name": "mlp_train", "kind": "mlp_train", "batch": 4096, "width": 256, "layers": 4,
         "steps": 10},
        {"name": "mlp_forward", "kind": "mlp_forward", "rows": 65536, "max_batch": 65536,
         "width": 256, "layers": 4},
        {"name": "warm_start", "kind": "warm_start", "storage": "f32", "radius": 24.0,
         "length": 512, "tau": 0.8, "max_batch": 4096, "width": 256, "layers": 4},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the listed ranges (sizes over their logarithm)."""
    kind = rng.choice(["tube", "tube", "tube", "tree", "tree", "ensemble", "monitored",
                       "mlp_train", "mlp_forward", "warm_start"])
    wall = rng.choice(["elastic", "elastic", "elastic", "bounceback"])
    if kind in ("tube", "monitored"):
        storage = rng.choice(["f64", "f32", "f32", "f16s", "bf16s"])
        radius = round(_log(rng, 5.0, 40.0), 1)
        length = int(_log(rng, 33, 1025))
        # FP64 sites cost ten times an FP32 one's time
        most = (2e8 if storage != "f64" else 2e7) / (math.pi * radius * radius * length)
        return {"kind": kind, "storage": storage, "radius": radius, "length": length,
                "tau": round(rng.uniform(0.6, 1.0), 3), "wall": wall,
                "steps": int(_log(rng, 1, min(101, max(2.0, most))))}
    if kind == "tree":
        return {"kind": kind, "storage": rng.choice(["f32", "f16s", "bf16s"]),
                "depth": rng.randint(2, 6), "radius": round(_log(rng, 12.0, 36.0), 1),
                "tau": round(rng.uniform(0.6, 0.9), 3), "wall": wall,
                "steps": int(_log(rng, 1, 60))}
    if kind == "ensemble":
        return {"kind": kind, "storage": rng.choice(["f32", "f16s", "bf16s"]),
                "members": int(_log(rng, 3, 48)), "family": rng.randrange(1000),
                "steps": int(_log(rng, 5, 100))}
    width, layers = rng.choice([256, 256, 256, 128, 100]), rng.choice([4, 4, 4, 3, 2])
    if kind == "mlp_train":
        return {"kind": kind, "batch": int(_log(rng, 100, 16385)), "width": width,
                "layers": layers, "steps": rng.randint(1, 12)}
    if kind == "mlp_forward":
        rows = int(_log(rng, 100, 131073))
        return {"kind": kind, "rows": rows, "max_batch": rng.choice([rows, 4096, 16384]),
                "width": width, "layers": layers}
    return {"kind": "warm_start", "storage": rng.choice(["f32", "f16s"]),
            "radius": round(_log(rng, 6.0, 24.0), 1), "length": int(_log(rng, 64, 513)),
            "tau": round(rng.uniform(0.6, 1.0), 3), "max_batch": rng.choice([4096, 16384]),
            "width": width, "layers": layers}


# ------------------------------------------------------------------- inputs

_geometry = {}  # voxelised vessels by their sizes: a user voxelises a vessel once


def _members(case, seed):
    """The vessels of a case: (geometry, tau, kappa) with the seed's inflow."""
    kind = case["kind"]
    key = tuple(sorted((k, v) for k, v in case.items()
                       if k in ("kind", "radius", "length", "depth", "members", "family")))
    if key not in _geometry:
        if kind == "tree":
            geo = I.murray_tree(seed=0, depth=case["depth"], root_radius=case["radius"])
            geo.meta.clear()
            made = [(geo, None, 0.75 * case["radius"] / 0.5)]
        elif kind == "ensemble":
            made = [(I.tube(p["radius"], p["length"], u_mean=0.01, u_amp=0.005,
                            period=p["period"]), p["tau"], p["kappa"])
                    for p in I.tube_ensemble(seed=case["family"], count=case["members"],
                                             stiffness=(0.2, 5.0), tau=(0.6, 1.0))]
        else:
            made = [(I.tube(case["radius"], case["length"]), None,
                     0.75 * case["radius"] / 0.5)]
        if len(_geometry) > 16:
            _geometry.clear()
        _geometry[key] = made
    rng = np.random.default_rng([seed, 1])
    out = []
    for geo, tau, kappa in _geometry[key]:
        inlet = geo.iolets[0]
        if kind != "ensemble":
            inlet.u_mean, inlet.u_amp, inlet.period = 0.025, 0.015, 4000.0
            # a narrower vessel carries a slower flow: the density drop of a
            # tube is 24 nu L u / R^2, held to a few percent here
            if kind in ("tube", "monitored"):
                nu = (case["tau"] - 0.5) / 3.0
                u = min(0.03, 0.08 * case["radius"] ** 2 / (24.0 * nu * case["length"]))
                inlet.u_mean, inlet.u_amp = u, 0.6 * u
        inlet.phase = float(rng.uniform(0.0, 2.0 * math.pi))
        out.append((geo, case["tau"] if tau is None else tau, kappa))
    return out


def _coords(labels):
    """Fluid voxels in canonical order (z fastest), as a device tensor [n][3]."""
    parts = []
    slab = max(1, (1 << 28) // (labels.shape[1] * labels.shape[2]))
    for x0 in range(0, labels.shape[0], slab):
        c = torch.nonzero(torch.from_numpy(labels[x0:x0 + slab]).to(DEVICE) == 1)
        c[:, 0] += x0
        parts.append(c.to(torch.int32))
    return torch.cat(parts)


def _fields(coords, seed):
    """Smooth flow fields of the seed: |rho - 1| <= 1e-3, |u_k| <= 0.01."""
    g = np.random.default_rng([seed, 2])
    waves = []
    for k in range(4):
        v = g.normal(size=3)
        v *= 2.0 * math.pi / (g.uniform(24.0, 64.0) * np.linalg.norm(v))
        waves.append((v, g.uniform(0.0, 2.0 * math.pi)))
    c = coords.to(torch.float64)
    s = [torch.sin(c[:, 0] * v[0] + c[:, 1] * v[1] + c[:, 2] * v[2] + ph) for v, ph in waves]
    return 1.0 + 1e-3 * s[0], torch.stack([0.01 * a for a in s[1:]], 1)


def _lattice(geo, storage, tau, kappa, wall):
    from paper_2108_08783_gb300 import Lattice
    lat = Lattice(geo.labels, geo.iolets, storage=storage, tau=tau)
    lat.set_wall(wall, rho0=1.0, F=F_WALL, kappa=kappa)
    return lat


def _network(case, seed):
    from paper_2108_08783_gb300 import MLP
    net = MLP(N_GLOBAL + 2, case["width"], case["layers"], 3,
              max_batch=case.get("max_batch", case.get("batch")))
    net.set_params(_theta(case, seed))
    return net


def _theta(case, seed):
    return I.mlp_init(seed, N_GLOBAL + 2, case["width"], case["layers"], 3, bias_scale=0.1)


def _samples(seed, m):
    """Training pairs in the ranges of the tube family's features and scaled fields."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    x = torch.rand(m, N_GLOBAL + 2, device=DEVICE, generator=g)
    x[:, 2] = x[:, 2] * 2.0 - 1.3  # log10 of the stiffness
    xi, eta = x[:, N_GLOBAL], x[:, N_GLOBAL + 1]
    t = torch.stack([(1.0 - xi) * (0.5 + x[:, 0]), 0.05 * torch.sin(6.0 * xi) * eta,
                     2.0 * (1.0 - eta * eta) * (0.8 + 0.4 * x[:, 3])], 1)
    return x, t


def _tube_frame(case, seed):
    """What lbm_warm_frame holds for the case's tube and the seed's run."""
    r, length, tau = case["radius"], case["length"], case["tau"]
    g = np.random.default_rng([seed, 3])
    u, eh = g.uniform(0.01, 0.04), math.exp(g.uniform(math.log(0.05), math.log(5.0)))
    c = (int(2 * math.ceil(r) + 4) - 1) / 2.0
    feats = [r / 24.0, length / 512.0, math.log10(eh), u / 0.04, 2.0 * (tau - 0.5)]
    return dict(centre=(c, c, 0.0), axis=(0.0, 0.0, 1.0), z0=0.5, length=length, radius=r,
                features=feats, rho_scale=24.0 * (tau - 0.5) / 3.0 * length * u / r ** 2,
                u_scale=u)


# --------------------------------------------------------------------- a pass

class _Fields:
    """Device buffers of a lattice's (or several lattices') density and velocity."""

    def __init__(self, n, storage):
        self.rho = torch.empty(n, dtype=torch.float64, device=DEVICE)
        self.u = torch.empty((n, 3), dtype=torch.float64, device=DEVICE)
        self.dtype = FIELD[storage]

    def take(self, lats):
        at = 0
        for lat in lats:
            lat.moments_into(self.rho[at:at + lat.n], self.u[at:at + lat.n])
            at += lat.n
        # the density as its deviation from 1, which 16 bits can hold
        return (self.rho - 1.0).to(self.dtype), self.u.to(self.dtype)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp_train":
        x, t = _samples(seed, case["batch"] * case["steps"])
        return dict(case=case, net=_network(case, seed), x=x, t=t)
    if kind == "mlp_forward":
        return dict(case=case, net=_network(case, seed), x=_samples(seed, case["rows"])[0])
    if kind == "warm_start":
        from paper_2108_08783_gb300 import warm_frame
        geo = I.tube(case["radius"], case["length"], u_mean=0.02)
        lat = _lattice(geo, case["storage"], case["tau"], 12.0, "elastic")
        return dict(case=case, net=_network(case, seed), lat=lat,
                    frame=warm_frame(**_tube_frame(case, seed)),
                    fields=_Fields(lat.n, case["storage"]))
    lats = []
    for k, (geo, tau, kappa) in enumerate(_members(case, seed)):
        lat = _lattice(geo, case["storage"], tau, kappa, case.get("wall", "elastic"))
        rho, u = _fields(_coords(geo.labels), seed + 1000 * k)
        lat.init_fields(rho.cpu().numpy(), u.cpu().numpy())
        lats.append(lat)
    state = dict(case=case, lats=lats, fields=_Fields(sum(l.n for l in lats), case["storage"]))
    if kind == "ensemble":
        from paper_2108_08783_gb300 import Ensemble
        state["ens"] = Ensemble(lats)
    if kind == "monitored":
        state["ring"] = torch.zeros((case["steps"], 1 + lats[0].n_iolets), dtype=torch.float64,
                                    pin_memory=True)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "tube" or kind == "tree":
        lat = state["lats"][0]
        lat.step(case["steps"])
        drho, u = state["fields"].take([lat])
        return {"drho": drho, "u": u}
    if kind == "monitored":
        lat, ring = state["lats"][0], state["ring"].numpy()
        for k in range(case["steps"]):
            lat.step_diag(1, out=ring[k])
        drho, u = state["fields"].take([lat])
        lat.sync()  # the rows are complete, and the run is checked for instability
        diag = state["ring"].clone() if case["storage"] == "f64" else state["ring"].float()
        return {"diagnostics": diag, "drho": drho, "u": u}
    if kind == "ensemble":
        ens = state["ens"]
        ens.step(case["steps"])
        ens.sync()
        drho, u = state["fields"].take(state["lats"])
        return {"drho": drho, "u": u}
    net = state["net"]
    if kind == "mlp_train":
        b = case["batch"]
        for k in range(case["steps"]):
            net.train_step(state["x"][k * b:(k + 1) * b], state["t"][k * b:(k + 1) * b], lr=1e-3)
        return net.params()
    if kind == "mlp_forward":
        return net.forward(state["x"])
    lat = state["lat"]
    lat.warm_start(net, state["frame"])
    drho, u = state["fields"].take([lat])
    return {"drho": drho, "u": u}


def _sites(case):
    if case["kind"] == "warm_start":
        case = dict(case, kind="tube")
    return sum(geo.n_fluid() for geo, _, _ in _members(case, 0))


def work(case):
    kind = case["kind"]
    if kind in ("mlp_train", "mlp_forward"):
        shapes = I.mlp_shapes(N_GLOBAL + 2, case["width"], case["layers"], 3)
        macs = sum(r * c for r, c in shapes)
        params = sum(r * c + r for r, c in shapes)
        if kind == "mlp_forward":
            rows = case["rows"]
            return {"bytes": 4 * (rows * (N_GLOBAL + 5) + params), "flops": 2 * macs * rows}
        # forward, input errors (all layers but the first) and weight gradients;
        # samples read once, parameters and both Adam moments read and written
        b, steps = case["batch"], case["steps"]
        return {"bytes": steps * 4 * (b * (N_GLOBAL + 5) + 6 * params),
                "flops": steps * 2 * b * (3 * macs - shapes[0][0] * shapes[0][1])}
    n, size = _sites(case), BYTES[case["storage"]]
    fields = 4 * size * n  # the fields handed back
    if kind == "warm_start":
        shapes = I.mlp_shapes(N_GLOBAL + 2, case["width"], case["layers"], 3)
        return {"bytes": 19 * size * n + fields, "flops": 2 * n * sum(r * c for r, c in shapes)}
    # every step reads and writes the 19 populations of every site
    return {"bytes": case["steps"] * 38 * size * n + fields,
            "flops": case["steps"] * FLOP_SITE * n}


# ------------------------------------------------------- the same pass in FP64

_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
      (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
_OPP = [_C.index((-a, -b, -c)) for a, b, c in _C]


def _exact_flow(case, seed):
    """LBGK with two population arrays: collide everywhere, then every site
    pulls each direction from its neighbour or rebuilds it at the boundary."""
    f64 = dict(dtype=torch.float64, device=DEVICE)
    rhos, us, omegas, kappas, nbrs = [], [], [], [], [[] for _ in _C]
    iolets, profiles, at = [], [], 0
    for k, (geo, tau, kappa) in enumerate(_members(case, seed)):
        xyz = _coords(geo.labels).long()
        n = xyz.shape[0]
        nx, ny, nz = (s + 2 for s in geo.labels.shape)
        grid = torch.full((nx, ny, nz), -1, dtype=torch.int32, device=DEVICE)
        inner = grid[1:-1, 1:-1, 1:-1]
        lab = torch.from_numpy(geo.labels).to(DEVICE)
        for q in range(len(geo.iolets)):
            inner[lab == 2 + q] = -2 - (len(iolets) + q)
        del lab
        flat = grid.view(-1)
        here = ((xyz[:, 0] + 1) * ny + xyz[:, 1] + 1) * nz + xyz[:, 2] + 1
        flat[here] = torch.arange(at, at + n, dtype=torch.int32, device=DEVICE)
        for i, (a, b, c) in enumerate(_C):
            nbrs[i].append(flat[here + (a * ny + b) * nz + c])
        del grid, flat, inner, here
        for io in geo.iolets:
            ax = np.asarray(io.axis) / np.linalg.norm(io.axis)
            d = xyz.to(torch.float64) - torch.tensor(io.centre, **f64)
            along = d @ torch.tensor(ax, **f64)
            r2 = (d * d).sum(1) - along * along
            iolets.append((io, ax, at))
            profiles.append((2.0 * (1.0 - r2 / io.radius ** 2)).clamp_min(0.0))
        rho, u = _fields(xyz.to(torch.int32), seed + 1000 * k)
        rhos.append(rho)
        us.append(u)
        omegas.append(torch.full((n,), 1.0 / tau, **f64))
        kappas.append(torch.full((n,), kappa, **f64))
        at += n
    nbr = [torch.cat(v) for v in nbrs]
    omega, kappa = torch.cat(omegas), torch.cat(kappas)
    elastic = case.get("wall", "elastic") == "elastic"

    def equilibrium(i, rho, ux, uy, uz):
        a, b, c = _C[i]
        cu = a * ux + b * uy + c * uz
        return _W[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu
                              - 1.5 * (ux * ux + uy * uy + uz * uz))

    # links leaving the fluid, by the direction j they rebuild: (sites, iolet or -1)
    leaving = [[] for _ in _C]
    touches = {}
    for j in range(1, 19):
        code = nbr[_OPP[j]]
        out = torch.nonzero(code < 0).squeeze(1)
        which = -2 - code[out]
        for q in torch.unique(which).tolist():
            sites = out[which == q]
            leaving[j].append((q, sites))
            if q >= 0:
                touches.setdefault(q, []).append(sites)
    touches = {q: torch.unique(torch.cat(v)) for q, v in touches.items()}

    rho, u = torch.cat(rhos), torch.cat(us)
    f = [equilibrium(i, rho, u[:, 0], u[:, 1], u[:, 2]) for i in range(19)]

    def moments():
        rho = f[0].clone()
        j = [torch.zeros_like(rho) for _ in range(3)]
        for i in range(1, 19):
            rho += f[i]
            for d in range(3):
                if _C[i][d]:
                    j[d] += _C[i][d] * f[i]
        return rho, [v / rho for v in j]

    diag = []
    for n in range(case["steps"]):
        rho, (ux, uy, uz) = moments()
        if case["kind"] == "monitored":
            row = [float(rho.sum())]
            for q, (io, ax, _) in enumerate(iolets):
                s = touches[q]
                row.append(float((rho[s] * (ux[s] * ax[0] + uy[s] * ax[1] + uz[s] * ax[2])).sum()))
            diag.append(row)
        new = [None] * 19
        back = []  # boundary values, from the state before the collision
        for j in range(1, 19):
            i = _OPP[j]
            for q, s in leaving[j]:
                r, a, b, c, om = rho[s], ux[s], uy[s], uz[s], omega[s]
                if q == -1 and not elastic:
                    back.append((j, s, f[i][s] + om * (equilibrium(i, r, a, b, c) - f[i][s])))
                    continue
                keep = (1.0 - om) * (f[j][s] - equilibrium(j, r, a, b, c))
                if q == -1:
                    de = kappa[s] * ((r - 1.0) / 3.0).clamp_min(0.0)
                    w = (F_WALL + de) / (1.0 + de)
                    back.append((j, s, equilibrium(j, r, w * a, w * b, w * c) + keep))
                    continue
                io, ax, first = iolets[q]
                if io.kind == 0:
                    g = io.u_mean
                    if io.period > 0:
                        g += io.u_amp * math.sin(2.0 * math.pi * n / io.period + io.phase)
                    v = g * profiles[q][s - first]
                    back.append((j, s, equilibrium(j, r, v * ax[0], v * ax[1], v * ax[2]) + keep))
                else:
                    back.append((j, s, equilibrium(j, torch.full_like(r, io.rho), a, b, c) + keep))
        for i in range(19):
            star = f[i] + omega * (equilibrium(i, rho, ux, uy, uz) - f[i])
            new[i] = star if i == 0 else star[nbr[_OPP[i]].clamp_min(0)]
        for j, s, v in back:
            new[j][s] = v
        f[:] = new
    rho, u = moments()
    out = {"drho": rho - 1.0, "u": torch.stack(u, 1)}
    if case["kind"] == "monitored":
        out["diagnostics"] = torch.tensor(diag, dtype=torch.float64)
    return out


def _exact_layers(case, theta):
    layers, o = [], 0
    for r, c in I.mlp_shapes(N_GLOBAL + 2, case["width"], case["layers"], 3):
        layers.append((theta[o:o + r * c].view(r, c), theta[o + r * c:o + r * c + r]))
        o += r * c + r
    return layers


def _exact_forward(case, theta, x):
    hs = [x.double()]
    layers = _exact_layers(case, theta)
    for l, (w, b) in enumerate(layers):
        z = hs[-1] @ w.T + b
        hs.append(z if l == len(layers) - 1 else torch.tanh(z))
    return hs


def exact(case, seed):
    kind = case["kind"]
    if kind in ("tube", "tree", "monitored", "ensemble"):
        return _exact_flow(case, seed)
    theta = torch.from_numpy(_theta(case, seed)).to(DEVICE).double()
    if kind == "mlp_forward":
        return _exact_forward(case, theta, _samples(seed, case["rows"])[0])[-1]
    if kind == "mlp_train":
        x, t = _samples(seed, case["batch"] * case["steps"])
        m, v, b = torch.zeros_like(theta), torch.zeros_like(theta), case["batch"]
        for k in range(case["steps"]):
            hs = _exact_forward(case, theta, x[k * b:(k + 1) * b])
            d = 2.0 * (hs[-1] - t[k * b:(k + 1) * b].double()) / (3 * b)
            grads = []
            for l, (w, _) in reversed(list(enumerate(_exact_layers(case, theta)))):
                grads += [d.sum(0), (d.T @ hs[l]).reshape(-1)]
                if l:
                    d = (d @ w) * (1.0 - hs[l] ** 2)
            g = torch.cat(grads[::-1])
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            theta = theta - 1e-3 * (m / (1 - 0.9 ** (k + 1))) / (
                (v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
        return theta
    fr = _tube_frame(case, seed)
    xyz = _coords(I.tube(case["radius"], case["length"]).labels).double()
    d = xyz[:, :2] - torch.tensor(fr["centre"][:2], dtype=torch.float64, device=DEVICE)
    r = d.norm(dim=1)
    er = d / r.clamp_min(1e-300)[:, None] * (r > 1e-12)[:, None]
    x = torch.empty((xyz.shape[0], N_GLOBAL + 2), dtype=torch.float64, device=DEVICE)
    x[:, :N_GLOBAL] = torch.tensor(fr["features"], dtype=torch.float64, device=DEVICE)
    x[:, N_GLOBAL] = (xyz[:, 2] - fr["z0"]) / fr["length"]
    x[:, N_GLOBAL + 1] = r / fr["radius"]
    y = _exact_forward(case, theta, x)[-1]
    u = fr["u_scale"] * torch.cat([y[:, 1:2] * er, y[:, 2:3]], 1)
    return {"drho": fr["rho_scale"] * y[:, 0], "u": u}
