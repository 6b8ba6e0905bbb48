"""Performance cases of the library: what its users run, over the range of
sizes, storages and options that they run it with.

A droplet case is one interval of a simulation between two observations, as
the monitor, the warm-start campaign and the late-spreading run make it:
`steps` time steps, then the observables and the node positions of every
droplet, and for single droplets up to a few million cells the density and
velocity fields of a snapshot.  Each pass continues the run.  The other
kinds are a run steered from the host step by step (`monitor`), and training
and inference of the warm-start network (`train`, `predict`).

`exact` restates the time step and the network in plain torch, FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from paper_2503_20605_gb300 import warmstart as W

STORE_BYTES = {"f32": 4, "f16": 2, "bf16": 2}
ZCUT, EPS_FLAT = 0.05, 0.1          # the paper's contact-radius parameters


def _drop(name, nx, ny, nz, R, level, theta, storage, steps, sigma=0.005, xi=2.0, tau=1.0, lam=1.0, volcorr=True,
          fields=True, start="sphere", walls=True, ks=0.0, ka=0.0, kind="drop"):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "R": R, "level": level, "theta": theta,
            "storage": storage, "steps": steps, "sigma": sigma, "xi": xi, "tau": tau, "lam": lam,
            "volcorr": volcorr, "fields": fields, "start": start, "walls": walls, "ks": ks, "ka": ka}


def listed():
    return [
        # the smallest droplet: 32^3 in FP32 without volume correction (parity
        # and convergence checks, quick parameter scans); five short kernels a step
        _drop("parity32_f32", 32, 32, 32, 8.0, 3, 90.0, "f32", 500, sigma=0.01, volcorr=False),
        # the paper's statics setting (Sec. III A): 80 x 80 x 60, R0 = 20, 20 480
        # triangles, acute angle
        _drop("statics80_f32", 80, 80, 60, 20.0, 5, 45.0, "f32", 500, xi=4.0),
        # the 128^3 statics droplet of the benchmark, 16-bit and FP32 storage
        _drop("statics128_f16", 128, 128, 128, 24.0, 5, 90.0, "f16", 500, xi=2.4),
        _drop("statics128_f32", 128, 128, 128, 24.0, 5, 90.0, "f32", 300, xi=2.4),
        # the same droplet steered from the host: positions up, one step,
        # positions and observables down, every step (one call's latency)
        _drop("monitor128_f16", 128, 128, 128, 24.0, 5, 90.0, "f16", 1, xi=2.4, fields=False, kind="monitor"),
        # early spreading, viscosity ratio 10 (ray casting every step), BF16
        _drop("spreading256_bf16", 256, 256, 128, 40.0, 6, 20.0, "bf16", 100, tau=0.8, lam=10.0, fields=False),
        # 64 independent droplets of uneven sizes in one context (a parameter study)
        {"name": "batch64_f16", "kind": "batch", "n": 64, "spec_seed": 2025, "storage": "f16", "steps": 50},
        # the warm-start campaign's contexts: uneven boxes, viscosity ratios of 0.1 to 10
        {"name": "warm32_f16", "kind": "warm", "n": 32, "spec_seed": 1, "storage": "f16", "steps": 100},
        # late (viscous) spreading from a spherical cap, R0 = 60 with 327 680
        # triangles: the largest mesh
        _drop("tanner60_f16", 320, 320, 98, 60.0, 7, 22.5, "f16", 100, sigma=0.01, xi=3.0, fields=False, start="cap"),
        # an elastic (Skalak) capsule relaxing in a box periodic in all three
        # directions, odd sides
        _drop("capsule_f32", 61, 53, 47, 12.0, 4, 0.0, "f32", 500, sigma=0.0, volcorr=False, start="stretched",
              walls=False, ks=0.02, ka=0.1),
        # the network on a campaign's 1546 equilibria, batches of 128
        {"name": "train1546", "kind": "train", "samples": 1546, "batch": 128, "epochs": 4},
        # predicted shapes of a held-out set: one short call
        {"name": "predict200", "kind": "predict", "samples": 200, "max_batch": 256},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["drop", "drop", "drop", "drop", "monitor", "batch", "warm", "train", "predict"])
    if kind == "train":
        batch = round(_log(rng, 32, 512))
        return {"kind": "train", "samples": batch + rng.randrange(1, 1200), "batch": batch,
                "epochs": rng.randrange(1, 4)}
    if kind == "predict":
        return {"kind": "predict", "samples": round(_log(rng, 1, 5000)), "max_batch": rng.choice([64, 200, 256, 1000])}
    storage = rng.choice(["f32", "f16", "bf16"])
    if kind in ("batch", "warm"):
        return {"kind": kind, "n": round(_log(rng, 3, 32)), "spec_seed": rng.randrange(1, 1 << 20), "storage": storage,
                "steps": rng.randrange(20, 50)}
    R = _log(rng, 6.0, 30.0)
    xi = max(2.0, 0.1 * R)
    theta = rng.uniform(40.0, 150.0)
    nx, ny, nz = W.case_box(theta, R, xi)
    nx, ny, nz = nx + rng.randrange(0, 12), ny + rng.randrange(0, 12), nz + rng.randrange(0, 8)
    lam = 1.0 if rng.random() < 0.6 else _log(rng, 0.2, 8.0)
    # relaxation times within the campaign's range when the viscosities differ
    tau = rng.uniform(0.7, 1.2) if lam == 1.0 else W.tau_out_for(lam)
    c = _drop("", nx, ny, nz, R, I.level_for_radius(R), theta, storage, 1 if kind == "monitor" else rng.randrange(50, 300),
              sigma=rng.uniform(0.004, 0.01), xi=xi, tau=tau, lam=lam, volcorr=rng.random() < 0.7,
              fields=kind == "drop" and nx * ny * nz < 1_500_000, kind=kind)
    del c["name"]
    return c


# ------------------------------------------------------------------- inputs
def _rotated_sphere(level, R, rng):
    """Icosphere of radius R about the origin, turned by a random rotation."""
    xyz, tri = I.icosphere(level, R)
    q, r = np.linalg.qr(rng.normal(size=(3, 3)))
    q = q * np.sign(np.diag(r))
    if np.linalg.det(q) < 0.0:
        q[:, 0] = -q[:, 0]
    return xyz @ q.T, tri


def _specs(case):
    """One droplet case for every droplet of the case's context."""
    if case["kind"] == "batch":
        src = I.workload_batch(case["n"], case["spec_seed"], case["storage"])
    elif case["kind"] == "warm":
        src = [W.case_spec(t, R, lam, case["storage"]) for t, R, lam in I.warmstart_cases(case["n"], case["spec_seed"])]
    else:
        return [case]
    return [_drop("", s.nx, s.ny, s.nz, s.R, s.level, s.theta_deg, s.storage, case["steps"], sigma=s.sigma, xi=s.xi,
                  tau=s.tau, lam=s.lam, fields=False) for s in src]


def _mesh(spec, rng):
    """(mesh given to the library, positions it then starts from or None, faces):
    the droplet a fraction of a cell off the middle, turned, at h = xi."""
    sx, sy = rng.uniform(-0.5, 0.5, 2)
    cx, cy = spec["nx"] / 2.0 + sx, spec["ny"] / 2.0 + sy
    xyz, tri = _rotated_sphere(spec["level"], spec["R"], rng)
    if spec["start"] == "cap":
        g = iblb.iblb_cap_profile(90.0)
        return iblb.iblb_deform_mesh(g, spec["R"], xyz, tri, cx, cy, 0.5 + spec["xi"]), None, tri
    cz = spec["nz"] / 2.0 + rng.uniform(-0.5, 0.5) if not spec["walls"] else 0.5 + spec["R"] + spec["xi"]
    c = np.array([cx, cy, cz])
    if spec["start"] == "stretched":
        s = rng.uniform(1.15, 1.3)
        return xyz + c, xyz * np.array([s, 1.0 / math.sqrt(s), 1.0 / math.sqrt(s)]) + c, tri
    return xyz + c, None, tri


def _network_data(case, seed):
    """Cases (theta_eq, R0, lambda) and the profile of the spherical cap of
    that angle about its mid-height, with the scatter of binned mesh nodes."""
    n = case["samples"]
    x = I.warmstart_cases(n, seed)
    th = np.radians(x[:, :1])
    c = np.cos(th)
    rho = (4.0 / (2.0 - 3.0 * c + c ** 3)) ** (1.0 / 3.0)
    zc = 0.5 * rho * (1.0 - c)
    phi = (np.arange(iblb.NPHI) + 0.5)[None, :] * math.pi / iblb.NPHI
    d = zc + rho * c                 # height of the start point above the sphere's centre
    b = d * np.cos(phi)
    r = -b + np.sqrt(b * b + rho * rho - d * d)
    base = np.where(np.cos(phi) < 0.0, zc / np.maximum(-np.cos(phi), 1e-12), np.inf)
    return x, np.minimum(r, base) + 2e-3 * np.random.default_rng(seed + 7).normal(size=(n, iblb.NPHI))


class _Run:
    """A context or a network with what the program keeps beside it."""

    def __init__(self, case):
        self.case, self.ctx, self.net = case, None, None

    def __del__(self):
        if self.ctx is not None:
            iblb.iblb_destroy(self.ctx)
        if self.net is not None:
            iblb.iblb_mlp_destroy(self.net)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    s = _Run(case)
    if case["kind"] in ("train", "predict"):
        s.x, s.y = _network_data(case, seed)
        params = I.mlp_init(seed) if case["kind"] == "train" else W.load_params()
        s.net = iblb.iblb_mlp_create(params, case["batch"] if case["kind"] == "train" else case["max_batch"], _stream())
        return s
    specs = _specs(case)
    s.n = len(specs)
    s.ctx = iblb.iblb_batch_create(
        [iblb.lattice_desc(p["nx"], p["ny"], p["nz"], tau_out=p["tau"], lam=p["lam"], storage=p["storage"],
                           walls=int(p["walls"])) for p in specs],
        [iblb.physics_desc(sigma=p["sigma"], theta_eq_deg=p["theta"] if p["walls"] else None, xi=p["xi"],
                           volume_correction=p["volcorr"], shear_modulus=p["ks"], area_modulus=p["ka"])
         for p in specs], _stream())
    rng = np.random.default_rng(seed)
    for k, p in enumerate(specs):
        xyz, moved, tri = _mesh(p, rng)
        iblb.iblb_set_membrane(s.ctx, k, xyz, tri)
        if moved is not None:
            iblb.iblb_set_nodes(s.ctx, k, moved)
    if case["kind"] == "monitor":
        # page-locked buffers, as a program that transfers every step keeps them
        s.up = torch.from_numpy(xyz).pin_memory().numpy()
        s.down = torch.empty(xyz.shape, dtype=torch.float64, pin_memory=True).numpy()
    return s


def run(s):
    c = s.case
    if c["kind"] == "predict":
        return iblb.iblb_mlp_predict(s.net, s.x)
    if c["kind"] == "train":
        losses = iblb.iblb_mlp_train(s.net, s.x, s.y, c["epochs"], c["batch"], 1e-3, 0)
        return {"losses": losses, "params": iblb.iblb_mlp_get_params(s.net)}
    if c["kind"] == "monitor":
        iblb.iblb_set_nodes(s.ctx, 0, s.up)
        iblb.iblb_step(s.ctx, 1)
        return {"nodes": iblb.iblb_get_nodes(s.ctx, 0, s.down), "obs": iblb.iblb_observe(s.ctx, 0, ZCUT, EPS_FLAT)}
    iblb.iblb_step(s.ctx, c["steps"])
    if s.n > 1:
        obs = _columns(iblb.iblb_observe_all(s.ctx, ZCUT, EPS_FLAT))
        return {"obs": obs, "nodes": np.concatenate([iblb.iblb_get_nodes(s.ctx, k) for k in range(s.n)])}
    out = {"obs": iblb.iblb_observe(s.ctx, 0, ZCUT, EPS_FLAT), "nodes": iblb.iblb_get_nodes(s.ctx, 0)}
    if c["fields"]:
        out["rho"], out["u"] = iblb.iblb_get_macros(s.ctx, 0)
    return out


def _columns(obs):
    return {k: np.array([o[k] for o in obs]) for k in obs[0]}


def work(case):
    if case["kind"] in ("train", "predict"):
        n, p = case["samples"], I.mlp_init(0).size
        dense = 2.0 * (3 * 256 + 2 * 256 * 256 + 256 * 64)
        if case["kind"] == "predict":
            return {"bytes": n * (3 + 64) * 8.0 + 4.0 * p, "flops": n * dense}
        used = case["epochs"] * (n // case["batch"])
        # parameters and two moments read and written, samples read once
        return {"bytes": n * 67 * 8.0 + 24.0 * p, "flops": used * (3.0 * case["batch"] * dense + 12.0 * p)}
    nbytes = flops = 0.0
    for s in _specs(case):
        cells = s["nx"] * s["ny"] * (s["nz"] - 2 * int(s["walls"]))
        nodes = 10 * 4 ** s["level"] + 2
        # a step reads and writes every population and node position once;
        # about 250 operations a cell, 64 stencil cells both ways and the faces a node
        nbytes += s["steps"] * (38.0 * STORE_BYTES[s["storage"]] * cells + 48.0 * nodes)
        flops += s["steps"] * (250.0 * cells + 1500.0 * nodes)
        # the observables' mass and the snapshot read the populations once more
        nbytes += cells * (19.0 * STORE_BYTES[s["storage"]] + (32.0 if s["fields"] else 0.0)) + 24.0 * nodes
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------ the same in 64 bits
_C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
               (1, -1, 0), (-1, 1, 0), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1), (1, 0, 1), (-1, 0, -1),
               (1, 0, -1), (-1, 0, 1)])
_WT = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
_OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]


def _norm(v):
    return torch.sqrt((v * v).sum(-1))


class _Exact:
    """One droplet's time step (Sec. II) in FP64."""

    def __init__(self, spec, mesh, device):
        self.p, self.dev = spec, device
        self.walls = int(spec["walls"])
        self.nx, self.ny, self.nz = spec["nx"], spec["ny"], spec["nz"] - 2 * self.walls
        xyz, moved, tri = mesh
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=device)  # noqa: E731
        self.ref, self.tri = t(xyz), t(tri.astype(np.int64))
        self.q = t(moved) if moved is not None else self.ref.clone()
        self.V0 = float(self.volume(self.ref))
        self.R0 = (3.0 * self.V0 / (4.0 * math.pi)) ** (1.0 / 3.0)
        self.s = torch.zeros((19, self.nz, self.ny, self.nx), dtype=torch.float64, device=device)  # f_i - w_i
        self.rho = self.u = None

    def volume(self, q):
        a, b, c = q[self.tri[:, 0]], q[self.tri[:, 1]], q[self.tri[:, 2]]
        return (a * torch.linalg.cross(b, c)).sum() / 6.0

    def node_forces(self):
        p, q, tri = self.p, self.q, self.tri
        n = len(q)
        v = [q[tri[:, k]] for k in range(3)]
        N = torch.linalg.cross(v[1] - v[0], v[2] - v[0])
        length = _norm(N)
        hat, area = N / length[:, None], 0.5 * length
        zero = torch.zeros((n, 3), dtype=torch.float64, device=self.dev)
        # dA/dq_k = n x (q_k+2 - q_k+1) / 2
        grad = [0.5 * torch.linalg.cross(hat, v[(k + 2) % 3] - v[(k + 1) % 3]) for k in range(3)]
        phi, normal = zero.clone(), zero.clone()
        chi = torch.zeros(n, dtype=torch.float64, device=self.dev)
        for k in range(3):
            phi.index_add_(0, tri[:, k], -p["sigma"] * grad[k])
            normal.index_add_(0, tri[:, k], hat)
            chi.index_add_(0, tri[:, k], area)
        if p["ks"] or p["ka"]:
            E1, E2 = self.ref[tri[:, 1]] - self.ref[tri[:, 0]], self.ref[tri[:, 2]] - self.ref[tri[:, 0]]
            e1, e2 = v[1] - v[0], v[2] - v[0]
            H = torch.stack([(E1 * E1).sum(-1), (E1 * E2).sum(-1), (E2 * E2).sum(-1)])
            det = H[0] * H[2] - H[1] * H[1]
            S11, S12, S22 = H[2] / det, -H[1] / det, H[0] / det
            A0 = 0.5 * torch.sqrt(det)
            trace = S11 * (e1 * e1).sum(-1) + 2.0 * S12 * (e1 * e2).sum(-1) + S22 * (e2 * e2).sum(-1)
            b, r = 0.5 * trace - 1.0, area / A0
            # w = ks/12 (I1^2 + 2 I1 - 2 I2) + ka/12 I2^2, I1 = 2 b, I2 = r^2 - 1
            w_r = (-p["ks"] + p["ka"] * (r * r - 1.0)) * r / 3.0
            w_b = p["ks"] * (2.0 * b + 1.0) / 3.0
            h1 = S11[:, None] * e1 + S12[:, None] * e2
            h2 = S12[:, None] * e1 + S22[:, None] * e2
            half = [-(h1 + h2), h1, h2]      # half the trace's gradient at each corner
            for k in range(3):
                phi.index_add_(0, tri[:, k], -w_r[:, None] * grad[k] - (A0 * w_b)[:, None] * half[k])
        if p["walls"]:
            A = p["sigma"] * 10.0 / (3.0 * p["xi"]) * (1.0 + math.cos(math.radians(p["theta"])))
            x = p["xi"] / torch.clamp(q[:, 2] - 0.5, min=0.5 * p["xi"])
            Pi = A * (x ** 6 - x ** 3)
            phi += (-(chi / 3.0) * Pi / _norm(normal))[:, None] * normal
        return phi

    def stencil(self):
        """Cell indices and weights of every node's 4 x 4 x 4 support (-1: no fluid cell)."""
        base = torch.floor(self.q)
        d = torch.arange(-1, 3, device=self.dev)
        f = self.q - base
        r = torch.abs(f[:, :, None] - d)                     # distances to the support cells
        near = (3.0 - 2.0 * r + torch.sqrt(torch.clamp(1.0 + 4.0 * r - 4.0 * r * r, min=0.0))) / 8.0
        far = (5.0 - 2.0 * r - torch.sqrt(torch.clamp(-7.0 + 12.0 * r - 4.0 * r * r, min=0.0))) / 8.0
        w = torch.where(r <= 1.0, near, far)
        c = base.long()[:, :, None] + d
        X, Y, Z = c[:, 0] % self.nx, c[:, 1] % self.ny, c[:, 2] - self.walls
        if not self.walls:
            Z = Z % self.nz
        cell = X[:, None, None, :] + self.nx * (Y[:, None, :, None] + self.ny * Z[:, :, None, None])
        wt = w[:, 0][:, None, None, :] * w[:, 1][:, None, :, None] * w[:, 2][:, :, None, None]
        ok = ((Z >= 0) & (Z < self.nz))[:, :, None, None].expand_as(cell)
        return torch.where(ok, cell, 0).reshape(-1), torch.where(ok, wt, 0.0).reshape(-1)

    def inside(self):
        """Cells with an odd number of surface crossings below them on their vertical line."""
        v = [self.q[self.tri[:, k]] for k in range(3)]
        lo = torch.ceil(torch.minimum(torch.minimum(v[0], v[1]), v[2])[:, :2])
        hi = torch.floor(torch.maximum(torch.maximum(v[0], v[1]), v[2])[:, :2])
        span = (hi - lo).max(0).values.long().tolist()
        flips = torch.zeros((self.nz + 1, self.ny, self.nx), dtype=torch.int32, device=self.dev).reshape(-1)

        def edge(a, b, px, py):
            return (b[:, 0] - a[:, 0]) * (py - a[:, 1]) - (b[:, 1] - a[:, 1]) * (px - a[:, 0])
        for dx in range(span[0] + 1):
            for dy in range(span[1] + 1):
                px, py = lo[:, 0] + dx, lo[:, 1] + dy
                e0, e1, e2 = edge(v[1], v[2], px, py), edge(v[2], v[0], px, py), edge(v[0], v[1], px, py)
                hit = ((e0 > 0) & (e1 > 0) & (e2 > 0)) | ((e0 < 0) & (e1 < 0) & (e2 < 0))
                hit &= (px <= hi[:, 0]) & (py <= hi[:, 1])
                e0, e1, e2, px, py = e0[hit], e1[hit], e2[hit], px[hit], py[hit]
                z = (e0 * v[0][hit, 2] + e1 * v[1][hit, 2] + e2 * v[2][hit, 2]) / (e0 + e1 + e2)
                first = torch.clamp(torch.floor(z).long() + 1 - self.walls, 0, self.nz)
                at = px.long() % self.nx + self.nx * (py.long() % self.ny + self.ny * first)
                flips.index_add_(0, at, torch.ones_like(at, dtype=torch.int32))
        odd = torch.cumsum(flips.reshape(self.nz + 1, self.ny, self.nx)[:-1], 0) % 2
        return odd == 1

    def pulled(self, i):
        """Population i after streaming, halfway bounce-back at the walls."""
        cx, cy, cz = (int(k) for k in _C[i])
        if not (self.walls and cz):
            return torch.roll(self.s[i], (cz, cy, cx), (0, 1, 2))
        out = torch.empty_like(self.s[i])
        moved = torch.roll(self.s[i], (cy, cx), (1, 2)) if cx or cy else self.s[i]
        if cz > 0:
            out[1:], out[0] = moved[:-1], self.s[_OPP[i]][0]
        else:
            out[:-1], out[-1] = moved[1:], self.s[_OPP[i]][-1]
        return out

    def step(self):
        p = self.p
        cells = self.nx * self.ny * self.nz
        cell, wt = self.stencil()
        phi = self.node_forces()
        F = torch.empty((3, cells), dtype=torch.float64, device=self.dev)
        for k in range(3):
            F[k] = torch.bincount(cell, weights=wt * phi[:, k].repeat_interleave(64), minlength=cells)
        F = F.reshape(3, self.nz, self.ny, self.nx)
        tau = p["tau"]
        if p["lam"] != 1.0:
            tau = p["tau"] + (p["lam"] - 1.0) * (p["tau"] - 0.5) * self.inside().double()
        new = torch.stack([self.pulled(i) for i in range(19)])
        drho = new.sum(0)
        rho = 1.0 + drho
        u = [0.5 * F[k] for k in range(3)]
        for i in range(1, 19):
            for k in range(3):
                if _C[i, k]:
                    u[k] = u[k] + float(_C[i, k]) * new[i]
        u = [a / rho for a in u]
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        src = 1.0 - 0.5 / tau
        for i in range(19):
            cu, cF = torch.zeros_like(rho), torch.zeros_like(rho)
            for k in range(3):
                if _C[i, k]:
                    cu = cu + float(_C[i, k]) * u[k]
                    cF = cF + float(_C[i, k]) * F[k]
            eq = _WT[i] * (drho + rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu))
            new[i] += (eq - new[i]) / tau + src * _WT[i] * (3.0 * (cF - uF) + 9.0 * cu * cF)
        self.s, self.rho, self.u = new, rho, torch.stack(u)
        flat = self.u.reshape(3, -1)
        self.q = self.q + torch.stack([(flat[k][cell] * wt).reshape(-1, 64).sum(1) for k in range(3)], 1)
        if p["volcorr"]:
            c = self.q.mean(0)
            self.q = c + (self.q - c) * (self.V0 / self.volume(self.q)) ** (1.0 / 3.0)

    def observe(self):
        q, tri, R0 = self.q, self.tri, self.R0
        v = [q[tri[:, k]] for k in range(3)]
        area = 0.5 * _norm(torch.linalg.cross(v[1] - v[0], v[2] - v[0]))
        V, z = float(self.volume(q)), q[:, 2]
        zmin, zmax = float(z.min()), float(z.max())
        ell, RV = 0.5 * (zmax - zmin), (3.0 * V / (4.0 * math.pi)) ** (1.0 / 3.0)

        def angle(R):
            return 180.0 if ell >= R else math.degrees(2.0 * math.atan(math.sqrt(3.0 * ell ** 3 / (R ** 3 - ell ** 3))))
        zp = 0.5 + ZCUT * R0
        a = torch.cat([tri[:, 0], tri[:, 1], tri[:, 2]])
        b = torch.cat([tri[:, 1], tri[:, 2], tri[:, 0]])
        cut = (a < b) & ((z[a] < zp) != (z[b] < zp))
        a, b = a[cut], b[cut]
        pts = (q[a] + ((zp - z[a]) / (z[b] - z[a]))[:, None] * (q[b] - q[a]))[:, :2]
        zz = torch.stack([w[:, 2] for w in v])
        flat = (zz.mean(0) < 0.5 * (zmin + zmax)) & (zz.max(0).values - zz.min(0).values < EPS_FLAT * R0)
        chi = float(area[flat].sum())
        c = q.mean(0).tolist()
        return {"mass": float((1.0 + self.s.sum(0)).sum()), "volume": V, "area": float(area.sum()), "zmin": zmin,
                "zmax": zmax, "theta_R0_deg": angle(R0), "theta_RV_deg": angle(RV),
                "rc_cut": float(_norm(pts - pts.mean(0)).mean()) if len(pts) else 0.0,
                "rc_flat": math.sqrt(chi / math.pi), "n_cut": float(len(pts)), "chi_flat": chi,
                "status": None, "clamped": None, "cx": c[0], "cy": c[1], "cz": c[2]}


def _features(x):
    return np.stack([(x[:, 0] - 90.0) / 70.0, (x[:, 1] - 16.0) / 8.0, np.log10(x[:, 2])], 1)


def _layers(params):
    out, at = [], 0
    for i, o in ((3, 256), (256, 256), (256, 256), (256, 64)):
        out.append([params[at:at + i * o].reshape(o, i), params[at + i * o:at + i * o + o]])
        at += i * o + o
    return out


def _exact_network(case, seed):
    x, y = _network_data(case, seed)
    if case["kind"] == "predict":
        h = _features(x)
        layers = _layers(W.load_params().astype(np.float64))
        for k, (w, b) in enumerate(layers):
            h = h @ w.T + b
            h = np.tanh(h) if k < 3 else h
        return h
    params = torch.from_numpy(I.mlp_init(seed).astype(np.float64))
    m, v = torch.zeros_like(params), torch.zeros_like(params)
    x, y = torch.from_numpy(_features(x)), torch.from_numpy(y)
    perm, state, t, losses = list(range(len(x))), 0, 0, []
    mask = (1 << 64) - 1
    for _ in range(case["epochs"]):
        for i in range(len(x) - 1, 0, -1):        # Fisher-Yates from a splitmix64 stream
            state = (state + 0x9E3779B97F4A7C15) & mask
            r = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
            r = ((r ^ (r >> 27)) * 0x94D049BB133111EB) & mask
            j = (r ^ (r >> 31)) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        total, nb = 0.0, len(x) // case["batch"]
        for b in range(nb):
            idx = perm[b * case["batch"]:(b + 1) * case["batch"]]
            p = params.clone().requires_grad_(True)
            h = x[idx]
            for k, (w, c) in enumerate(_layers(p)):
                h = h @ w.T + c
                h = torch.tanh(h) if k < 3 else h
            loss = ((h - y[idx]) ** 2).mean()
            loss.backward()
            total += float(loss)
            t += 1
            m = 0.9 * m + 0.1 * p.grad
            v = 0.999 * v + 0.001 * p.grad ** 2
            params = params - 1e-3 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
        losses.append(total / nb)
    return {"losses": np.array(losses), "params": params.numpy()}


def exact(case, seed):
    if case["kind"] in ("train", "predict"):
        return _exact_network(case, seed)
    device = "cuda" if torch.cuda.is_available() else "cpu"
    rng = np.random.default_rng(seed)
    obs, nodes = [], []
    for spec in _specs(case):
        e = _Exact(spec, _mesh(spec, rng), device)
        for _ in range(spec["steps"]):
            e.step()
        obs.append(e.observe())
        nodes.append(e.q.cpu().numpy())
    if len(obs) > 1:
        return {"obs": {k: None if obs[0][k] is None else np.array([o[k] for o in obs]) for k in obs[0]},
                "nodes": np.concatenate(nodes)}
    out = {"obs": obs[0], "nodes": nodes[0]}
    if case["fields"]:
        out["rho"], out["u"] = e.rho.reshape(-1).cpu().numpy(), e.u.reshape(-1).cpu().numpy()
    return out
