"""What the framework is timed on: the particle step in the forms that programs call it (small and
large ensembles, one to four scalars, batches of ensembles, curved walls, IECM, both precisions of
the moment sums, caller-owned buffers), the gridpoint solve, the coupled loop, and the learned
surrogate (its fields, its gradient and its training).

Ensembles are advanced from where the pass before left them, as a time loop does: a state holds the
context, the node fields and the step number. Meshes are built once per size and kept, as a program
keeps its grid. `exact` is the same computation in 64 bits with plain torch: the method's equations,
a neighbour walk, the P1 finite elements with a CG, the network with autograd.
"""
import functools
import math

import numpy as np
import torch

from paper_1006_0549_gb300 import lpdf
from paper_1006_0549_gb300 import workloads as wl

DT = 1e-3
NU = {"channel": 1.0 / 180.0, "bump": 1.0 / 180.0, "cavity": 1e-4}
LID = {"channel": 0.0, "bump": 0.0, "cavity": 1.0}
MESH_SEED = 1006054902


def _steps(name, mesh, nx, ny, ppe, ns, steps, each=True, sums=0, adv=-1, mom=-1):
    return {"name": name, "kind": "steps", "mesh": mesh, "nx": nx, "ny": ny, "ppe": ppe, "ns": ns, "steps": steps,
            "each": each, "sums": sums, "adv": adv, "mom": mom}


def listed():
    return [
        # the 1,000-triangle channel of the coupled runs, ten steps with the statistics of each:
        # small ensembles, where launches and latency count; never tuned, as in the time loop
        _steps("steps-channel-50k", "channel", 25, 20, 50, 1, 10),
        # the production channel (50,000 triangles, 25M particles): the configuration that a
        # throughput run holds, with the launch variants that the tuner picks for it
        _steps("steps-channel-25m", "channel", 250, 100, 500, 1, 4, adv=5, mom=1),
        # the lid-driven cavity with four scalars: many thin elements, few particles in each, long walks
        _steps("steps-cavity-20m", "cavity", 316, 316, 100, 4, 4, adv=1, mom=1),
        # a channel of odd sizes with compensated moment sums (statistics to 1e-9), never tuned
        _steps("steps-compensated-3m", "channel", 131, 53, 217, 1, 4, sums=1),
        # walls of any shape: the channel with a bump on its bottom wall, mirrored inside the walk
        _steps("steps-walls-7m", "bump", 180, 71, 288, 1, 4, adv=5, mom=1),
        # IECM micromixing with a reaction: fluxes and slopes from the statistics after every step
        {"name": "mixing-5m", "kind": "mixing", "mesh": "channel", "nx": 250, "ny": 100, "ppe": 100, "ns": 3, "steps": 2},
        # a batch of independent channels of uneven size in one multi-component mesh, by CUDA graphs
        {"name": "batched-16", "kind": "batched", "mesh": "channel", "count": 16, "tri_lo": 2000, "tri_hi": 12000,
         "ppe_lo": 50, "ppe_hi": 400, "ns": 1, "steps": 4},
        # one step on the buffers of a host code that owns all device memory
        {"name": "static-1m", "kind": "static", "mesh": "channel", "nx": 100, "ny": 41, "ppe": 125, "ns": 1},
        # the whole method on the small channel: step, statistics, relaxation and pressure solve for
        # the next step's fields, the CGs starting from the previous solution
        {"name": "coupled-50k", "kind": "coupled", "mesh": "channel", "nx": 25, "ny": 20, "ppe": 50, "ns": 1},
        # the gridpoint solve of the production channel from cold: 25,000 unknowns, both CGs
        {"name": "solve-25k-nodes", "kind": "solve", "mesh": "channel", "nx": 250, "ny": 100, "ns": 1},
        # node fields of the cavity's 100,489 nodes from the trained network instead of the solve
        {"name": "surrogate-100k-nodes", "kind": "surrogate", "mesh": "cavity", "nx": 316, "ny": 316, "ns": 4},
        # training the network: 50 Adam steps on minibatches of 1024 rows
        {"name": "train-1024", "kind": "train", "rows": 25600, "batch": 1024, "steps": 50},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "mixing", "batched", "static", "coupled", "solve", "surrogate",
                       "train", "gradient"])
    if kind == "train":
        b = _log(rng, 100, 4096)
        return {"kind": kind, "rows": b * rng.randint(2, 20) + rng.randint(0, b - 1), "batch": b,
                "steps": rng.randint(20, 80)}
    if kind == "gradient":
        return {"kind": kind, "batch": _log(rng, 1, 20000)}
    mesh = rng.choice(["channel", "cavity", "bump"] if kind == "steps" else ["channel", "cavity"]
                      if kind in ("solve", "surrogate", "static") else ["channel"])
    tri = _log(rng, 500, 2000 if kind == "coupled" else 10000 if kind == "batched" else 60000)
    ny = max(6, int(math.sqrt(tri / 5.0)) + rng.randint(-2, 3))
    nx = max(6, tri // (2 * ny) + rng.randint(-1, 1))
    case = {"kind": kind, "mesh": mesh, "nx": nx, "ny": ny, "ns": rng.randint(1, 4)}
    if kind == "solve" and mesh == "cavity":
        case.update(nx=min(nx, 60), ny=min(ny, 60))
    steps = rng.randint(1, 6)
    ppe = min(_log(rng, 20, 500), max(20, 40_000_000 // (2 * nx * ny * steps)))
    if kind == "steps":
        case.update(ppe=ppe, steps=steps, each=rng.random() < 0.7, sums=int(rng.random() < 0.25))
        case.update(zip(("adv", "mom"), rng.choice([(-1, -1), (5, 1), (4, 1), (1, 1)])))
    elif kind == "mixing":
        case.update(ppe=ppe, ns=3, steps=min(steps, 4))
    elif kind == "batched":
        lo = rng.randint(20, 100)
        case = {"kind": kind, "mesh": "channel", "count": rng.randint(2, 16), "tri_lo": max(500, tri // 3),
                "tri_hi": tri + 500, "ppe_lo": lo, "ppe_hi": lo + rng.randint(1, 200), "ns": rng.randint(1, 2),
                "steps": rng.randint(1, 4)}
    elif kind == "static":
        case.update(ppe=min(ppe, 200))
    elif kind == "coupled":
        case.update(ppe=rng.randint(50, 200), ns=rng.randint(1, 2))
    return case


# ------------------------------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=None)
def _host_mesh(kind, nx, ny):
    if kind == "cavity":
        return wl.cavity_mesh(nx, ny, MESH_SEED)
    return (wl.channel_mesh if kind == "channel" else wl.bump_channel_mesh)(nx, ny, MESH_SEED)


@functools.lru_cache(maxsize=None)
def _mesh(kind, nx, ny):
    return lpdf.Mesh(_host_mesh(kind, nx, ny))


@functools.lru_cache(maxsize=None)
def _base_fields(kind, nx, ny, ns):
    return wl.synthetic_node_fields(_host_mesh(kind, nx, ny), ns, seed=5)


@functools.lru_cache(maxsize=None)
def _batch(count, tri_lo, tri_hi, ppe_lo, ppe_hi):
    wk = wl.batched_channels(count, (tri_lo, tri_hi), (ppe_lo, ppe_hi))
    fields = [wl.synthetic_node_fields(m, 1, seed=5 + k) for k, m in enumerate(wk.mesh.parts)]
    return wk, lpdf.Mesh(wk.mesh), fields


def _fields(base, ns, seed):
    """Node fields of the seed: the synthetic ones of the mesh, every column scaled by up to 5 %."""
    f = np.zeros((base.shape[0], wl.n_fields_padded(ns)), dtype=np.float32)
    f[:, :22] = base[:, :22]
    f[:, 22:22 + ns] = base[:, 22:23]
    f *= (1.0 + 0.05 * np.random.default_rng(seed).uniform(-1.0, 1.0, f.shape[1])).astype(np.float32)
    return torch.from_numpy(f).cuda()


def _particles(mesh, ppe, ns, seed):
    """A seeded ensemble in element order: positions inside the elements, Gaussian velocities about
    the mean profile, gamma-distributed frequencies, scalars between 0 and 1 (device tensors)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    V = torch.from_numpy(mesh.node_xy[mesh.tri]).cuda()                       # (E, 3, 2)
    n = mesh.n_tri * ppe
    elem = torch.arange(mesh.n_tri, device="cuda", dtype=torch.int32).repeat_interleave(ppe)
    r = torch.rand((n, 3), generator=g, device="cuda", dtype=torch.float64).clamp_min_(1e-9).log_().neg_()
    r = 0.97 * r / r.sum(1, keepdim=True) + 0.01
    xy = torch.zeros((n, 2), dtype=torch.float64, device="cuda")
    for k in range(3):
        xy += r[:, k:k + 1] * V[:, k].repeat_interleave(ppe, 0)
    out = {"x": xy[:, 0].float(), "y": xy[:, 1].float()}
    yw = torch.minimum(xy[:, 1], 2.0 - xy[:, 1]).clamp_min(0.0)
    del r, xy
    sigma, U, om = 0.1, 0.0, 1.0
    if mesh.kind == "channel":
        yp = 180.0 * yw
        sigma, U = 1.0, torch.where(yp < 11.0, yp, yp.clamp_min(1.0).log() / 0.41 + 5.2)
        om = 1.0 / (0.123 * yw.clamp_min(10.0 / 180.0))
    for k in ("u", "v", "w"):
        out[k] = (sigma * torch.randn(n, generator=g, device="cuda") + (U if k == "u" else 0.0)).float()
    e = torch.zeros(n, device="cuda")
    for _ in range(4):
        e -= torch.rand(n, generator=g, device="cuda").clamp_min_(1e-7).log_()
    out["omega"] = (0.25 * e * om).float()
    out["psi"] = torch.rand((ns, n), generator=g, device="cuda")
    out["elem"] = elem
    out["pid"] = torch.arange(n, device="cuda", dtype=torch.int32)
    return out


def _sources(case):
    ns = case["ns"]
    if case["mesh"] == "cavity":
        xy = [(0.25, 0.25), (0.75, 0.25), (0.5, 0.5), (0.5, 0.8)]
        return [(x, y, 0.01, a) for a, (x, y) in enumerate(xy[:ns])]
    return [(0.25, 0.67 + 0.22 * a, 0.02, a) for a in range(2 if case["kind"] == "mixing" else ns)]


def _params(case, seed, **more):
    mesh = case["mesh"]
    if case["kind"] == "mixing":
        more = dict(mixing=1, react_k=4.0, react_a=0, react_b=1, react_p=2)
    if case["kind"] == "coupled":
        more = dict(gmodel=0, pressure_solve=1, dpdx0=-1.0, cg_warm_start=1)
    if case["kind"] == "solve":
        more = dict(gmodel=0, pressure_solve=1, dpdx0=0.0 if mesh == "cavity" else -1.0)
    src = _sources(case) if case["kind"] not in ("solve", "surrogate") else []
    return lpdf.make_params(nu=NU[mesh], dt=DT, seed=seed, ns=case["ns"], lid_u=LID[mesh], sources=src, **more)


def _batch_components(case, wk, seed):
    keys = [1000003 * seed + k for k in range(case["count"])]
    return [(key, [(s[0][0], s[0][1], s[0][2], a) for a in range(case["ns"])]) for key, s in zip(keys, wk.sources)]


def _batch_key(case):
    return tuple(case[k] for k in ("count", "tri_lo", "tri_hi", "ppe_lo", "ppe_hi"))


def _statistics(case, seed):
    return wl.synthetic_statistics(_host_mesh(case["mesh"], case["nx"], case["ny"]), case["ns"], seed)


def _network(seed):
    rng = np.random.default_rng(seed)
    p = wl.mlp_init_params(seed)
    at = 0
    for fi, fo in ((8, 128), (128, 128), (128, 128), (128, 7)):       # biases that are not zero
        p[at + fi * fo:at + fi * fo + fo] = 0.1 * rng.standard_normal(fo)
        at += fi * fo + fo
    return p


def _norm(feat, tgt):
    one = np.ones(7)
    return np.concatenate([feat.mean(0), feat.std(0), one, tgt.mean(0), tgt.std(0)]).astype(np.float32)


def _surrogate_net(case, seed):
    """The network and the standardisation that a training on such statistics ends with: inputs of
    these nodes, targets of the size that the simplified Langevin model gives."""
    feat = _features64(case, torch.from_numpy(_statistics(case, seed)).cuda()).cpu().numpy()
    return _network(seed), _norm(feat, np.array([[-2.6, -0.5, -0.5, -2.6, -2.6, 1.6, 0.7], [-1.5, 0.5, 0.5, -1.5, -1.5, 2.6, 1.3]]))


def _rows(case, seed):
    return wl.mlp_random_data(case.get("rows", case["batch"]), seed)


def _train_norm(case, seed):
    feat, tgt = wl.mlp_random_data(4096, seed)
    return _norm(feat, tgt)


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if kind in ("train", "gradient"):
        feat, tgt = _rows(case, seed)
        s.update(feat=torch.from_numpy(feat).cuda(), tgt=torch.from_numpy(tgt).cuda(), net=lpdf.MLP(case["batch"]))
        s["net"].set_params(_network(seed), _train_norm(case, seed))
        return s
    ns = case["ns"]
    if kind == "batched":
        wk, mesh, base = _batch(*_batch_key(case))
        parts = [_particles(m, ppe, ns, 31 * seed + k) for k, (m, ppe) in enumerate(zip(wk.mesh.parts, wk.n_per_elem))]
        for p, off in zip(parts, wk.mesh.tri_off):
            p["elem"] += int(off)
        state = {k: torch.cat([p[k] for p in parts], dim=-1) for k in parts[0]}
        s["F"] = torch.cat([_fields(f, ns, seed + k) for k, f in enumerate(base)])
        params = lpdf.make_params(nu=wk.nu, dt=wk.dt, seed=seed, ns=ns)
    else:
        key = (case["mesh"], case["nx"], case["ny"])
        # the solves of a coupled run start from the solution that its own mesh holds
        mesh = lpdf.Mesh(_host_mesh(*key)) if kind == "coupled" else _mesh(*key)
        params = _params(case, seed, moment_sums=case.get("sums", 0))
        if kind in ("solve", "surrogate"):
            s.update(mesh=mesh, params=params, S=torch.from_numpy(_statistics(case, seed)).cuda(),
                     F=torch.zeros((mesh.n_nodes, wl.n_fields_padded(ns)), device="cuda"))
            if kind == "surrogate":
                s["net"] = lpdf.MLP(1024)
                s["net"].set_params(*_surrogate_net(case, seed))
                s["net"].set_policy(check_every=1 << 30, threshold=1e30)
                mesh.surrogate_relax_solve(s["net"], params, s["S"], s["F"], 1e-6)   # the checking call
            return s
        state = _particles(_host_mesh(*key), case["ppe"], ns, seed)
        s["F"] = _fields(_base_fields(*key, 1), ns, seed)
    s.update(mesh=mesh, params=params, step=1,
             S=torch.zeros((mesh.n_nodes, 11 + 2 * ns), dtype=torch.float64, device="cuda"))
    if kind == "static":
        s["state"] = state
        return s
    ctx = s["ctx"] = lpdf.Context(mesh, params, int(state["x"].shape[0]))
    if kind == "batched":
        ctx.set_components(_batch_components(case, wk, seed))
        ctx.set_tune(5, 1)
    if case.get("adv", -1) >= 0:
        ctx.set_tune(case["adv"], case["mom"])
    if kind == "mixing":
        s["flux"] = torch.zeros((mesh.n_nodes, 3 * ns), dtype=torch.float64, device="cuda")
        s["beta"] = torch.zeros((mesh.n_nodes, 3 * ns), dtype=torch.float32, device="cuda")
        ctx.set_iecm(s["beta"])
    ctx.set_state(state)
    torch.cuda.synchronize()
    return s


# --------------------------------------------------------------------------------------------- run

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "train":
        losses = s["net"].train(s["feat"], s["tgt"], case["batch"], case["steps"], 1e-3)
        return {"losses": losses, "params": s["net"].get_params()[0]}
    if kind == "gradient":
        g, loss = s["net"].gradient(s["feat"], s["tgt"])
        return {"grad": g, "loss": loss}
    if kind == "solve":
        s["mesh"].elliptic_relax_solve(s["params"], s["S"], s["F"], 1e-8)
        return {"fields": s["F"]}
    if kind == "surrogate":
        s["mesh"].surrogate_relax_solve(s["net"], s["params"], s["S"], s["F"], 1e-8)
        return {"fields": s["F"]}
    if kind == "static":
        lpdf.pdf_step_static(s["mesh"], s["params"], s["state"], s["F"], s["step"], s["S"], read_status=False)
        s["step"] += 1
        return {"stats": s["S"], **s["state"]}
    ctx, out = s["ctx"], {}
    if kind == "coupled":
        ctx.pdf_step(s["F"], s["step"])
        ctx.grid_statistics(s["S"])
        s["mesh"].elliptic_relax_solve(s["params"], s["S"], s["F"], 1e-8)
        s["step"] += 1
        return {"stats": s["S"], "fields": s["F"], **ctx.get_state()}
    n = case["steps"]
    if kind == "batched" or (kind == "steps" and not case["each"]):
        ctx.pdf_steps(s["F"], s["step"], n)
        ctx.grid_statistics(s["S"])
    else:
        for k in range(n):
            ctx.pdf_step(s["F"], s["step"] + k)
            ctx.grid_statistics(s["S"])
            if kind == "mixing":
                ctx.grid_flux_statistics(s["flux"])
                s["mesh"].iecm_coefficients(case["ns"], s["S"], s["flux"], s["beta"])
                out = {"flux": s["flux"], "beta": s["beta"]}
    s["step"] += n
    # the snapshot that a run of n steps ends with
    return {"stats": s["S"], **out, **ctx.get_state()}


def work(case):
    kind = case["kind"]
    if kind in ("train", "gradient"):
        b, steps = case["batch"], case.get("steps", 1)
        return {"bytes": steps * b * 60.0 + 2 * 4 * lpdf.MLP_NPARAMS, "flops": steps * 6.0 * b * lpdf.MLP_NPARAMS}
    ns = case["ns"]
    if kind == "batched":
        wk = _batch(*_batch_key(case))[0]
        nodes, tri, n = wk.mesh.n_nodes, wk.mesh.n_tri, wk.n_particles
    else:
        nodes, tri = (case["nx"] + 1) * (case["ny"] + 1), 2 * case["nx"] * case["ny"]
        n = tri * case.get("ppe", 0)
    grid = nodes * (8.0 * (11 + 2 * ns) + 4.0 * wl.n_fields_padded(ns))      # statistics and node fields
    if kind == "solve":
        return {"bytes": grid + tri * 150.0, "flops": tri * 2000.0}
    if kind == "surrogate":
        return {"bytes": grid + tri * 100.0, "flops": nodes * 2.0 * lpdf.MLP_NPARAMS + tri * 200.0}
    steps = case.get("steps", 1)
    snapshot = 0.0 if kind == "static" else n * 4.0 * (8 + ns)
    # a step reads x, y, u, v, w, omega, psi, elem, pid and writes all but pid
    return {"bytes": steps * (n * 4.0 * (15 + 2 * ns) + grid) + snapshot, "flops": steps * n * (500.0 + 100.0 * ns)}


# ------------------------------------------------------------------------------------------- exact
# The same results in 64 bits with plain torch.

class _Geometry:
    """Elements, shape-function gradients, neighbours and periodic pairing of a mesh."""

    def __init__(self, mesh):
        self.box, self.period, dev = mesh.box, mesh.period_x, "cuda"
        xy, tri, tag = mesh.node_xy, mesh.tri.astype(np.int64), mesh.edge_tag
        master = np.arange(len(xy))
        if self.period > 0:
            left = {y: i for i, (x, y) in enumerate(xy) if x == mesh.box[0]}
            for i in np.nonzero(xy[:, 0] == mesh.box[1])[0]:
                master[i] = left[xy[i, 1]]
        a, b = master[tri], master[np.roll(tri, -1, axis=1)]                  # edge k: vertex k -> k + 1
        N = len(xy)
        fwd, back = (a * N + b).ravel(), (b * N + a).ravel()
        order = np.argsort(fwd)
        at = np.searchsorted(fwd[order], back).clip(max=len(fwd) - 1)
        hit = fwd[order][at] == back
        nbr = np.where(hit, order[at] // 3, -1).reshape(-1, 3)
        nbr[(tag == wl.EDGE_WALL) | (tag == wl.EDGE_MOVING_WALL)] = -1
        wall = nbr < 0
        ends = xy[tri], xy[np.roll(tri, -1, axis=1)]
        sides = [(ends[0][..., d] == ends[1][..., d]) & ((ends[0][..., d] == lo) | (ends[0][..., d] == hi))
                 for d, lo, hi in ((0, *mesh.box[:2]), (1, *mesh.box[2:]))]
        self.edge_walls = bool((wall & ~sides[0] & ~sides[1]).any())
        self.moving = torch.from_numpy(tag == wl.EDGE_MOVING_WALL).to(dev)
        self.xy, self.tri = torch.from_numpy(xy).to(dev), torch.from_numpy(tri).to(dev)
        self.nbr, self.master = torch.from_numpy(nbr).to(dev), torch.from_numpy(master).to(dev)
        p = self.xy[self.tri]                                                 # (E, 3, 2)
        q, r = p.roll(-1, 1), p.roll(-2, 1)
        det = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - (p[:, 1, 1] - p[:, 0, 1]) * (p[:, 2, 0] - p[:, 0, 0])
        self.area, self.cx = 0.5 * det, p[:, :, 0].mean(1)
        self.grad = torch.stack([q[..., 1] - r[..., 1], r[..., 0] - q[..., 0]], -1) / det[:, None, None]
        self.wall_k = [(e, k) for e, k in zip(*np.nonzero(wall))]
        self.p = p

    def weights(self, e, x, y):
        """Barycentric weights (n, 3) of (x, y) in e, the nearest periodic image of the point."""
        if self.period > 0:
            d = self.cx[e] - x
            x = torch.where(d.abs() > 0.5 * self.period, x + torch.sign(d) * self.period, x)
        g, p = self.grad[e], self.p[e]
        l1 = g[:, 1, 0] * (x - p[:, 0, 0]) + g[:, 1, 1] * (y - p[:, 0, 1])
        l2 = g[:, 2, 0] * (x - p[:, 0, 0]) + g[:, 2, 1] * (y - p[:, 0, 1])
        return torch.stack([1.0 - l1 - l2, l1, l2], 1)

    def locate(self, e, z, lid):
        """The owners of the positions in z, walking from e; walls of any shape mirror on the way."""
        e = e.clone()
        live = torch.arange(len(e), device=e.device)
        for _ in range(72):
            lam = self.weights(e[live], z["x"][live], z["y"][live])
            nb = self.nbr[e[live]][:, [1, 2, 0]]                               # across the edge opposite vertex a
            inner = torch.where(nb >= 0, lam, torch.full_like(lam, 1e9))
            lo, a = inner.min(1)
            go = lo < -1e-13
            e[live[go]] = nb[go, a[go]]
            stuck = ~go & (lam.amin(1) < -1e-13)
            if self.edge_walls and stuck.any():
                i, k = live[stuck], (lam[stuck].argmin(1) + 1) % 3
                s, t = self.p[e[i], k], self.p[e[i], (k + 1) % 3]
                d, q = t - s, torch.stack([z["x"][i], z["y"][i]], 1)
                f = s + ((q - s) * d).sum(1, keepdim=True) / (d * d).sum(1, keepdim=True) * d
                m = 2 * f - q
                m[:, 0] -= self.period * torch.floor((m[:, 0] - self.box[0]) / self.period) if self.period > 0 else 0.0
                z["x"][i], z["y"][i] = m[:, 0], m[:, 1]
                z["u"][i] = torch.where(self.moving[e[i], k], 2 * lid, 0.0) - z["u"][i]
                z["v"][i], z["w"][i] = -z["v"][i], -z["w"][i]
                go = go | stuck
            live = live[go]
            if not len(live):
                break
        return e


def _philox(c, key):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    def mul(a, b):
        p0, p1 = a * (b & 0xFFFF), a * (b >> 16)
        t = p1 + (p0 >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (p0 & 0xFFFF)

    k0, k1 = key & 0xFFFFFFFF, key >> 32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _normals(pid, step, key):
    z = torch.zeros_like(pid)
    w = []
    for block in (0, 1):
        w += _philox([pid, z + (step & 0xFFFFFFFF), z + (step >> 32), z + block], key)
    out = []
    for a, b in ((0, 1), (2, 3), (4, 5)):
        r = torch.sqrt(-2.0 * torch.log((w[a] + 0.5) * 2.0 ** -32))
        t = 2.0 * math.pi * (w[b] + 0.5) * 2.0 ** -32
        out += [r * torch.cos(t), r * torch.sin(t)]
    return out


def _step64(geo, z, F, step, key, case, sources, beta):
    """One step of the particles z (x, y, u, v, w, omega, psi, elem, pid in 64 bits), in place."""
    x0, x1, y0, y1 = geo.box
    nu, lid = NU[case["mesh"]], LID[case["mesh"]]
    dt, sdt, s2nu = float(np.float32(DT)), math.sqrt(DT), math.sqrt(2.0 * nu)
    z1, z2, z3, z4, z5, z6 = (sdt * v for v in _normals(z["pid"], step, key))
    e, x, y, u, v, w, om = (z[k].clone() for k in ("elem", "x", "y", "u", "v", "w", "omega"))
    lam = geo.weights(e, x, y)
    corner = geo.tri[e]
    at = lambda T, c: (lam * T[corner, c]).sum(1)                             # noqa: E731
    Ur, Vr, Wr = u - at(F, 0), v - at(F, 1), w - at(F, 2)
    c0 = at(F, 19).clamp_min(0.0).sqrt()
    z["u"] = u + (-at(F, 12) + 2 * nu * at(F, 9) + at(F, 14) * Ur + at(F, 15) * Vr) * dt \
        + s2nu * (at(F, 3) * z1 + at(F, 4) * z2) + c0 * z3
    z["v"] = v + (-at(F, 13) + 2 * nu * at(F, 10) + at(F, 16) * Ur + at(F, 17) * Vr) * dt \
        + s2nu * (at(F, 5) * z1 + at(F, 6) * z2) + c0 * z4
    z["w"] = w + (2 * nu * at(F, 11) + at(F, 18) * Wr) * dt + s2nu * (at(F, 7) * z1 + at(F, 8) * z2) + c0 * z5
    Om = at(F, 20)
    z["omega"] = (om - 5.0 * Om * (om - Om) * dt - at(F, 21) * Om * om * dt
                  + (2.5 * Om * Om * om.clamp_min(0.0)).sqrt() * z6).abs()     # C3 = 5, C4 = 1/4
    psi, ns = z["psi"], case["ns"]
    rate = 4.0 * psi[0] * psi[1] if beta is not None else 0.0
    new = []
    for a in range(ns):
        cond = at(F, 22 + a)
        src = 0.0
        if beta is not None:
            cond = cond + sum(at(beta, 3 * a + c) * d for c, d in enumerate((Ur, Vr, Wr)))
            src = rate if a == 2 else -rate
        new.append(psi[a] - (psi[a] - cond) * Om * dt + src * dt)              # C_phi = 2
    z["psi"] = torch.stack(new)
    z["x"], z["y"] = x + u * dt + s2nu * z1, y + v * dt + s2nu * z2
    if geo.period > 0:
        z["x"] = z["x"] - geo.period * torch.floor((z["x"] - x0) / geo.period)
    if not geo.edge_walls:
        for _ in range(8):
            for c, lo, hi, on in (("y", y0, y1, True), ("x", x0, x1, geo.period == 0)):
                if on:
                    low, high = z[c] < lo, z[c] > hi
                    z[c] = torch.where(low, 2 * lo - z[c], torch.where(high, 2 * hi - z[c], z[c]))
                    moving = lid if c == "y" else 0.0
                    z["u"] = torch.where(low, -z["u"], torch.where(high, 2 * moving - z["u"], z["u"]))
                    for q in ("v", "w"):
                        z[q] = torch.where(low | high, -z[q], z[q])
    z["elem"] = geo.locate(e, z, lid)
    for sx, sy, sr, a in sources:
        sx, sy, sr = (float(np.float32(t)) for t in (sx, sy, sr))
        z["psi"][a] = torch.where((z["x"] - sx) ** 2 + (z["y"] - sy) ** 2 < sr * sr, 1.0, z["psi"][a])


def _sums64(geo, z, quantities):
    lam = geo.weights(z["elem"], z["x"], z["y"])
    node = geo.master[geo.tri[z["elem"]]]
    out = torch.zeros((len(geo.xy), len(quantities)), dtype=torch.float64, device="cuda")
    for c, q in enumerate(quantities):
        for a in range(3):
            out[:, c].index_add_(0, node[:, a], lam[:, a] * q)
    return out[geo.master]


def _stats64(geo, z, raw=False):
    u, v, w, psi = z["u"], z["v"], z["w"], z["psi"]
    S = _sums64(geo, z, [torch.ones_like(u), u, v, w, u * u, u * v, u * w, v * v, v * w, w * w, z["omega"], *psi,
                         *(psi * psi)])
    if raw:
        return S
    some = S[:, :1] > 0
    m = torch.where(some, S / torch.where(some, S[:, :1], 1.0), 0.0)
    out, ns = m.clone(), len(psi)
    out[:, 0] = S[:, 0]
    for c, (a, b) in enumerate(((1, 1), (1, 2), (1, 3), (2, 2), (2, 3), (3, 3))):
        out[:, 4 + c] -= m[:, a] * m[:, b]
    out[:, 11 + ns:] -= m[:, 11:11 + ns] ** 2
    return out


def _slopes64(geo, z, S):
    q = [z[c] * p for p in z["psi"] for c in ("u", "v", "w")]
    flux = _sums64(geo, z, q) / S[:, :1].clamp_min(1e-300)
    ns = len(z["psi"])
    flux -= torch.stack([S[:, 1 + c] * S[:, 11 + a] for a in range(ns) for c in range(3)], 1)
    R = S[:, [4, 5, 6, 5, 7, 8, 6, 8, 9]].reshape(-1, 3, 3)
    ok = torch.linalg.det(R) > 1e-12 * (S[:, [4, 7, 9]].sum(1) / 3).clamp_min(0.0) ** 3
    beta = torch.linalg.solve(torch.where(ok[:, None, None], R, torch.eye(3, dtype=R.dtype, device=R.device)),
                              flux.reshape(-1, ns, 3).transpose(1, 2)).transpose(1, 2).reshape(-1, 3 * ns)
    return flux, torch.where(ok[:, None], beta, 0.0)


def _z64(state):
    z = {k: v.double() for k, v in state.items() if k not in ("elem", "pid")}
    return {**z, "elem": state["elem"].long(), "pid": state["pid"].long()}


_STATE = ("x", "y", "u", "v", "w", "omega", "psi", "elem", "pid")


def _no_state():
    return dict.fromkeys(_STATE)       # listed in an order of the library's own after several steps


class _Fem:
    """P1 finite elements on the mesh with periodic partners merged (rows of slaves stay empty)."""

    def __init__(self, geo):
        self.geo, self.n = geo, len(geo.xy)
        self.d = geo.master[geo.tri]                                          # (E, 3)
        self.own = geo.master == torch.arange(self.n, device="cuda")
        self.darea = self.gather(geo.area[:, None].expand(-1, 3))
        self.wall = torch.zeros(self.n, dtype=torch.bool, device="cuda")
        self.normal = torch.zeros((self.n, 2), dtype=torch.float64, device="cuda")
        e, k = (torch.tensor([int(t[i]) for t in geo.wall_k], device="cuda") for i in (0, 1))
        t = geo.p[e, (k + 1) % 3] - geo.p[e, k]
        nrm = torch.stack([-t[:, 1], t[:, 0]], 1) / t.norm(dim=1, keepdim=True)
        self.seg = geo.tri[e, k], geo.tri[e, (k + 1) % 3]
        for end in ((self.d[e, k]), (self.d[e, (k + 1) % 3])):
            self.wall[end] = True
            self.normal.index_add_(0, end, nrm)
        self.normal /= self.normal.norm(dim=1, keepdim=True).clamp_min(1e-300)

    def gather(self, v):
        """Sum of element-corner values (E, 3, ...) at their nodes."""
        out = torch.zeros((self.n,) + v.shape[2:], dtype=torch.float64, device="cuda")
        return out.index_add_(0, self.d.reshape(-1), v.reshape((-1,) + v.shape[2:]))

    def gradient(self, f):
        return torch.einsum("eam,ead->emd", f[self.d], self.geo.grad)          # (E, m, 2)

    def recover(self, ev):
        a = self.geo.area.reshape((-1,) + (1,) * (ev.dim() - 1)) * ev
        out = self.gather(a[:, None].expand((-1, 3) + ev.shape[1:]))
        return out / self.darea.clamp_min(1e-300).reshape((-1,) + (1,) * (ev.dim() - 1))

    def matrix(self, mass, stiff):
        K = torch.einsum("ead,ebd->eab", self.geo.grad, self.geo.grad) * (self.geo.area * stiff)[:, None, None]
        M = (torch.ones((3, 3), device="cuda", dtype=torch.float64) + torch.eye(3, device="cuda", dtype=torch.float64)) / 12.0
        A = K + mass * self.geo.area[:, None, None] * M
        idx = torch.stack([self.d[:, :, None].expand(-1, 3, 3).reshape(-1), self.d[:, None].expand(-1, 3, 3).reshape(-1)])
        return torch.sparse_coo_tensor(idx, A.reshape(-1), (self.n, self.n)).coalesce().to_sparse_csr(), \
            self.gather(torch.diagonal(A, dim1=1, dim2=2)).clamp_min(1e-300)

    def solve(self, A, diag, b, x, free):
        """Jacobi-preconditioned CG to 1e-13 of the starting residual, on the free rows."""
        free = free[:, None].double()
        r = (b - A @ x) * free
        p = z = r / diag[:, None]
        rz, r0 = (r * z).sum(0), r.norm(dim=0)
        for k in range(6000):
            q = (A @ p) * free
            pq = (p * q).sum(0)
            al = torch.where(pq > 0, rz / pq, 0.0)
            x, r = x + al * p, r - al * q
            z = r / diag[:, None]
            new = (r * z).sum(0)
            p = z + torch.where(rz > 0, new / rz, 0.0) * p
            rz = new
            if k % 50 == 49 and bool((r.norm(dim=0) <= 1e-13 * r0).all()):
                break
        return x


def _solve64(geo, case, S, G=None):
    """Node fields from statistics; G: (G11, G12, G21, G22, G33, C0 eps) per node from a network."""
    fem, ns, m = _Fem(geo), case["ns"], geo.master
    S = S[m]
    U, R, Om = S[:, 1:4], S[:, 4:10], S[:, 10]
    k = 0.5 * (R[:, 0] + R[:, 3] + R[:, 5])
    eps = k * Om
    gU = fem.recover(fem.gradient(U))[m]                                       # (n, 3, 2)
    lap = fem.recover(torch.stack([fem.gradient(gU[:, i])[:, [0, 1], [0, 1]].sum(1) for i in range(3)], 1))
    P = -(R[:, 0] * gU[:, 0, 0] + R[:, 1] * (gU[:, 0, 1] + gU[:, 1, 0]) + R[:, 3] * gU[:, 1, 1] + R[:, 2] * gU[:, 2, 0]
          + R[:, 4] * gU[:, 2, 1])
    F = torch.zeros((fem.n, wl.n_fields_padded(ns)), dtype=torch.float64, device="cuda")
    F[:, 0:3], F[:, 3:9], F[:, 9:12], F[:, 20] = U, gU.reshape(-1, 6), lap, Om
    F[:, 21] = torch.where(eps > 1e-12, 0.73 - 0.5 * P / eps.clamp_min(1e-12), 0.73)
    F[:, 22:22 + ns] = S[:, 11:11 + ns]
    if G is None:
        ec = eps.clamp_min(1e-12)
        L = 0.134 * torch.maximum(k.clamp_min(0.0) ** 1.5 / ec, 72.0 * NU[case["mesh"]] ** 0.75 / ec ** 0.25)
        A, diag = fem.matrix(1.0, (L * L)[fem.d].mean(1))
        n1, n2 = fem.normal.T
        src = -0.75 * 2.1 * eps[:, None] * torch.tensor([1.0, 0.0, 1.0, 1.0], device="cuda", dtype=torch.float64)
        g = torch.stack([-4.5 * eps * n1 * n1, -4.5 * eps * n1 * n2, -4.5 * eps * n2 * n2, 0.0 * eps], 1)
        M = fem.matrix(1.0, 0.0 * geo.area)[0]
        wp = fem.solve(A, diag, M @ src, torch.where(fem.wall[:, None], g, 0.0), fem.own & ~fem.wall)[m]
        kc = k.clamp_min(1e-12)
        G11, G12, G22, G33 = (wp[:, 0] - 0.5 * eps) / kc, wp[:, 1] / kc, (wp[:, 2] - 0.5 * eps) / kc, (wp[:, 3] - 0.5 * eps) / kc
        c0e = (-2.0 / 3.0 * (eps + R[:, 0] * G11 + 2 * R[:, 1] * G12 + R[:, 3] * G22 + R[:, 5] * G33)).clamp_min(0.0)
        T = torch.stack([U[:, 0] ** 2 + R[:, 0], U[:, 0] * U[:, 1] + R[:, 1], U[:, 1] ** 2 + R[:, 3]], 1)
        gT = fem.gradient(T)
        div = torch.stack([gT[:, 0, 0] + gT[:, 1, 1], gT[:, 1, 0] + gT[:, 2, 1]], 1)
        b = fem.gather(-geo.area[:, None] * torch.einsum("ead,ed->ea", geo.grad, div))
        A, diag = fem.matrix(0.0, torch.ones_like(geo.area))
        p = fem.solve(A, diag, b[:, None], torch.zeros((fem.n, 1), dtype=torch.float64, device="cuda"), fem.own)[m]
        F[:, 12:14] = fem.recover(fem.gradient(p)[:, 0])
        F[:, 12] += 0.0 if case["mesh"] == "cavity" else -1.0
        G = torch.stack([G11, G12, G12, G22, G33, c0e], 1)
    F[:, 14:20] = G
    return F[m]


def _features64(case, S):
    """The network's inputs per node from statistics."""
    geo = _Geometry(_host_mesh(case["mesh"], case["nx"], case["ny"]))
    seg = _Fem(geo).seg
    S = S[geo.master]
    k, Om = 0.5 * (S[:, 4] + S[:, 7] + S[:, 9]), S[:, 10]
    eps = k * Om
    best, ew = torch.full_like(k, 1e300), torch.zeros_like(k)
    a, t = geo.xy[seg[0]], geo.xy[seg[1]] - geo.xy[seg[0]]
    for lo in range(0, len(k), 8192):
        for im in ((-1, 0, 1) if geo.period > 0 else (0,)):
            q = geo.xy[lo:lo + 8192, None] - a - torch.tensor([im * geo.period, 0.0], device="cuda")
            s = ((q * t).sum(-1) / (t * t).sum(-1)).clamp(0.0, 1.0)
            d, i = (q - s[..., None] * t).norm(dim=-1).min(1)
            s = s.gather(1, i[:, None])[:, 0]
            near = d < best[lo:lo + 8192]
            best[lo:lo + 8192] = torch.where(near, d, best[lo:lo + 8192])
            ew[lo:lo + 8192] = torch.where(near, (1 - s) * eps[seg[0][i]] + s * eps[seg[1][i]], ew[lo:lo + 8192])
    b = [S[:, c] / (2 * k) - (1.0 / 3.0 if c in (4, 7, 9) else 0.0) for c in range(4, 10)]      # 11 12 13 22 23 33
    II = b[0] ** 2 + b[3] ** 2 + b[5] ** 2 + 2 * (b[1] ** 2 + b[2] ** 2 + b[4] ** 2)
    return torch.stack([best, k.log(), Om.log(), b[0], b[3], b[1], II, (ew / eps).log()], 1)


def _unpack(p):
    out, at = [], 0
    for fi, fo in ((8, 128), (128, 128), (128, 128), (128, 7)):
        out += [p[at:at + fi * fo].reshape(fo, fi), p[at + fi * fo:at + fi * fo + fo]]
        at += fi * fo + fo
    return out


def _net64(p, norm, feat):
    a, q = (feat - norm[0:8]) / norm[8:16], _unpack(p)
    for l in range(3):
        a = torch.tanh(a @ q[2 * l].T + q[2 * l + 1])
    return a @ q[6].T + q[7]


def _gradient64(p, norm, feat, tgt):
    p = p.detach().requires_grad_(True)
    d = _net64(p, norm, feat) - (tgt - norm[23:30]) / norm[30:37]
    loss = (norm[16:23] * d * d).sum() / (7 * len(feat))
    loss.backward()
    return p.grad, float(loss.detach())


def _exact_network(case, seed):
    feat, tgt = (torch.from_numpy(t).cuda().double() for t in _rows(case, seed))
    p = torch.from_numpy(_network(seed)).cuda().double()
    norm = torch.from_numpy(_train_norm(case, seed)).cuda().double()
    if case["kind"] == "gradient":
        g, loss = _gradient64(p, norm, feat, tgt)
        return {"grad": g, "loss": loss}
    m, v, losses, b = torch.zeros_like(p), torch.zeros_like(p), [], case["batch"]
    for s in range(case["steps"]):
        c = s % (len(feat) // b)
        g, loss = _gradient64(p, norm, feat[c * b:(c + 1) * b], tgt[c * b:(c + 1) * b])
        losses.append(loss)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - 1e-3 * (m / (1 - 0.9 ** (s + 1))) / ((v / (1 - 0.999 ** (s + 1))).sqrt() + 1e-8)
    return {"losses": np.array(losses), "params": p}


def _exact_steps(mesh, case, state, F, key, sources):
    """(statistics, fluxes, slopes, particles) after the case's steps from `state`."""
    geo, z, F = _Geometry(mesh), _z64(state), F.double()
    mixing = case["kind"] == "mixing"
    beta = torch.zeros((len(geo.xy), 3 * case["ns"]), dtype=torch.float64, device="cuda") if mixing else None
    S = flux = None
    for k in range(case.get("steps", 1)):
        _step64(geo, z, F, 1 + k, key, case, sources, beta)
        if mixing:
            S = _stats64(geo, z)
            flux, beta = _slopes64(geo, z, S)
    return geo, S if mixing else _stats64(geo, z, raw=case["kind"] == "static"), flux, beta, z


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "gradient"):
        return _exact_network(case, seed)
    ns = case["ns"]
    if kind == "batched":
        wk, _, base = _batch(*_batch_key(case))
        stats = []
        for k, (m, ppe, comp) in enumerate(zip(wk.mesh.parts, wk.n_per_elem, _batch_components(case, wk, seed))):
            state = _particles(m, ppe, ns, 31 * seed + k)
            stats.append(_exact_steps(m, case, state, _fields(base[k], ns, seed + k), *comp)[1])
        return {"stats": torch.cat(stats), **_no_state()}
    mesh = _host_mesh(case["mesh"], case["nx"], case["ny"])
    if kind in ("solve", "surrogate"):
        S, G = torch.from_numpy(_statistics(case, seed)).cuda(), None
        if kind == "surrogate":
            p, norm = (torch.from_numpy(t).cuda().double() for t in _surrogate_net(case, seed))
            y = _net64(p, norm, _features64(case, S)) * norm[30:37] + norm[23:30]
            Om, k = S[:, 10:11], 0.5 * (S[:, 4] + S[:, 7] + S[:, 9])[:, None]
            G = torch.cat([Om * y[:, :5], (k * Om * y[:, 5:6]).clamp_min(0.0)], 1)
        return {"fields": _solve64(_Geometry(mesh), case, S, G)}
    state = _particles(mesh, case["ppe"], ns, seed)
    F = _fields(_base_fields(case["mesh"], case["nx"], case["ny"], 1), ns, seed)
    geo, S, flux, beta, z = _exact_steps(mesh, case, state, F, seed, _sources(case))
    out = {"stats": S}
    if kind == "coupled":
        out["fields"] = _solve64(geo, case, S)
    if kind == "mixing":
        out.update(flux=flux, beta=beta)
    one = {**{k: z[k] for k in _STATE[:7]}, "elem": None, "pid": None}
    return {**out, **(one if case.get("steps", 1) == 1 else _no_state())}
