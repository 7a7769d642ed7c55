"""The work that users of this framework have it do, as cases to be timed and compared.

Kinds of cases, each one pass through the public entry points:

* ``column``   a column advances a stretch of coupled steps, then the whole state is read
               out: FP64 totals, density and velocity fields into pinned buffers, and the
               bubbles (the end-to-end workflow of the benchmark, between two outputs);
* ``replay``   a run in SI units from creation to close, a read of the bubble after
               every step and later every ten (``replay.run``);
* ``restart``  a checkpoint of the populations and the bubbles is loaded, the column
               advances, and the populations are read back for the next checkpoint;
* ``batch``    independent columns of different sizes advance together, all fields read;
* ``adjoint``  loss and gradients of the terminal-velocity mismatch through autograd.

Lattices, diameters, closures and counts are those of the repository's workloads
(``workloads.py``, ``replay.py``, ``bench.py``); the ragged and odd ones are generic.
"""
import math

import numpy as np
import torch

STORAGE = {"f32": (0, 1.0), "f16": (1, 256.0), "bf16": (2, 1.0)}   # code, scale (as bench.py)
WALLS = {"walls": 0x3F, "free_top": 0x7F, "periodic_xy": 0x30}
COLUMN_SIZES = ((32, 32, 64), (48, 48, 96), (64, 64, 128), (96, 96, 192), (128, 128, 256))
SWARM_DENSITY = 100000 / (384 * 384 * 768)
# Largest site-steps for which exact() stays within its time.
EXACT_SITE_STEPS = 6.0e9


def _column(name, nx, ny, nz, storage="f32", omega=1.6, bubbles=1, diameter=2.0, steps=100,
            walls="walls", noise=1e-4, options=False, point=False):
    """bubbles 1: one bubble near the axis at nz/8; more: a swarm in the bottom fifth."""
    return {"name": name, "kind": "column", "nx": nx, "ny": ny, "nz": nz, "storage": storage,
            "omega": omega, "bubbles": bubbles, "diameter": diameter, "steps": steps,
            "walls": walls, "noise": noise, "options": options, "point": point}


def listed():
    return [
        # The smallest calls: the paper's 9 mm run (13 x 13 x 40, odd rows, free-slip top),
        # the bubble read after every step at first, as the replay of Table 4 does.
        {"name": "replay_9mm", "kind": "replay", "d_mm": 9.0, "aspect": 1.25, "seconds": 0.06},
        # The small single-bubble validation column: launches and latency count.
        _column("single_small_f32", 32, 32, 64),
        # A mid-size swarm in 16 bits (the crop that the precision figures are taken on).
        _column("swarm_crop_bf16", 64, 64, 128, "bf16", 1.7, 463, noise=0.0),
        # Odd rows at a size between the small and the large columns.
        _column("single_odd_f32", 127, 127, 255, steps=50),
        # The large single column in both precisions, a snapshot every 100 steps.
        _column("single_large_f32", 256, 256, 512),
        _column("single_large_f16", 256, 256, 512, "f16"),
        # The benchmark's dispersed swarm, released at rest, in both precisions.
        _column("swarm_f32", 384, 384, 768, "f32", 1.7, 100000, steps=50, noise=0.0),
        _column("swarm_f16", 384, 384, 768, "f16", 1.7, 100000, steps=50, noise=0.0),
        # All Table 1 forces, the -sum F reaction and the free-slip top, in a swarm.
        _column("swarm_options_f32", 128, 128, 256, "f32", 1.7, 3704, steps=50, noise=0.0,
                walls="free_top", options=True),
        # Restart from a population checkpoint, ragged sizes, periodic sides.
        {"name": "restart_ragged_f32", "kind": "restart", "nx": 130, "ny": 70, "nz": 150,
         "storage": "f32", "omega": 1.8, "bubbles": 12, "steps": 20, "walls": "periodic_xy"},
        # The grid-independence and stability sweep: 64 columns of five sizes.
        {"name": "batch_64_f32", "kind": "batch", "columns": 64, "storage": "f32", "steps": 40},
        # Gradients of the terminal-velocity mismatch.
        {"name": "adjoint_128", "kind": "adjoint", "nx": 128, "ny": 128, "nz": 256, "omega": 1.6,
         "diameter": 2.5, "steps": 120, "every": 30, "window": 40},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("column", "column", "column", "swarm", "swarm", "replay", "restart",
                       "batch", "adjoint"))
    nx = int(_log(rng, 24, 300))
    ny = int(min(320, max(24, nx * rng.uniform(0.7, 1.4))))
    nz = int(min(640, max(32, nx * rng.uniform(1.2, 2.4))))
    storage = rng.choice(("f32", "f16", "bf16"))
    omega = round(rng.uniform(1.0, 1.9), 3)
    walls = rng.choice(("walls", "walls", "free_top", "periodic_xy"))
    if kind == "replay":
        d = rng.choice((2, 3, 4, 5, 6, 7, 8, 9, 10))
        return {"kind": "replay", "d_mm": float(d), "aspect": 1.25 if d < 4 else
                rng.choice((1.25, 0.625)), "seconds": round(rng.uniform(0.01, 0.06), 3)}
    if kind == "restart":
        n = int(_log(rng, 24, 128))
        return {"kind": "restart", "nx": n, "ny": max(24, int(n * rng.uniform(0.6, 1.2))),
                "nz": int(n * rng.uniform(1.2, 2.2)), "storage": storage, "omega": omega,
                "bubbles": rng.randint(1, 24), "steps": rng.randint(2, 30), "walls": walls}
    if kind == "batch":
        return {"kind": "batch", "columns": int(_log(rng, 2, 64)), "storage": storage,
                "steps": rng.randint(5, 40)}
    if kind == "adjoint":
        n = int(_log(rng, 24, 128))
        return {"kind": "adjoint", "nx": n, "ny": n, "nz": int(n * rng.uniform(1.2, 2.0)),
                "omega": omega, "diameter": round(rng.uniform(1.5, 3.0), 3),
                "steps": rng.randint(20, 120), "every": rng.randint(8, 40), "window": 10}
    c = _column("", nx, ny, nz, storage, omega, steps=rng.randint(10, 100), walls=walls,
                diameter=round(rng.uniform(1.5, 3.0), 3))
    del c["name"]
    if kind == "swarm":
        c["bubbles"] = max(2, int(nx * ny * nz * SWARM_DENSITY * rng.uniform(0.3, 1.5)))
        c["noise"] = 0.0
        c["steps"] = min(c["steps"], 50)
        c["options"] = rng.random() < 0.3
        c["point"] = rng.random() < 0.2
    return c


# ---- inputs ---------------------------------------------------------------------------

def _noise(case, seed, amp):
    """A Gaussian perturbation of the initial velocity, [3, nz, ny, nx] on the GPU (FP64)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 11)
    shape = (3, case["nz"], case["ny"], case["nx"])
    return amp * torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)


def _swarm(rng, n, dims, zmax, max_d=4.0):
    """Lognormal diameters of mean 1.5 and deviation 0.3, centres uniform below zmax."""
    s2 = math.log(1.0 + (0.3 / 1.5) ** 2)
    d = np.minimum(rng.lognormal(math.log(1.5) - 0.5 * s2, math.sqrt(s2), n), max_d)
    r = 0.5 * d
    top = np.array([dims[0], dims[1], zmax], dtype=np.float64)
    pos = r[:, None] + rng.random((n, 3)) * np.maximum(top[None, :] - 2.0 * r[:, None], 0.0)
    return pos, d


def _bubbles(case, seed):
    """(pos [n, 3], diam [n]) of a column or restart case."""
    rng = np.random.default_rng([int(seed), 17])
    dims = (case["nx"], case["ny"], case["nz"])
    n = case["bubbles"]
    if case["kind"] == "column" and n == 1:
        centre = np.array([dims[0] / 2.0, dims[1] / 2.0, max(dims[2] / 8.0, 5.0)])
        return (centre + rng.uniform(-0.5, 0.5, 3))[None, :], np.array([case["diameter"]])
    return _swarm(rng, n, dims, max(0.2 * dims[2], 6.0))


def _populations(case, seed):
    """Populations near equilibrium, [19, nz, ny, nx] FP64 on the GPU, library order."""
    u = _noise(case, seed, 1e-3)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 104729 + 3)
    rho = 1.0 + 1e-4 * torch.randn(u.shape[1:], generator=gen, device="cuda", dtype=torch.float64)
    return torch.stack(_equilibrium(rho, u))


def _batch_columns(case, seed):
    """Sizes as the repository's seeded sweep draws them; omega, d and place by the seed."""
    sizes = np.random.default_rng(1234)
    rng = np.random.default_rng([int(seed), 29])
    cols = []
    for _ in range(case["columns"]):
        dims = COLUMN_SIZES[int(sizes.integers(len(COLUMN_SIZES)))]
        pos = np.array([dims[0] / 2.0, dims[1] / 2.0, dims[2] / 8.0]) + rng.uniform(-0.5, 0.5, 3)
        cols.append((dims, float(rng.uniform(1.0, 1.9)), pos, float(rng.uniform(1.5, 3.0))))
    return cols


def _pinned(n):
    return torch.empty(n, dtype=torch.float64, pin_memory=True)


def prepare(case, seed):
    from paper_1710_07073_gb300 import lbm, replay
    from paper_1710_07073_gb300.adjoint import TerminalVelocityProblem

    kind = case["kind"]
    state = {"case": case, "lbm": lbm}
    if kind == "replay":
        su = replay.setup(case["d_mm"], case["aspect"])
        su["pos"] = su["pos"] + _replay_shift(seed)
        state.update(setup=su, replay=replay)
        return state
    if kind == "adjoint":
        rng = np.random.default_rng([int(seed), 5])
        prob = TerminalVelocityProblem(
            dims=(case["nx"], case["ny"], case["nz"]), omega=case["omega"],
            positions=_adjoint_place(case, seed), steps=case["steps"],
            checkpoint_every=case["every"], window=case["window"], target=8e-5, g=1e-5)
        state.update(problem=prob, u0=_noise(case, seed, 1e-4).float().requires_grad_(True),
                     drag=torch.tensor(1.0 + 0.1 * rng.uniform(-1, 1), requires_grad=True),
                     diameter=torch.tensor(case["diameter"], requires_grad=True))
        return state
    code, scale = STORAGE[case["storage"]]
    params = lbm.lbm_default_params()
    if kind == "batch":
        cols = _batch_columns(case, seed)
        b = lbm.Batch([c[0] for c in cols], [c[1] for c in cols], None, code, scale, params=params)
        lbm.lbm_batch_set_bubbles(b.h, [1] * len(cols), np.concatenate([c[2] for c in cols]),
                                  None, np.array([c[3] for c in cols]))
        sites = [d[0] * d[1] * d[2] for d in b.dims]
        state.update(batch=b, sites=sites, rho=_pinned(sum(sites)), u=_pinned(3 * sum(sites)))
        return state
    if case.get("options"):
        params.forces = lbm.LBM_FORCE_LIFT | lbm.LBM_FORCE_STRESS
        params.reaction = lbm.LBM_REACTION_ALL
    if case.get("point"):
        params.mapping = lbm.LBM_MAP_POINT
    dims = (case["nx"], case["ny"], case["nz"])
    col = lbm.Column(dims, case["omega"], WALLS[case["walls"]], storage=code, scale=scale,
                     params=params)
    S = dims[0] * dims[1] * dims[2]
    pos, diam = _bubbles(case, seed)
    state.update(column=col, pos=pos.reshape(-1), diam=diam)
    if kind == "restart":
        f = _pinned(19 * S)
        f.copy_(_populations(case, seed).reshape(-1))
        state.update(checkpoint=f.numpy())
        return state
    if case["noise"] > 0.0:
        lbm.lbm_set_fields(col.ctx, None, _noise(case, seed, case["noise"]).cpu().numpy())
    lbm.lbm_set_bubbles(col.ctx, state["pos"], None, diam)
    state.update(rho=_pinned(S), u=_pinned(3 * S))
    return state


def _replay_shift(seed):
    return np.random.default_rng([int(seed), 3]).uniform(-0.4, 0.4, 3)


def _adjoint_place(case, seed):
    rng = np.random.default_rng([int(seed), 9])
    return (np.array([case["nx"] / 2.0, case["ny"] / 2.0, max(case["nz"] / 8.0, 6.0)])
            + rng.uniform(-0.5, 0.5, 3))[None, :]


def run(state):
    case, lbm = state["case"], state["lbm"]
    kind = case["kind"]
    if kind == "replay":
        h = state["replay"].run(state["setup"], seconds=case["seconds"])
        return {"z": h["z"], "u_b": h["u_b"], "u_l": h["u_l"], "active": h["active"]}
    if kind == "adjoint":
        for t in ("u0", "drag", "diameter"):
            state[t].grad = None
        loss = state["problem"].loss(state["drag"], state["diameter"], state["u0"])
        loss.backward()
        return {"loss": loss.detach(), "drag": state["drag"].grad,
                "diameter": state["diameter"].grad, "u0": state["u0"].grad}
    if kind == "batch":
        b = state["batch"]
        lbm.lbm_batch_step(b.h, case["steps"])
        rho, u = state["rho"].numpy(), state["u"].numpy()
        at = 0
        for c, s in enumerate(state["sites"]):
            lbm.lbm_batch_get_fields(b.h, c, s, out_rho=rho[at:at + s], out_u=u[3 * at:3 * (at + s)])
            at += s
        return {"rho": state["rho"], "u": state["u"], **lbm.lbm_batch_get_bubbles(b.h)}
    ctx = state["column"].ctx
    if kind == "restart":
        lbm.lbm_set_populations(ctx, state["checkpoint"])
        lbm.lbm_set_bubbles(ctx, state["pos"], None, state["diam"])
        lbm.lbm_step(ctx, case["steps"])
        return {"f": lbm.lbm_get_populations(ctx), **lbm.lbm_get_bubbles(ctx)}
    lbm.lbm_step(ctx, case["steps"])
    totals = lbm.lbm_get_totals(ctx)
    lbm.lbm_get_fields(ctx, out_rho=state["rho"].numpy(), out_u=state["u"].numpy())
    return {"totals": totals, "rho": state["rho"], "u": state["u"], **lbm.lbm_get_bubbles(ctx)}


def work(case):
    """Per step, each population read and written once; each input and output once.

    About 260 FP32 operations per site and step (moments, equilibrium, relaxation)."""
    kind = case["kind"]
    if kind == "replay":
        s = _replay_setup(case)
        S, steps, elem, io = s["nx"] * s["ny"] * s["nz"], s["steps"], 4, 0
    elif kind == "batch":
        S = sum(d[0] * d[1] * d[2] for d, _, _, _ in _batch_columns(case, 0))
        steps, elem, io = case["steps"], 4 if case["storage"] == "f32" else 2, 32
    else:
        S = case["nx"] * case["ny"] * case["nz"]
        steps = case["steps"]
        if kind == "adjoint":
            # Forward 152 B; reverse 228 B (read f and the adjoint, write the adjoint); the
            # gradient and the initial field in FP32.
            return {"bytes": float(S) * (380.0 * steps + 24.0), "flops": 800.0 * S * steps}
        elem = 4 if case["storage"] == "f32" else 2
        io = 304 if kind == "restart" else 32
    return {"bytes": float(S) * (38.0 * elem * steps + io), "flops": 260.0 * S * steps}


# ---- the same in 64 bits, in plain torch ------------------------------------------------

_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
      (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
_OPP = [_C.index((-a, -b, -c)) for a, b, c in _C]
_MIRZ = [_C.index((a, b, -c)) for a, b, c in _C]


def _dot(c, v):
    s = None
    for k in range(3):
        if c[k]:
            t = v[k] if c[k] > 0 else -v[k]
            s = t if s is None else s + t
    return s


def _equilibrium(rho, u):
    base = 1.0 - 1.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
    out = []
    for j in range(19):
        if j == 0:
            out.append(_W[0] * rho * base)
        else:
            cu = _dot(_C[j], u)
            out.append(_W[j] * rho * (base + cu * (3.0 + 4.5 * cu)))
    return out


def _moments(f):
    rho = f[0].clone()
    for j in range(1, 19):
        rho = rho + f[j]
    m = []
    for a in range(3):
        t = None
        for j in range(1, 19):
            if _C[j][a]:
                v = f[j] if _C[j][a] > 0 else -f[j]
                t = v if t is None else t + v
        m.append(t)
    return rho, m


def _collide(f, omega, force):
    rho, m = _moments(f)
    u = [(m[a] + 0.5 * force[a]) / rho if force is not None else m[a] / rho for a in range(3)]
    pref = 1.0 - 0.5 * omega
    base = 1.0 - 1.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
    uF = u[0] * force[0] + u[1] * force[1] + u[2] * force[2] if force is not None else None
    post = []
    for j in range(19):
        cu = _dot(_C[j], u)
        feq = _W[j] * rho * (base if cu is None else base + cu * (3.0 + 4.5 * cu))
        g = f[j] - omega * (f[j] - feq)
        if force is not None:
            t = -3.0 * uF
            if j:
                t = t + (3.0 + 9.0 * cu) * _dot(_C[j], force)
            g = g + pref * _W[j] * t
        post.append(g)
    return post


def _face(n, c, device):
    """Cells of an axis whose source one step against c lies outside."""
    m = torch.zeros(n, dtype=torch.bool, device=device)
    if c > 0:
        m[0] = True
    elif c < 0:
        m[-1] = True
    return m


def _stream(post, walls):
    nz, ny, nx = post[0].shape
    dev = post[0].device
    free_top = bool(walls & 0x40)
    out = [post[0]]
    for j in range(1, 19):
        cx, cy, cz = _C[j]
        moved = torch.roll(post[j], (cz, cy, cx), (0, 1, 2))
        cross = None
        for c, n, bit, shape in ((cx, nx, 0x01, (1, 1, nx)), (cy, ny, 0x04, (1, ny, 1)),
                                 (cz, nz, 0x10, (nz, 1, 1))):
            if not c or not (walls & bit) or (bit == 0x10 and free_top and c < 0):
                continue
            m = _face(n, c, dev).reshape(shape)
            cross = m if cross is None else cross | m
        if free_top and cz < 0:
            mirrored = torch.roll(post[_MIRZ[j]], (cy, cx), (1, 2))
            moved = torch.where(_face(nz, cz, dev).reshape(nz, 1, 1), mirrored, moved)
        if cross is not None:
            moved = torch.where(cross, post[_OPP[j]], moved)
        out.append(moved)
    return out


def _vorticity(u, walls):
    free_top = bool(walls & 0x40)

    def diff(a, d):
        f, ax = u[a], 2 - d
        hi, lo = torch.roll(f, -1, ax), torch.roll(f, 1, ax)
        if walls & (1 << (2 * d)):
            n = f.shape[ax]
            top = 1.0 if (d == 2 and free_top) else -1.0
            first = torch.arange(n, device=f.device) == 0
            last = torch.arange(n, device=f.device) == n - 1
            shape = [1, 1, 1]
            shape[ax] = n
            lo = torch.where(first.reshape(shape), -f, lo)
            hi = torch.where(last.reshape(shape), top * f, hi)
        return 0.5 * (hi - lo)

    return [diff(2, 1) - diff(1, 2), diff(0, 2) - diff(2, 0), diff(1, 0) - diff(0, 1)]


def _windows(x, n, dims, walls, point):
    """Flat node indices [b, k^3] and normalised weights of each bubble's window."""
    idx, wts = [], []
    K = int(2.0 * float(n.detach().max())) + 3
    for a in range(3):
        xa, L = x[:, a:a + 1], dims[a]
        lo = torch.floor((xa - n[:, None]).detach())
        cells = lo + torch.arange(K, device=x.device, dtype=torch.float64)[None, :]
        if point:
            t = (cells + 0.5 - xa) / n[:, None]
            q = 1.0 - t * t
            w = torch.where(t.abs() <= 1.0, q * q, torch.zeros_like(q))
        else:
            s1 = torch.clamp((cells + 1.0 - xa) / n[:, None], -1.0, 1.0)
            s0 = torch.clamp((cells - xa) / n[:, None], -1.0, 1.0)
            w = ((s1 ** 5 - s0 ** 5) / 5.0 - 2.0 * (s1 ** 3 - s0 ** 3) / 3.0 + (s1 - s0))
        if walls & (1 << (2 * a)):
            w = torch.where((cells >= 0) & (cells < L), w, torch.zeros_like(w))
            cells = torch.clamp(cells, 0, L - 1)
        else:
            cells = torch.remainder(cells, L)
        wts.append(w / w.sum(1, keepdim=True))
        idx.append(cells.long())
    w3 = wts[2][:, :, None, None] * wts[1][:, None, :, None] * wts[0][:, None, None, :]
    i3 = ((idx[2][:, :, None, None] * dims[1] + idx[1][:, None, :, None]) * dims[0]
          + idx[0][:, None, None, :])
    b = x.shape[0]
    return i3.reshape(b, -1), w3.reshape(b, -1)


def _interpolate(fields, x, n, dims, walls, point, chunk):
    out = []
    for k in range(0, x.shape[0], chunk):
        i, w = _windows(x[k:k + chunk], n[k:k + chunk], dims, walls, point)
        out.append(torch.stack([(f.reshape(-1)[i] * w).sum(1) for f in fields], 1))
    return torch.cat(out)


def _spread(psi, x, n, dims, walls, point, chunk):
    S = dims[0] * dims[1] * dims[2]
    phi = [torch.zeros(S, dtype=torch.float64, device=x.device) for _ in range(3)]
    for k in range(0, x.shape[0], chunk):
        i, w = _windows(x[k:k + chunk], n[k:k + chunk], dims, walls, point)
        for a in range(3):
            phi[a] = phi[a].index_add(0, i.reshape(-1), (psi[k:k + chunk, a:a + 1] * w).reshape(-1))
    return [p.reshape(dims[2], dims[1], dims[0]) for p in phi]


class _Bubbles:
    """x, u, ul, psi [n, 3], diam [n], active [n]; prev: whether ul holds a step's value."""

    def __init__(self, x, diam):
        self.x, self.d = x, diam
        self.u, self.ul, self.psi = (torch.zeros_like(x) for _ in range(3))
        self.active = torch.ones(x.shape[0], dtype=torch.bool, device=x.device)
        self.prev = False


def _advance(b, ul, om, dims, walls, p):
    """Ten sub-steps of Newton's law with the added mass on the left (all bubbles)."""
    d = b.d[:, None]
    vol = math.pi * d ** 3 / 6.0
    rho_b = p["rho_ratio"]
    meff = (rho_b + 0.5) * vol
    eo = (1.0 - rho_b) * p["g"] * d * d / p["sigma"]
    nu = (2.0 / p["omega"] - 1.0) / 6.0
    fb = torch.zeros_like(b.x)
    fb = torch.cat([fb[:, :2], (1.0 - rho_b) * vol * p["g"]], 1)
    dul = ul - b.ul if b.prev else torch.zeros_like(ul)
    fs = vol * dul if p["options"] else torch.zeros_like(ul)
    fvm_l = 0.5 * vol * dul
    e = 1.0 / (1.0 + 0.163 * eo ** 0.757)
    eo_d = eo / e ** (2.0 / 3.0)
    f_eo = 0.00105 * eo_d ** 3 - 0.0159 * eo_d ** 2 - 0.0204 * eo_d + 0.474
    x, u, total = b.x, b.u, torch.zeros_like(b.x)
    r, dt = 0.5 * d, 0.1
    for _ in range(10):
        v = u - ul
        s2 = (v * v).sum(1, keepdim=True)
        speed = torch.where(s2 > 0, torch.sqrt(torch.where(s2 > 0, s2, torch.ones_like(s2))),
                            torch.zeros_like(s2))
        re = speed * d / nu
        re_e = torch.where(re > 0, torch.where(re > 0, re, torch.ones_like(re)) ** 0.687,
                           torch.zeros_like(re))
        cdv = torch.maximum(torch.minimum(24.0 * nu / d * (1.0 + 0.15 * re_e), 48.0 * nu / d),
                            8.0 / 3.0 * eo / (eo + 4.0) * speed)
        fd = -0.5 * cdv * math.pi * r * r * v * p["drag_scale"]
        if p["options"]:
            cl = torch.where(eo_d < 4.0, torch.minimum(0.288 * torch.tanh(0.121 * re), f_eo),
                             torch.where(eo_d <= 10.0, f_eo, torch.full_like(f_eo, -0.29)))
            fd = fd - cl * vol * torch.cross(v, om, dim=1)
        accel = (fb + fd + fvm_l + fs) / meff
        total = total + (fd + fs + 0.5 * vol * (dul - accel) if p["options"] else fd)
        u = u + accel * dt
        x = x + u * dt
        xs, us = [], []
        for a in range(3):
            xa, ua, L = x[:, a:a + 1], u[:, a:a + 1], float(dims[a])
            if walls & (1 << (2 * a)):
                low, high = xa < r, xa > L - r
                xa = torch.where(low, r, torch.where(high, L - r, xa))
                ua = torch.where(low, torch.clamp(ua, min=0.0),
                                 torch.where(high, torch.clamp(ua, max=0.0), ua))
            else:
                xa = xa - L * torch.floor((xa / L).detach())
            xs.append(xa)
            us.append(ua)
        x, u = torch.cat(xs, 1), torch.cat(us, 1)
    return x, u, -total / 10.0


def _step(f, b, dims, walls, p, chunk=4096):
    """One coupled step; returns the new populations and bubbles."""
    rho, m = _moments(f)
    nodes = [c / rho for c in m]
    n = 1.5 * b.d
    ul = _interpolate(nodes, b.x, n, dims, walls, p["point"], chunk)
    om = (_interpolate(_vorticity(nodes, walls), b.x, n, dims, walls, p["point"], chunk)
          if p["options"] else None)
    del rho, m, nodes
    x, u, psi = _advance(b, ul, om, dims, walls, p)
    live = b.active[:, None]
    nb = _Bubbles(torch.where(live, x, b.x), b.d)
    nb.u, nb.ul = torch.where(live, u, b.u), torch.where(live, ul, b.ul)
    nb.psi, nb.prev = torch.where(live, psi, b.psi), True
    force = _spread(torch.where(live, psi, torch.zeros_like(psi)), nb.x, n, dims, walls,
                    p["point"], chunk)
    top = (nb.x[:, 2] >= dims[2] - 0.5 * b.d) if walls & 0x20 else torch.zeros_like(b.active)
    nb.active = b.active & ~top
    return _stream(_collide(f, p["omega"], force), walls), nb


def _physics(case, omega, **more):
    return {"omega": omega, "g": 1e-5, "sigma": 5.84e-6, "rho_ratio": 1e-3, "drag_scale": 1.0,
            "options": bool(case.get("options")), "point": bool(case.get("point")), **more}


def _f64(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def _sorted_bubbles(pos, diam):
    """Bubbles by diameter (windows of one chunk alike), and the way back."""
    order = np.argsort(diam, kind="stable")
    back = torch.as_tensor(np.argsort(order, kind="stable"), device="cuda")
    return _Bubbles(_f64(pos[order]), _f64(diam[order])), back


def _bubble_outputs(b, back):
    return {"pos": b.x[back], "vel": b.u[back], "ul": b.ul[back], "psi": b.psi[back],
            "active": b.active[back].cpu().numpy()}


def _fields(f):
    rho, m = _moments(f)
    return rho, [c / rho for c in m]


def _rest(dims, u=None):
    nx, ny, nz = dims
    rho = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    if u is None:
        return [w * rho for w in _W]
    return _equilibrium(rho, u)


def _replay_setup(case):
    """Appendix A's conversion of the physical column, by its formulas."""
    d = case["d_mm"] * 1e-3
    lcf, tcf = 1.0 / (case["aspect"] * d), 1e4
    mcf = lcf ** 3 / 1000.0
    n = int(round(0.15 * lcf))
    return {"nx": n, "ny": n, "nz": int(round(0.45 * lcf)), "lcf": lcf, "tcf": tcf,
            "omega": 1.0 / (3.0 * 1e-6 * lcf * lcf / tcf + 0.5), "g": 9.81 * lcf / tcf ** 2,
            "sigma": 0.073 * mcf / tcf ** 2, "d": d * lcf, "steps": int(round(case["seconds"] * tcf)),
            "pos": np.array([0.5 * n, 0.5 * n, (0.005 + 0.5 * d) * lcf])}


def exact(case, seed):
    kind = case["kind"]
    w = work(case)["flops"] / (800.0 if kind == "adjoint" else 260.0)
    if w > (1.0e9 if kind == "adjoint" else EXACT_SITE_STEPS):
        return None
    with torch.no_grad():
        if kind == "replay":
            return _exact_replay(case, seed)
        if kind == "batch":
            return _exact_batch(case, seed)
        if kind == "adjoint":
            return _exact_adjoint(case, seed)
        dims = (case["nx"], case["ny"], case["nz"])
        walls = WALLS[case["walls"]]
        b, back = _sorted_bubbles(*_bubbles(case, seed))
        p = _physics(case, case["omega"])
        if kind == "restart":
            f = list(_populations(case, seed))
        else:
            f = _rest(dims, _noise(case, seed, case["noise"]) if case["noise"] > 0.0 else None)
        for _ in range(case["steps"]):
            f, b = _step(f, b, dims, walls, p)
        if kind == "restart":
            return {"f": torch.stack(f).reshape(-1), **_bubble_outputs(b, back)}
        rho, u = _fields(f)
        totals = torch.stack([rho.sum()] + [(rho * c).sum() for c in u])
        return {"totals": totals, "rho": rho.reshape(-1), "u": torch.stack(u).reshape(-1),
                **_bubble_outputs(b, back)}


def _exact_replay(case, seed):
    s = _replay_setup(case)
    dims, walls = (s["nx"], s["ny"], s["nz"]), 0x7F
    b = _Bubbles(_f64((s["pos"] + _replay_shift(seed))[None, :]), _f64([s["d"]]))
    p = _physics(case, s["omega"], g=s["g"], sigma=s["sigma"])
    f = _rest(dims)
    z, ub, ul, act = [], [], [], []
    step, v = 0, s["tcf"] / s["lcf"]
    while step < s["steps"]:
        k = 1 if step < 300 else min(10, s["steps"] - step)
        for _ in range(k):
            f, b = _step(f, b, dims, walls, p)
        step += k
        z.append(float(b.x[0, 2]) / s["lcf"])
        ub.append(float(b.u[0, 2]) * v)
        ul.append(float(b.ul[0, 2]) * v)
        act.append(bool(b.active[0]))
        if not act[-1]:
            break
    return {"z": np.array(z), "u_b": np.array(ub), "u_l": np.array(ul), "active": np.array(act)}


def _exact_batch(case, seed):
    rhos, us, bs = [], [], []
    for dims, omega, pos, d in _batch_columns(case, seed):
        b, f = _Bubbles(_f64(pos[None, :]), _f64([d])), _rest(dims)
        p = _physics(case, omega)
        for _ in range(case["steps"]):
            f, b = _step(f, b, dims, 0x3F, p)
        rho, u = _fields(f)
        rhos.append(rho.reshape(-1))
        us.append(torch.stack(u).reshape(-1))
        bs.append(_bubble_outputs(b, torch.zeros(1, dtype=torch.long, device="cuda")))
    joined = {k: torch.cat([b[k] for b in bs]) for k in ("pos", "vel", "ul", "psi")}
    return {"rho": torch.cat(rhos), "u": torch.cat(us), **joined,
            "active": np.concatenate([b["active"] for b in bs])}


def _exact_adjoint(case, seed):
    """Reverse mode by torch, a step at a time from stored states (every 16th, then all)."""
    dims, walls = (case["nx"], case["ny"], case["nz"]), 0x3F
    rng = np.random.default_rng([int(seed), 5])
    scale = torch.tensor(1.0 + 0.1 * rng.uniform(-1, 1)).double().cuda()
    diam = torch.tensor(case["diameter"]).double().cuda().reshape(1)
    u0 = _noise(case, seed, 1e-4).float().double()
    p = _physics(case, case["omega"], drag_scale=scale)
    first = torch.stack(_rest(dims, u0))
    place = _f64(_adjoint_place(case, seed))

    def advance(s, d, sd, prev):
        b = _Bubbles(s[1], d)
        b.u, b.ul, b.prev = s[2], s[3], prev
        g, nb = _step(list(s[0].unbind(0)), b, dims, walls, {**p, "drag_scale": sd})
        return torch.stack(g), nb.x, nb.u, nb.ul

    zero = torch.zeros_like(place)
    s, kept, rise = (first, place, zero, zero), [], []
    for k in range(case["steps"]):
        if k % 16 == 0:
            kept.append(s)
        s = advance(s, diam, scale, k > 0)
        rise.append(float(s[2][0, 2]))
    off = sum(rise[-case["window"]:]) / case["window"] - 8e-5
    seed_u = 2.0 * off / case["window"]
    adj = [torch.zeros_like(t) for t in s]
    g_scale, g_diam = torch.zeros_like(scale), torch.zeros_like(diam)
    for seg in range(len(kept) - 1, -1, -1):
        states = [kept[seg]]
        hi = min(case["steps"], 16 * (seg + 1))
        for k in range(16 * seg, hi - 1):
            states.append(advance(states[-1], diam, scale, k > 0))
        for k in range(hi - 1, 16 * seg - 1, -1):
            if k >= case["steps"] - case["window"]:
                adj[2][0, 2] += seed_u
            with torch.enable_grad():
                ins = [t.detach().requires_grad_(True) for t in states.pop()]
                d, sd = diam.detach().requires_grad_(True), scale.detach().requires_grad_(True)
                out = advance(ins, d, sd, k > 0)
                got = torch.autograd.grad(out, ins + [d, sd], adj, allow_unused=True)
            adj = [torch.zeros_like(t) if g is None else g for t, g in zip(ins, got)]
            g_diam, g_scale = g_diam + got[4], g_scale + got[5]
        kept.pop()
    with torch.enable_grad():
        u = u0.detach().requires_grad_(True)
        g_u0, = torch.autograd.grad(torch.stack(_rest(dims, u)), u, adj[0])
    return {"loss": torch.tensor(off * off, dtype=torch.float64), "drag": g_scale,
            "diameter": g_diam.reshape(()), "u0": g_u0}
