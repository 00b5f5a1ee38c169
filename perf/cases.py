"""The work this framework is measured on: time stepping of the spectral-element solver over
its range of sizes and orders, many shots, uneven models, the stiffness action, the material
gradient, and the learned surrogate's inference and training gradient.

Every case goes through the public entry points (``sem``, ``adjoint``, ``surrogate``). The
inputs are made here from the seed alone; ``exact`` restates each path in float64 with plain
PyTorch. Conventions (those of include/sem.h): local point p = i + n j + n^2 k, global lattice
node gx + Gx (gy + Gy gz), element corner c = a + 2 b + 4 d.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2606_12850_gb300 import adjoint, sem, surrogate

SIDE = 4000.0  # m, longest edge of a model
LAYERS = ((5000.0, 3000.0), (3500.0, 2600.0), (2000.0, 2200.0))  # (vp, rho) bottom up; vs = vp / 1.73
F0 = 10.0  # Hz, Ricker
FORCE = 1.0e10  # N


def listed():
    return [
        # the smallest model a user runs (the 8^3 homogeneous cube of the tests) from host
        # buffers to host seismograms and state: launches and host copies count
        {"name": "run_cube8_host", "kind": "run", "nx": 8, "ny": 8, "nz": 8, "ngll": 5, "steps": 100, "host": True},
        # the framework's main path at the benchmark's order: a layered model larger than L2,
        # restarted from a device state, 256 surface receivers
        {"name": "run_n5_48", "kind": "run", "nx": 48, "ny": 48, "nz": 48, "ngll": 5, "steps": 24, "host": False},
        # the same path at the other orders of the (h, p) sweep, on meshes no brick divides
        {"name": "run_n3_odd", "kind": "run", "nx": 45, "ny": 41, "nz": 50, "ngll": 3, "steps": 24, "host": False},
        {"name": "run_n7_odd", "kind": "run", "nx": 25, "ny": 21, "nz": 23, "ngll": 7, "steps": 24, "host": False},
        {"name": "run_n9_odd", "kind": "run", "nx": 16, "ny": 15, "nz": 17, "ngll": 9, "steps": 24, "host": False},
        # many shots of one model, as the surrogate's training data are made
        {"name": "shots32_n5_20", "kind": "shots", "nx": 20, "ny": 20, "nz": 20, "ngll": 5, "shots": 32, "steps": 24},
        # f = -K u on caller arrays: an eigenvalue or implicit solver around the operator
        {"name": "stiffness_n5_40", "kind": "stiffness", "nx": 44, "ny": 36, "nz": 40, "ngll": 5},
        # full-waveform inversion: seismograms, misfit and the gradient in rho, kappa, mu
        {"name": "gradient_n5_20", "kind": "gradient", "nx": 20, "ny": 20, "nz": 20, "ngll": 5, "steps": 64},
        # several uneven models of mixed order stepped together
        {"name": "group_mixed", "kind": "group", "models": "16:4,12:5,18:5,10:6,9:7,7:8", "steps": 30},
        # the surrogate answering a catalogue of sources, and one source
        {"name": "surrogate_4096", "kind": "sur_forward", "batch": 4096},
        {"name": "surrogate_1", "kind": "sur_forward", "batch": 1},
        # one training step's loss and gradients, read back
        {"name": "surrogate_grad_256", "kind": "sur_gradient", "batch": 256},
    ]


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "shots", "stiffness", "gradient", "group", "sur_forward",
                       "sur_gradient"])

    def box(ngll, lo, hi):
        points = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        n = (points / ngll ** 3) ** (1.0 / 3.0)
        side = lambda: max(2, int(round(n * rng.uniform(0.8, 1.25))))  # noqa: E731
        return {"nx": side(), "ny": side(), "nz": side(), "ngll": ngll}

    if kind == "run":
        return {"kind": "run", **box(rng.randint(3, 10), 4e4, 4e6), "steps": rng.randint(11, 30),
                "host": rng.random() < 0.25}
    if kind == "shots":
        return {"kind": "shots", **box(rng.randint(3, 7), 3e4, 6e5), "shots": rng.randint(2, 33),
                "steps": rng.randint(11, 30)}
    if kind == "stiffness":
        return {"kind": "stiffness", **box(rng.randint(3, 10), 4e4, 6e6)}
    if kind == "gradient":
        return {"kind": "gradient", **box(rng.randint(4, 7), 3e4, 6e5), "steps": rng.randint(20, 60)}
    if kind == "group":
        models = ["%d:%d" % (rng.randint(4, 14), rng.randint(4, 8)) for _ in range(rng.randint(2, 6))]
        return {"kind": "group", "models": ",".join(models), "steps": rng.randint(12, 30)}
    if kind == "sur_forward":
        return {"kind": "sur_forward", "batch": int(round(math.exp(rng.uniform(0.0, math.log(3000.0)))))}
    return {"kind": "sur_gradient", "batch": int(round(math.exp(rng.uniform(math.log(4.0), math.log(256.0)))))}


# ---- inputs ---------------------------------------------------------------------------------


def box_mesh(nx, ny, nz, ngll, seed, jitter=0.1):
    """A jittered lattice of hexahedra of edge SIDE / max(n): ibool, corners, layer of each element."""
    n, N = ngll, ngll - 1
    h = SIDE / max(nx, ny, nz)
    rs = np.random.RandomState(seed % (1 << 31))
    verts = np.stack(np.meshgrid(np.arange(nz + 1), np.arange(ny + 1), np.arange(nx + 1), indexing="ij")[::-1],
                     axis=-1) * h
    if min(nx, ny, nz) > 1:
        verts[1:-1, 1:-1, 1:-1] += rs.uniform(-jitter * h, jitter * h, (nz - 1, ny - 1, nx - 1, 3))
    ez, ey, ex = (g.ravel() for g in np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij"))
    ctrl = np.stack([verts[ez + (c >> 2 & 1), ey + (c >> 1 & 1), ex + (c & 1)] for c in range(8)], axis=1)
    Gx, Gy, Gz = nx * N + 1, ny * N + 1, nz * N + 1
    kk, jj, ii = (g.ravel() for g in np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij"))
    node0 = (ex + Gx * (ey + Gy * ez)).astype(np.int32) * np.int32(N)
    ibool = node0[:, None] + (ii + Gx * (jj + Gy * kk)).astype(np.int32)[None, :]
    return ibool, ctrl, (Gx, Gy, Gz), np.minimum(3 * ez // nz, 2), h


def materials(ctrl, layer, np3, seed):
    """Three layers with a Gaussian velocity anomaly of 5 % (per element), float32 [nspec][ngll^3]."""
    rs = np.random.RandomState((seed + 77) % (1 << 31))
    c = ctrl.mean(axis=1)
    x0 = c[rs.randint(len(c))]
    scale = 1.0 + 0.05 * np.exp(-((c - x0) ** 2).sum(axis=1) / (2.0 * (SIDE / 8.0) ** 2))
    vp = np.array([l[0] for l in LAYERS])[layer] * scale
    rho = np.array([l[1] for l in LAYERS])[layer]
    wide = lambda a: np.repeat(a.astype(np.float32)[:, None], np3, axis=1)  # noqa: E731
    return wide(rho), wide(vp), wide(vp / 1.73)


def gll(n):
    """GLL points, weights and the derivative matrix h[i][l] = l_l'(x_i), float64."""
    P = np.polynomial.legendre.Legendre.basis(n - 1)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real) if n > 2 else [], [1.0]])
    w = 2.0 / (n * (n - 1) * P(x) ** 2)
    b = np.array([1.0 / np.prod([x[l] - x[m] for m in range(n) if m != l]) for l in range(n)])
    h = np.array([[b[l] / b[i] / (x[i] - x[l]) if l != i else 0.0 for l in range(n)] for i in range(n)])
    h[np.arange(n), np.arange(n)] = -h.sum(axis=1)
    return x, w, h


def time_step(ngll, h):
    """Courant number 0.32 on the unjittered spacing (the jitter shrinks an edge by up to 20 %)."""
    x = gll(ngll)[0]
    return 0.32 * 0.5 * h * (x[1] - x[0]) / (1.05 * LAYERS[0][0])


def wavefield(grid, seed, scale, stream):
    """A field of three plane waves, 6 to 12 nodes per wavelength (what the orders resolve),
    float32 [nglob][3], on the GPU."""
    rs = np.random.RandomState((seed * 7 + stream) % (1 << 31))
    ax = [torch.arange(g, device="cuda", dtype=torch.float32) for g in grid]
    out = torch.zeros((grid[2], grid[1], grid[0], 3), device="cuda")
    for _ in range(3):
        d, phase, pol = rs.normal(size=3), rs.uniform(0.0, 6.28), rs.normal(size=3)
        k = d / np.linalg.norm(d) * 2.0 * math.pi / rs.uniform(6.0, 12.0)
        wave = torch.sin(k[2] * ax[2][:, None, None] + k[1] * ax[1][None, :, None] + k[0] * ax[0][None, None, :] + phase)
        out += wave[..., None] * torch.tensor(pol * scale, device="cuda", dtype=torch.float32)
    return out.reshape(-1, 3)


def model_inputs(nx, ny, nz, ngll, seed, shots=1, state=True):
    """Everything one model's run is given: mesh, material, time step, sources, receivers, state."""
    ibool, ctrl, grid, layer, h = box_mesh(nx, ny, nz, ngll, seed)
    rho, vp, vs = materials(ctrl, layer, ngll ** 3, seed)
    rs = np.random.RandomState((seed + 5) % (1 << 31))
    node = lambda x, y, z: int(x + grid[0] * (y + grid[1] * z))  # noqa: E731
    shallow = lambda: grid[2] - 1 - rs.randint(1, 2 * (ngll - 1))  # noqa: E731  (the top two element layers)
    src = [node(rs.randint(1, grid[0] - 1), rs.randint(1, grid[1] - 1), shallow()) for _ in range(shots)]
    force = rs.normal(size=(shots, 3)) * FORCE
    m = 16 if min(nx, ny) >= 16 else 4
    rec = [node((2 * i + 1) * grid[0] // (2 * m), (2 * j + 1) * grid[1] // (2 * m), grid[2] - 1)
           for j in range(m) for i in range(m)]
    dt = time_step(ngll, h)
    out = dict(ngll=ngll, ibool=ibool, ctrl=ctrl, nglob=grid[0] * grid[1] * grid[2], rho=rho, vp=vp, vs=vs, dt=dt,
               src=np.array(src, np.int32), force=force, rec=np.array(rec, np.int32), t0=8.0 * dt)
    if state:  # displacement, velocity and acceleration of the sizes such waves have
        out["state"] = [wavefield(grid, seed, s, q) for q, s in enumerate((1e-3, 5e-2, 2.0))]
    return out


def context(m):
    """The handle a user's program keeps: mesh, material and time step set."""
    ctx = sem.sem_create(m["ngll"], 0)
    sem.sem_set_mesh_corners(ctx, m["ibool"], m["ctrl"], m["nglob"])
    sem.sem_set_material(ctx, m["rho"], m["vp"], m["vs"])
    sem.sem_set_dt(ctx, m["dt"])
    return ctx


def box_of(case):
    return case["nx"], case["ny"], case["nz"], case["ngll"]


def group_models(case):
    return [(n, n, n, g) for n, g in (tuple(int(v) for v in t.split(":")) for t in case["models"].split(","))]


# the surrogate's network (the default surrogate.Spec), restated for exact()
IN, HID, C0, L0, STAGES, UP, MOMENTS = 9, 512, 64, 125, (96, 96, 96, 1152), (2, 2, 2, 1), 6
OUT_C, OUT_L = 192, 1000


def network_shapes():
    out = [(HID, IN), (HID,), (HID, HID), (HID,), (C0 * L0, HID), (C0 * L0,)]
    c = C0
    for co in STAGES:
        out += [(co, c, 3), (co,)]
        c = co
    return out


def network_params(seed):
    """He-uniform weights and small biases, float32, the library's order."""
    g = torch.Generator().manual_seed(seed)
    parts = []
    for s in network_shapes():
        bound = math.sqrt(6.0 / math.prod(s[1:])) if len(s) > 1 else 0.05
        parts.append((torch.rand(s, generator=g) * 2.0 - 1.0).mul_(bound).reshape(-1))
    return torch.cat(parts).numpy()


def network_inputs(batch, seed, targets):
    """Scaled source positions with unit moment tensors, and smooth decaying target traces."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    pos = torch.rand((batch, 3), generator=g, device="cuda") * 1.8 - 0.9
    mom = torch.randn((batch, MOMENTS), generator=g, device="cuda")
    x = torch.cat([pos, mom / mom.norm(dim=1, keepdim=True)], dim=1).contiguous()
    if not targets:
        return x, None
    t = torch.linspace(0.0, 1.0, OUT_L, device="cuda")
    at = torch.rand((batch, OUT_C, 1), generator=g, device="cuda") * 0.6 + 0.2
    amp = torch.randn((batch, OUT_C, 1), generator=g, device="cuda")
    s = (t - at) * 25.0
    return x, (amp * (1.0 - 2.0 * s * s) * torch.exp(-s * s)).contiguous()


# ---- prepare, run, work ---------------------------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": dict(case)}
    if kind in ("sur_forward", "sur_gradient"):
        B = case["batch"]
        s["model"] = surrogate.Model(surrogate.Spec(), max_batch=min(B, 256))
        s["model"].set_params(network_params(seed))
        s["x"], s["t"] = network_inputs(B, seed, kind == "sur_gradient")
        if kind == "sur_forward":
            s["y"] = torch.empty((B, OUT_C, OUT_L), device="cuda")
        return s
    if kind == "group":
        s["parts"] = []
        for k, b in enumerate(group_models(case)):
            m = model_inputs(*b, seed + 1000 * k)
            ctx = context(m)
            sem.sem_set_source_nodes(ctx, m["src"], m["force"], F0, m["t0"])
            s["parts"].append((ctx, m["state"], [torch.empty_like(f) for f in m["state"]]))
        s["group"] = sem.Group([p[0] for p in s["parts"]])
        return s
    S = case.get("shots", 1)
    m = model_inputs(*box_of(case), seed, shots=S, state=kind != "gradient" and kind != "shots")
    ctx = context(m)
    s["ctx"] = ctx
    if kind == "stiffness":
        s["u"], s["f"] = m["state"][0], torch.empty_like(m["state"][0])
        return s
    if S > 1:
        sem.sem_set_shots(ctx, S)
        sem.sem_set_shot_sources(ctx, np.arange(S), m["src"], m["force"], F0, m["t0"])
    else:
        sem.sem_set_source_nodes(ctx, m["src"], m["force"], F0, m["t0"])
    sem.sem_set_receiver_nodes(ctx, m["rec"])
    steps, nrec = case["steps"], len(m["rec"])
    if kind == "gradient":
        mu = (m["rho"] * m["vs"] * m["vs"]).astype(np.float32)
        kappa = (m["rho"] * m["vp"] * m["vp"]).astype(np.float32) - np.float32(4.0 / 3.0) * mu
        s["sim"] = adjoint.Simulation(ctx, m["dt"], steps, keep_all=True)
        s["mat"] = [torch.from_numpy(a).cuda().requires_grad_(True) for a in (m["rho"], kappa, mu)]
        s["obs"] = observed(nrec, steps, seed)
        return s
    if case.get("host"):
        s["state"] = [f.cpu().numpy() for f in m["state"]]
        return s
    if S > 1:  # a shot starts from rest; its state is of no use to the caller
        s["seis"] = torch.empty((S, nrec, 3, steps), device="cuda")
        s["zero"] = s["out"] = torch.empty((S, m["nglob"], 3), device="cuda")
        return s
    s["state"] = m["state"]
    s["out"] = [torch.empty_like(f) for f in m["state"]]
    s["seis"] = torch.empty((nrec, 3, steps), device="cuda")
    return s


def observed(nrec, steps, seed):
    """Recorded traces to fit: smooth, of the size the sources produce at the surface."""
    rs = np.random.RandomState((seed + 9) % (1 << 31))
    t = np.arange(steps) / steps
    a, f, p = rs.normal(size=(nrec, 3, 1)), rs.uniform(2.0, 9.0, (nrec, 3, 1)), rs.uniform(0.0, 6.28, (nrec, 3, 1))
    return torch.from_numpy((1e-6 * a * np.sin(6.28 * f * t + p)).astype(np.float32)).cuda()


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "run":
        ctx = s["ctx"]
        if case["host"]:
            sem.sem_set_state(ctx, *s["state"])
            seis = sem.sem_run(ctx, case["steps"])
            return {"seis": seis, "state": list(sem.sem_get_state(ctx))}
        sem.sem_set_state_dev(ctx, *s["state"])
        sem.sem_run_dev(ctx, case["steps"], s["seis"])
        sem.sem_get_state_dev(ctx, *s["out"])
        return {"seis": s["seis"], "state": s["out"]}
    if kind == "shots":
        ctx = s["ctx"]
        sem.sem_set_state_dev(ctx)  # from rest
        sem.sem_run_dev(ctx, case["steps"], s["seis"])
        sem.sem_get_state_dev(ctx, s["out"])
        return {"seis": s["seis"], "u": s["out"]}
    if kind == "stiffness":
        sem.sem_apply_stiffness(s["ctx"], s["u"], s["f"])
        return s["f"]
    if kind == "gradient":
        rho, kappa, mu = s["mat"]
        rho.grad = kappa.grad = mu.grad = None
        seis = adjoint.Seismograms.apply(rho, kappa, mu, s["sim"])
        loss = 0.5 * ((seis - s["obs"]) ** 2).sum()
        loss.backward()
        return {"seis": seis.detach(), "grad": [rho.grad, kappa.grad, mu.grad]}
    if kind == "group":
        for ctx, state, _ in s["parts"]:
            sem.sem_set_state_dev(ctx, *state)
        s["group"].step(case["steps"])
        for ctx, _, out in s["parts"]:
            sem.sem_get_state_dev(ctx, *out)
        return [out for _, _, out in s["parts"]]
    if kind == "sur_forward":
        s["model"].forward(s["x"], s["y"])
        return s["y"]
    loss = s["model"].loss_grad(s["x"], s["t"])
    return {"loss": loss, "grads": s["model"].get_grads()}


def sizes(nx, ny, nz, ngll):
    n = ngll - 1
    return nx * ny * nz * ngll ** 3, (nx * n + 1) * (ny * n + 1) * (nz * n + 1)


def step_work(box):
    """(bytes, flops) of one time step: per local point ibool, nine inverse-Jacobian terms, two
    moduli and J (52 B); per node u, v, a and 1/M read, u, v, a written (76 B); the six
    contractions, the Jacobian map, Hooke's law and the fluxes."""
    nloc, nglob = sizes(*box)
    return 52.0 * nloc + 76.0 * nglob, (36.0 * box[3] + 140.0) * nloc


def work(case):
    kind = case["kind"]
    if kind == "run":
        b, f = step_work(box_of(case))
        nglob = sizes(*box_of(case))[1]
        return {"bytes": case["steps"] * b + 72.0 * nglob, "flops": case["steps"] * f}
    if kind == "shots":
        nloc, nglob = sizes(*box_of(case))
        f = step_work(box_of(case))[1]
        S, K = case["shots"], case["steps"]
        return {"bytes": K * (52.0 * nloc + (72.0 * S + 4.0) * nglob) + 12.0 * S * nglob, "flops": K * S * f}
    if kind == "stiffness":
        nloc, nglob = sizes(*box_of(case))
        return {"bytes": 52.0 * nloc + 24.0 * nglob, "flops": (36.0 * case["ngll"] + 140.0) * nloc}
    if kind == "gradient":
        # a step forward (its displacement kept) and one back (the sweep of the adjoint field,
        # the strains of both fields and three sums per point); two fields of 12 B per node read
        b, f = step_work(box_of(case))
        nloc, nglob = sizes(*box_of(case))
        return {"bytes": case["steps"] * (2.0 * b + 36.0 * nglob) + 24.0 * nloc, "flops": case["steps"] * 3.0 * f}
    if kind == "group":
        each = [step_work(b) for b in group_models(case)]
        return {"bytes": case["steps"] * sum(e[0] for e in each), "flops": case["steps"] * sum(e[1] for e in each)}
    B = case["batch"]
    mul = IN * HID + HID * HID + HID * C0 * L0
    c, l = C0, L0
    for co, up in zip(STAGES, UP):
        l *= up
        mul += co * c * 3 * l
        c = co
    params = sum(math.prod(s) for s in network_shapes())
    if kind == "sur_forward":
        return {"bytes": 4.0 * (B * (IN + OUT_C * OUT_L) + params), "flops": 2.0 * mul * B}
    return {"bytes": 4.0 * (B * (IN + OUT_C * OUT_L) + 2 * params), "flops": 6.0 * mul * B}


# ---- the same in float64 --------------------------------------------------------------------


class Exact:
    """One model in float64: the stiffness action and the explicit Newmark scheme."""

    def __init__(self, m):
        n = m["ngll"]
        x, w, h = gll(n)
        dev = dict(device="cuda", dtype=torch.float64)
        self.n, self.nglob, self.dt = n, m["nglob"], m["dt"]
        self.ib = torch.from_numpy(m["ibool"]).cuda().long().reshape(-1)
        self.E = m["ibool"].shape[0]
        self.h = torch.tensor(h, **dev)
        self.w = torch.tensor(w, **dev)
        lo, hi = torch.tensor((1.0 - x) / 2.0, **dev), torch.tensor((1.0 + x) / 2.0, **dev)
        N = torch.stack([lo, hi])  # [corner bit][point]
        dN = torch.tensor([[-0.5] * n, [0.5] * n], **dev)
        ctrl = torch.from_numpy(m["ctrl"]).cuda().reshape(-1, 2, 2, 2, 3)  # [e][d][b][a][xyz]
        J = torch.stack([torch.einsum("edbac,dk,bj,ai->ekjic", ctrl, *t)
                         for t in ((N, N, dN), (N, dN, N), (dN, N, N))], dim=-1)  # [e][k][j][i][x][xi]
        self.det = (J[..., 0, 0] * (J[..., 1, 1] * J[..., 2, 2] - J[..., 1, 2] * J[..., 2, 1])
                    - J[..., 0, 1] * (J[..., 1, 0] * J[..., 2, 2] - J[..., 1, 2] * J[..., 2, 0])
                    + J[..., 0, 2] * (J[..., 1, 0] * J[..., 2, 1] - J[..., 1, 1] * J[..., 2, 0]))
        G = torch.empty_like(J)  # [..][xi][x]: the inverse, by cofactors
        for r in range(3):
            a, b = (r + 1) % 3, (r + 2) % 3
            for d in range(3):
                p, q = (d + 1) % 3, (d + 2) % 3
                G[..., r, d] = (J[..., p, a] * J[..., q, b] - J[..., p, b] * J[..., q, a]) / self.det
        self.G = G
        self.w3 = self.w[:, None, None] * self.w[None, :, None] * self.w[None, None, :]

    def moduli(self, m):
        rho, vp, vs = (torch.from_numpy(m[k]).cuda().double() for k in ("rho", "vp", "vs"))
        mu = rho * vs * vs
        return rho, rho * vp * vp - 4.0 / 3.0 * mu, mu

    def set_material(self, rho, kappa, mu):
        shape = (self.E, self.n, self.n, self.n)
        self.kappa, self.mu = kappa.reshape(shape), mu.reshape(shape)
        lump = (self.w3 * self.det * rho.reshape(shape)).reshape(-1)
        self.minv = 1.0 / torch.zeros(self.nglob, device="cuda", dtype=torch.float64).index_add(0, self.ib, lump)

    def force(self, u):
        """-K u, [nglob][3]."""
        e = u.index_select(0, self.ib).reshape(self.E, self.n, self.n, self.n, 3)
        d = torch.stack([torch.einsum("il,ekjlc->ekjic", self.h, e), torch.einsum("jl,eklic->ekjic", self.h, e),
                         torch.einsum("kl,eljic->ekjic", self.h, e)], dim=-1)
        g = sum(d[..., r, None] * self.G[..., None, r, :] for r in range(3))  # du_c / dx_d
        lam = self.kappa - 2.0 / 3.0 * self.mu
        tr = g[..., 0, 0] + g[..., 1, 1] + g[..., 2, 2]
        sig = self.mu[..., None, None] * (g + g.transpose(-1, -2))
        sig = sig + (lam * tr)[..., None, None] * torch.eye(3, device="cuda", dtype=torch.float64)
        t = sum(sig[..., x, None] * self.G[..., None, :, x] for x in range(3)) * (self.w3 * self.det)[..., None, None]
        f = -(torch.einsum("li,ekjlc->ekjic", self.h, t[..., 0]) + torch.einsum("lj,eklic->ekjic", self.h, t[..., 1])
              + torch.einsum("lk,eljic->ekjic", self.h, t[..., 2]))
        return torch.zeros_like(u).index_add(0, self.ib, f.reshape(-1, 3))

    def step(self, u, v, a, drive, *material):
        if material:
            self.set_material(*material)
        dt = self.dt
        u = u + dt * v + 0.5 * dt * dt * a
        v = v + 0.5 * dt * a
        a = (self.force(u) + drive) * self.minv[:, None]
        return u, v + 0.5 * dt * a, a

    def run(self, m, state, steps, shot=0, record=True, material=None):
        """(seismograms [nrec][3][steps] or None, the final u, v, a)."""
        u, v, a = (f.double() for f in state)
        node, f = int(m["src"][shot]), torch.tensor(m["force"][shot], device="cuda", dtype=torch.float64)
        rec = torch.from_numpy(m["rec"]).cuda().long()
        seis = []
        for k in range(steps):
            q = (math.pi * F0 * ((k + 1) * self.dt - m["t0"])) ** 2
            drive = torch.zeros_like(u)
            drive[node] = f * ((1.0 - 2.0 * q) * math.exp(-q))
            if material is None:
                u, v, a = self.step(u, v, a, drive)
            else:
                u, v, a = checkpoint(self.step, u, v, a, drive, *material, use_reentrant=False)
            if record:
                seis.append(u.index_select(0, rec))
        return torch.stack(seis, dim=-1) if record else None, [u, v, a]


def exact_network(flat, x):
    """The network's output [batch][192][1000] for float64 parameters (a flat vector)."""
    p, o = [], 0
    for s in network_shapes():
        p.append(flat[o:o + math.prod(s)].reshape(s))
        o += math.prod(s)
    gelu = lambda z: torch.nn.functional.gelu(z, approximate="tanh")  # noqa: E731
    h = x
    for q in range(3):
        h = gelu(h @ p[2 * q].T + p[2 * q + 1])
    h = h.reshape(-1, C0, L0)
    for q, up in enumerate(UP):
        if up > 1:
            h = h.repeat_interleave(up, dim=2)
        W, b = p[6 + 2 * q], p[7 + 2 * q]
        pad = torch.nn.functional.pad(h, (1, 1))
        h = sum(torch.matmul(W[:, :, d], pad[:, :, d:d + h.shape[2]]) for d in range(3)) + b[:, None]
        if q + 1 < len(UP):
            h = gelu(h)
    return torch.einsum("bk,bkct->bct", x[:, IN - MOMENTS:], h.reshape(-1, MOMENTS, OUT_C, OUT_L))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sur_forward", "sur_gradient"):
        flat = torch.from_numpy(network_params(seed)).cuda().double()
        x, t = network_inputs(case["batch"], seed, kind == "sur_gradient")
        if kind == "sur_forward":
            y = torch.empty((case["batch"], OUT_C, OUT_L), device="cuda", dtype=torch.float64)
            for b in range(0, case["batch"], 128):
                y[b:b + 128] = exact_network(flat, x[b:b + 128].double())
            return y
        flat.requires_grad_(True)
        total, n = 0.0, t.numel()
        for b in range(0, case["batch"], 64):
            part = ((exact_network(flat, x[b:b + 64].double()) - t[b:b + 64].double()) ** 2).sum() / n
            part.backward()
            total += float(part.detach())
        return {"loss": total, "grads": flat.grad}
    if kind == "group":
        out = []
        for k, b in enumerate(group_models(case)):
            m = model_inputs(*b, seed + 1000 * k)
            X = Exact(m)
            X.set_material(*X.moduli(m))
            out.append(X.run(m, m["state"], case["steps"], record=False)[1])
        return out
    S = case.get("shots", 1)
    m = model_inputs(*box_of(case), seed, shots=S, state=kind != "gradient" and kind != "shots")
    X = Exact(m)
    rest = [torch.zeros((m["nglob"], 3), device="cuda")] * 3
    if kind == "gradient":
        mu = (m["rho"] * m["vs"] * m["vs"]).astype(np.float32)
        kappa = (m["rho"] * m["vp"] * m["vp"]).astype(np.float32) - np.float32(4.0 / 3.0) * mu
        mat = [torch.from_numpy(a).cuda().double().requires_grad_(True) for a in (m["rho"], kappa, mu)]
        seis, _ = X.run(m, rest, case["steps"], material=mat)
        (0.5 * ((seis - observed(len(m["rec"]), case["steps"], seed).double()) ** 2).sum()).backward()
        return {"seis": seis.detach(), "grad": [a.grad for a in mat]}
    X.set_material(*X.moduli(m))
    if kind == "stiffness":
        return X.force(m["state"][0].double())
    if S > 1:
        runs = [X.run(m, rest, case["steps"], shot=q) for q in range(S)]
        return {"seis": torch.stack([r[0] for r in runs]), "u": torch.stack([r[1][0] for r in runs])}
    seis, state = X.run(m, m["state"], case["steps"])
    return {"seis": seis, "state": state}
