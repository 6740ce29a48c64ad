"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one pass through the public entry points (binding.Lattice, binding.Batch and the
adjoint calls): a stretch of a coupled run with its read-back, one step of a loop that exchanges
positions with the host, a stretch of a batched ensemble, or a recorded run with its gradient.
Results are returned in the precision of the context that computed them (the calls hand out
doubles in every precision).

`exact` restates the coupled step in double with plain torch, without this package's code.
"""
import functools
import math

import torch
import torch.utils.checkpoint

from paper_2305_18919_gb300 import binding
from paper_2305_18919_gb300.inputs import ALPHA_CLASSES, LJ_XI, icosphere

DEV = "cuda"
STORE = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
SIZE = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
# a run on a lattice up to this size starts every pass from its initial fields and shape; a
# larger one continues where the last pass left it, as a long production run does
RESTART_NODES = 64 ** 3


def listed():
    return [
        # the 32^3 shear benchmark (a droplet in FP64, the parity configuration): small kernels
        dict(name="shear32_fp64", kind="run", flow="shear", precision="fp64", nx=32, ny=32, nz=32,
             tau=1.0, wall_u=0.01, radius=6.0, shape="droplet", abar=0.01, eps=0.0, steps=100),
        # the smallest coupled call: one step between setting and reading positions, as a caller
        # does that owns the particle's motion or logs every step
        dict(name="coupled24_fp32", kind="coupled", flow="wetting", precision="fp32", nx=24, ny=24,
             nz=20, tau=1.0, wall_u=0.0, radius=5.0, shape="softly_coated", abar=0.005, eps=0.005,
             steps=1),
        # the static-wetting benchmark: an ordinary production lattice
        dict(name="wetting128x128x96_fp32", kind="run", flow="wetting", precision="fp32", nx=128,
             ny=128, nz=96, tau=1.0, wall_u=0.0, radius=20.0, shape="softly_coated", abar=1e-4,
             eps=5e-5, steps=50),
        # the headline benchmark: large shear, FP32, and the same with 16-bit storage
        dict(name="shear256_fp32", kind="run", flow="shear", precision="fp32", nx=256, ny=256,
             nz=256, tau=0.8, wall_u=0.02, radius=40.0, shape="rigidly_coated", abar=0.02, eps=0.0,
             steps=40),
        dict(name="shear256_fp16", kind="run", flow="shear", precision="fp16", nx=256, ny=256,
             nz=256, tau=0.8, wall_u=0.02, radius=40.0, shape="rigidly_coated", abar=0.02, eps=0.0,
             steps=40),
        # a ragged lattice in the other 16-bit type
        dict(name="shear180x132x95_bf16", kind="run", flow="shear", precision="bf16", nx=180,
             ny=132, nz=95, tau=0.9, wall_u=0.02, radius=22.0, shape="rigidly_coated", abar=0.02,
             eps=0.0, steps=40),
        # a double-precision run beyond the smallest (reference runs for the other precisions)
        dict(name="shear128_fp64", kind="run", flow="shear", precision="fp64", nx=128, ny=128,
             nz=128, tau=0.8, wall_u=0.02, radius=24.0, shape="rigidly_coated", abar=0.02, eps=0.0,
             steps=20),
        # no particle: a channel driven by a body force, on odd sizes
        dict(name="channel132x100x77_fp32", kind="run", flow="channel", precision="fp32", nx=132,
             ny=100, nz=77, tau=0.9, wall_u=0.0, radius=0.0, shape="droplet", abar=0.0, eps=0.0,
             steps=50),
        # the ensemble benchmark: a parameter sweep over uneven wetting boxes, and a small sweep
        dict(name="ensemble96_fp32", kind="ensemble", precision="fp32", boxes=96, lo=48, hi=96,
             steps=30),
        dict(name="ensemble12_fp16", kind="ensemble", precision="fp16", boxes=12, lo=32, hi=64,
             steps=40),
        # the adjoint benchmark (FP32 forward, the reverse pass in double) and its FP64 check copy
        dict(name="adjoint64_fp32", kind="adjoint", flow="wetting", precision="fp32", nx=64, ny=64,
             nz=64, tau=1.0, wall_u=0.0, radius=12.0, shape="softly_coated", abar=0.01, eps=0.01,
             steps=60, every=30),
        dict(name="adjoint24_fp64", kind="adjoint", flow="wetting", precision="fp64", nx=24, ny=24,
             nz=24, tau=1.0, wall_u=0.0, radius=5.0, shape="softly_coated", abar=0.01, eps=0.01,
             steps=60, every=20),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["run"] * 5 + ["coupled", "ensemble", "adjoint", "adjoint"])
    if kind == "ensemble":
        lo = rng.choice([24, 32, 48])
        return dict(kind=kind, precision=rng.choice(["fp64", "fp32", "fp16", "bf16"]) if lo < 48
                    else "fp32", boxes=log_int(2, 64), lo=lo, hi=2 * lo, steps=2 * rng.randint(1, 5))
    precision = rng.choice(["fp64", "fp32", "fp32", "fp16", "bf16"])
    flow = rng.choice(["shear", "wetting", "channel"])
    hi = {"fp64": 128, "fp32": 224, "fp16": 224, "bf16": 224}[precision]
    if kind == "adjoint":
        precision, flow, hi = rng.choice(["fp64", "fp32"]), rng.choice(["shear", "wetting"]), 64
    if kind == "coupled":
        flow, hi = rng.choice(["shear", "wetting"]), 128
    edge = log_int(20, hi)  # the lattice's size, each axis near it
    nx, ny = (4 * max(5, int(edge * rng.uniform(0.8, 1.2) / 4)) for _ in range(2))
    nz = max(18, int(edge * rng.uniform(0.7, 1.1)))
    if kind == "adjoint":
        nx, ny, nz = min(nx, 64), min(ny, 64), min(nz, 64)
    c = dict(kind=kind, flow=flow, precision=precision, nx=nx, ny=ny, nz=nz,
             tau=round(rng.uniform(0.7, 1.1), 3),
             wall_u=round(rng.uniform(0.005, 0.02), 4) if flow == "shear" else 0.0,
             radius=0.0 if flow == "channel" else round(min(nx, ny, nz) * rng.uniform(0.15, 0.24), 2),
             shape=rng.choice(["softly_coated", "rigidly_coated"]),
             abar=round(rng.uniform(0.005, 0.02), 4), eps=0.0)
    if flow == "wetting":
        c["abar"] = round(c["abar"] * 0.1, 5)
        c["eps"] = round(c["abar"] * rng.uniform(0.1, 1.0), 6)
    if kind == "run":
        most = 4e6 if precision == "fp64" else 2e8  # node steps
        c["steps"] = int(max(4, min(100, most / (nx * ny * nz))))
    elif kind == "coupled":
        c["steps"] = 1
    else:
        c["steps"] = rng.randint(10, 40)
        c["every"] = rng.randint(5, 20)
    return c


# --- inputs --------------------------------------------------------------------------------


@functools.lru_cache(maxsize=None)
def unit_sphere(sub):
    v, f = icosphere(sub)
    return torch.from_numpy(v), f


def subdivisions(c):
    """Icosphere refinement by radius, as the benchmarks choose it (coarser in the ensemble)."""
    radius = c["radius"]
    if c.get("swept"):
        return 3 if radius < 16 else 4 if radius < 24 else 5
    return 2 if radius < 5.5 else 3 if radius < 9 else 4 if radius < 16 else 5 if radius < 32 else 6


def ensemble_boxes(c):
    """The boxes of a sweep: uneven lattices, particles and interface classes (fixed by the case;
    the seed moves and stretches the particles)."""
    g = torch.Generator().manual_seed(1000 * c["boxes"] + c["lo"])
    edges = [c["lo"] + k * ((c["hi"] - c["lo"]) // 12 * 4) for k in range(4)]
    out = []
    for _ in range(c["boxes"]):
        e = [edges[int(torch.randint(4, (1,), generator=g))] for _ in range(3)]
        r = [float(x) for x in torch.rand(3, generator=g, dtype=torch.float64)]
        abar = 0.005 + 0.015 * r[1]
        out.append(dict(kind="run", flow="wetting", precision=c["precision"], nx=e[0], ny=e[1],
                        nz=e[2], tau=1.0, wall_u=0.0, radius=0.3 * min(e), swept=True,
                        shape=("droplet", "softly_coated", "rigidly_coated")[int(3 * r[0])],
                        abar=0.1 * abar, eps=0.01 * abar * r[2], steps=c["steps"]))
    return out


def particle(c, seed):
    """Reference vertices, faces and current vertices (host, double): a sphere, moved and slightly
    stretched by the seed."""
    if not c["radius"]:
        return None
    r = (torch.rand(5, generator=torch.Generator().manual_seed(seed), dtype=torch.float64) - 0.5).tolist()
    v, f = unit_sphere(subdivisions(c))
    zc = 0.5 + c["radius"] + 2.0 ** (1.0 / 6.0) * LJ_XI if c["flow"] == "wetting" else (c["nz"] - 1) / 2 + r[2]
    centre = torch.tensor([c["nx"] / 2 + r[0], c["ny"] / 2 + r[1], zc], dtype=torch.float64)
    a = 1.0 + 0.04 * r[3]
    if c["flow"] == "wetting":  # the height over the wall stays
        s = torch.tensor([a, 1.0 / a, 1.0], dtype=torch.float64)
    else:
        s = torch.tensor([a, 1.0 + 0.04 * r[4], 0.0], dtype=torch.float64)
        s[2] = 1.0 / (s[0] * s[1])
    return (centre + c["radius"] * v), f, (centre + c["radius"] * v * s)


def flow_field(c, seed):
    """rho [nz][ny][nx] and u [nz][ny][nx][3] (double, on the GPU): the undisturbed flow and a weak
    smooth disturbance whose phases come from the seed."""
    p = (2 * math.pi * torch.rand(6, generator=torch.Generator().manual_seed(seed + 7), dtype=torch.float64)).tolist()
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    x, y = (2 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n for n in (nx, ny))
    zf = torch.arange(nz, dtype=torch.float64, device=DEV)
    z = math.pi * (zf - 0.5) / (nz - 2)
    x, y, z, zf = x[None, None, :], y[None, :, None], z[:, None, None], zf[:, None, None]
    env = torch.sin(z)
    u = torch.empty((nz, ny, nx, 3), dtype=torch.float64, device=DEV)
    a = 1e-3
    u[..., 0] = a * env * torch.sin(y + p[0]) * torch.cos(2 * z + p[1])
    u[..., 1] = a * env * torch.sin(x + p[2])
    u[..., 2] = a * env * torch.sin(x + p[3]) * torch.cos(y + p[4])
    if c["flow"] == "shear":
        u[..., 0] += c["wall_u"] * (2 * (zf - 0.5) / (nz - 2) - 1)
    rho = (1.0 + 1e-4 * torch.sin(x + p[5]) * torch.cos(y) * env).expand(nz, ny, nx).contiguous()
    return rho, u


def walls(c):
    """Wall velocities (bottom, top) and the body force."""
    g = 2e-6 if c["flow"] == "channel" else 0.0
    return (-c["wall_u"], 0.0, 0.0), (c["wall_u"], 0.0, 0.0), (g, 0.0, 0.0)


def alpha(c):
    return tuple(c["abar"] * a for a in ALPHA_CLASSES[c["shape"]])


def add_particle(lat, c, seed):
    p = particle(c, seed)
    if p is None:
        return None
    lat.add_mesh(p[0].numpy(), p[1])
    lat.set_interface(alpha(c), 1.0, c["eps"], LJ_XI, int(c["flow"] == "wetting"), 1)
    lat.set_vertices(p[2].numpy())
    return p[2]


def prepare(case, seed):
    if case["kind"] == "ensemble":
        boxes = ensemble_boxes(case)
        batch = binding.Batch([binding.lattice_desc(b["nx"], b["ny"], b["nz"], b["tau"],
                                                    precision=b["precision"]) for b in boxes])
        q0 = [add_particle(lat, b, seed + k) for k, (lat, b) in enumerate(zip(batch.contexts, boxes))]
        return dict(case=case, batch=batch, q0=torch.cat(q0), q=[torch.empty_like(q).numpy() for q in q0])
    ub, ut, g = walls(case)
    lat = binding.Lattice(case["nx"], case["ny"], case["nz"], case["tau"], 1.0, ub, ut, g,
                          case["precision"])
    q0 = add_particle(lat, case, seed)
    rho, u = (t.cpu().numpy() for t in flow_field(case, seed))
    lat.init_equilibrium(rho, u)
    s = dict(case=case, lat=lat, q0=None)
    if case["nx"] * case["ny"] * case["nz"] <= RESTART_NODES:
        s["rho"], s["u"] = rho, u
    if q0 is not None:
        s["q_host"] = q0.numpy()
        s["q0"] = q0.to(DEV)
        s["q"] = torch.empty_like(s["q0"])
        s["q_read"] = torch.empty_like(q0).pin_memory().numpy()
        if case["kind"] == "adjoint":
            s["dJdq"] = observable(s["q_host"].shape[0], seed).numpy()
    return s


def observable(nv, seed):
    """dJ/dq of a smooth linear observable of the vertices."""
    k = torch.arange(nv, dtype=torch.float64)[:, None]
    p = torch.rand((1, 3), generator=torch.Generator().manual_seed(seed + 13), dtype=torch.float64)
    return torch.sin(0.37 * k + 2 * math.pi * p) / nv


# --- one pass ------------------------------------------------------------------------------


def moved(lat, q, q0, dtype):
    lat.vertices_device(q.data_ptr())
    return (q - q0).to(dtype)


def run(state):
    c = state["case"]
    dtype = STORE[c["precision"]]
    if c["kind"] == "ensemble":
        batch = state["batch"]
        batch.step(c["steps"])
        # each box has a stream of its own: its results are read through host buffers
        for lat, q in zip(batch.contexts, state["q"]):
            lat.vertices(q)
        rho, u = (torch.from_numpy(a) for a in batch.contexts[0].fields())
        q = torch.cat([torch.from_numpy(a) for a in state["q"]])
        return [(q - state["q0"]).to(dtype), rho.to(dtype), u.to(dtype)]
    lat = state["lat"]
    if c["kind"] == "coupled":
        lat.set_vertices(state["q_host"])
        lat.step_async(1)
        lat.vertices(state["q_read"])
        return [torch.from_numpy(state["q_read"] - state["q_host"]).to(dtype)]
    if "rho" in state:
        lat.init_equilibrium(state["rho"], state["u"])
        if state["q0"] is not None:
            lat.set_vertices(state["q_host"])
    if c["kind"] == "adjoint":
        lat.adjoint_record(c["steps"], c["every"])
        d = moved(lat, state["q"], state["q0"], dtype)
        return [d, torch.from_numpy(lat.adjoint_gradient(state["dJdq"])).to(dtype)]
    lat.step(c["steps"])
    rho, u = lat.fields_device()
    out = [rho.to(dtype), u.to(dtype)]
    if state["q0"] is not None:
        out.append(moved(lat, state["q"], state["q0"], dtype))
    return out


def work(case):
    """Populations read and written once per step (a step's lattice streams through the caches),
    the fields and positions handed out; a gradient also recomputes the run and reads two states
    and reads and writes the adjoint populations (double) per step."""
    boxes = ensemble_boxes(case) if case["kind"] == "ensemble" else [case]
    size = SIZE[case["precision"]]
    nodes = sum(b["nx"] * b["ny"] * (b["nz"] - 2) for b in boxes)
    nv = sum(10 * 4 ** subdivisions(b) + 2 for b in boxes if b["radius"])
    step_bytes, step_flops = 2 * 19 * size * nodes + 48 * nv, 250 * nodes + 2500 * nv
    if case["kind"] == "adjoint":
        step_bytes = 2 * step_bytes + (2 * 19 * size + 2 * 19 * 8) * nodes
        step_flops = 2 * step_flops + 500 * nodes + 8000 * nv
    shown = {"run": nodes, "ensemble": boxes[0]["nx"] * boxes[0]["ny"] * boxes[0]["nz"]}.get(case["kind"], 0)
    return {"bytes": case["steps"] * step_bytes + 4 * size * shown + 3 * size * nv,
            "flops": case["steps"] * step_flops}


# --- the same in double, with plain torch --------------------------------------------------

C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
     (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
     (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def along(c, v):
    """c . v for a lattice direction c and a vector field v [3][...]."""
    terms = [v[k] if c[k] > 0 else -v[k] for k in range(3) if c[k]]
    return sum(terms[1:], terms[0]) if terms else 0.0


def moments(f, F):
    """rho - 1 and u of populations' deviations f [19][...] with the force density F [3][...]."""
    d = f.sum(0)
    j = [sum(C[i][k] * f[i] for i in range(19) if C[i][k]) for k in range(3)]
    return d, [(j[k] + 0.5 * F[k]) / (1.0 + d) for k in range(3)]


def collide(f, F, tau):
    d, u = moments(f, F)
    uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
    out = []
    for i in range(19):
        cu, cF = along(C[i], u), along(C[i], F)
        feq = W[i] * (d + (1.0 + d) * (3 * cu + 4.5 * cu * cu - 1.5 * uu))
        src = W[i] * (1 - 0.5 / tau) * (3 * (cF - uF) + 9 * cu * cF)
        out.append(f[i] + (feq - f[i]) / tau + src)
    return out


def stream(fp, ub, ut):
    """Post-streaming deviations [19][nz][ny][nx] of post-collision ones, half-way bounce-back."""
    nz = fp[0].shape[0]
    out = []
    for i, c in enumerate(C):
        o = 0 if i == 0 else i + 1 if i % 2 else i - 1
        g = torch.roll(fp[i], (c[2], c[1], c[0]), (0, 1, 2))
        if c[2] > 0:
            wall = 6 * W[i] * sum(c[k] * ub[k] for k in range(3))
            g = torch.cat([g[:1], fp[o][1:2] + wall, g[2:]])
        elif c[2] < 0:
            wall = 6 * W[i] * sum(c[k] * ut[k] for k in range(3))
            g = torch.cat([g[:nz - 2], fp[o][nz - 2:nz - 1] + wall, g[nz - 1:]])
        out.append(g)
    return torch.stack(out)


def phi4(r):
    a = r.abs()
    near = (3 - 2 * a + torch.sqrt((1 + 4 * a - 4 * a * a).clamp(min=1e-300))) / 8
    far = (5 - 2 * a - torch.sqrt((-7 + 12 * a - 4 * a * a).clamp(min=1e-300))) / 8
    return torch.where(a <= 1, near, torch.where(a <= 2, far, torch.zeros_like(a)))


def stencil(q, shape):
    """Node indices [nv][64], weights [nv][64] and z layers of the delta stencils; nodes beyond the
    lattice have weight 0."""
    nz, ny, nx = shape
    base = torch.floor(q.detach()).long() - 1
    d = torch.arange(4, device=q.device)
    node = [base[:, k:k + 1] + d for k in range(3)]
    w = [phi4(node[k].double() - q[:, k:k + 1]) for k in range(3)]
    z = node[2]
    w[2] = torch.where((z >= 0) & (z < nz), w[2], torch.zeros_like(w[2]))
    z = z.clamp(0, nz - 1)
    idx = (z[:, :, None, None] * ny + (node[1] % ny)[:, None, :, None]) * nx + (node[0] % nx)[:, None, None, :]
    wt = w[2][:, :, None, None] * w[1][:, None, :, None] * w[0][:, None, None, :]
    zz = z[:, :, None, None].expand(wt.shape)
    return idx.reshape(len(q), 64), wt.reshape(len(q), 64), zz.reshape(len(q), 64)


def nodal_forces(q, ref, faces, theta, wall, nz):
    """Strain energy, volume penalty and wall forces of the interface, [nv][3]; theta = alpha1,
    alpha2, alpha3, eps."""
    x, X = q[faces], ref[faces]
    a, b, A, B = x[:, 1] - x[:, 0], x[:, 2] - x[:, 0], X[:, 1] - X[:, 0], X[:, 2] - X[:, 0]

    def dot(p, r):
        return (p * r).sum(1, keepdim=True)

    G11, G12, G22 = dot(a, a), dot(a, b), dot(b, b)
    g11, g12, g22 = dot(A, A), dot(A, B), dot(B, B)
    det, det0 = G11 * G22 - G12 * G12, g11 * g22 - g12 * g12
    A0 = 0.5 * torch.sqrt(det0)
    dI = A0 * 0.5 * theta[2]
    dL = A0 * (0.5 * (theta[0] - theta[2]) + 0.25 * (theta[0] + theta[1]) * torch.log(det / det0))
    Ea = dI * 2 * (g22 * a - g12 * b) / det0 + dL * 2 * (G22 * a - G12 * b) / det
    Eb = dI * 2 * (g11 * b - g12 * a) / det0 + dL * 2 * (G11 * b - G12 * a) / det
    f = torch.stack([Ea + Eb, -Ea, -Eb], 1)
    if wall:
        fz = 0.0
        gz = x[:, :, 2].mean(1)
        for zw in (0.5, nz - 1.5):
            dz = gz - zw
            s6 = (LJ_XI / dz) ** 6
            fz = fz + 48 * theta[3] * (s6 * s6 - 0.5 * s6) / dz
        f = f + torch.stack([torch.zeros_like(fz), torch.zeros_like(fz), fz / 3], 1)[:, None, :]
    m = ref.mean(0)

    def volume(y):
        y = y - m
        return (y[:, 0] * torch.linalg.cross(y[:, 1], y[:, 2])).sum() / 6

    coef = (volume(x) - volume(X)) / volume(X)
    n = torch.linalg.cross(a, b) / 6  # the volume gradient's share of each corner (closed surface)
    f = f - coef * n[:, None, :]
    return torch.zeros_like(q).index_add(0, faces.reshape(-1), f.reshape(-1, 3))


def step(f, q, theta, c, ref, faces):
    """One coupled step; returns f, q and the step's force density."""
    nz, ny, nx = f.shape[1:]
    ub, ut, g = walls(c)
    if q is None:
        F = [torch.full(f.shape[1:], g[k], dtype=f.dtype, device=f.device) for k in range(3)]
        return stream(collide(f, F, c["tau"]), ub, ut), None, F
    phi = nodal_forces(q, ref, faces, theta, c["flow"] == "wetting", nz)
    idx, w, zz = stencil(q, (nz, ny, nx))
    ws = torch.where((zz == 0) | (zz == nz - 1), torch.zeros_like(w), w)
    F = torch.zeros((nz * ny * nx, 3), dtype=f.dtype, device=f.device).index_add(
        0, idx.reshape(-1), (ws[:, :, None] * phi[:, None, :]).reshape(-1, 3))
    F = [F[:, k].reshape(nz, ny, nx) + g[k] for k in range(3)]
    f = stream(collide(f, F, c["tau"]), ub, ut)
    u = torch.stack(with_walls(moments(f, F)[1], ub, ut), -1).reshape(-1, 3)
    return f, q + (w[:, :, None] * u[idx]).sum(1), F


def with_walls(u, ub, ut):
    return [torch.cat([torch.full_like(u[k][:1], ub[k]), u[k][1:-1], torch.full_like(u[k][:1], ut[k])])
            for k in range(3)]


def simulate(c, seed, rest=False):
    """rho, u and the vertices after the case's steps."""
    ub, ut, _ = walls(c)
    p = particle(c, seed)
    if rest:
        f = torch.zeros((19, c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device=DEV)
    else:
        rho, u = flow_field(c, seed)
        f = at_equilibrium(rho, u)
    theta = torch.tensor(alpha(c) + (c["eps"],), dtype=torch.float64, device=DEV)
    q = ref = faces = None
    if p is not None:
        ref, faces, q = p[0].to(DEV), torch.from_numpy(p[1]).long().to(DEV), p[2].to(DEV)
    for _ in range(c["steps"]):
        f, q, F = step(f, q, theta, c, ref, faces)
    d, u = moments(f, F)
    d = torch.cat([torch.zeros_like(d[:1]), d[1:-1], torch.zeros_like(d[:1])])
    return 1.0 + d, torch.stack(with_walls(u, ub, ut), -1), q if q is None else q - p[2].to(DEV)


def at_equilibrium(rho, u):
    u = [u[..., k] for k in range(3)]
    uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    f = []
    for i in range(19):
        cu = along(C[i], u)
        f.append(W[i] * ((rho - 1.0) + rho * (3 * cu + 4.5 * cu * cu - 1.5 * uu)))
    return torch.stack(f)


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] == "ensemble":
            got = [simulate(b, seed + k, rest=True) for k, b in enumerate(ensemble_boxes(case))]
            return [torch.cat([g[2] for g in got]), got[0][0], got[0][1]]
        if case["kind"] == "coupled":
            return [simulate(case, seed)[2]]
        if case["kind"] == "run":
            rho, u, d = simulate(case, seed)
            return [rho, u] + ([] if d is None else [d])
    # the gradient, by reverse-mode differentiation of the whole run, one step at a time
    p = particle(case, seed)
    ref, faces, q0 = p[0].to(DEV), torch.from_numpy(p[1]).long().to(DEV), p[2].to(DEV)
    theta = torch.tensor(alpha(case) + (case["eps"],), dtype=torch.float64, device=DEV, requires_grad=True)
    f, q = at_equilibrium(*flow_field(case, seed)), q0

    def advance(f, q, theta):
        return step(f, q, theta, case, ref, faces)[:2]

    for _ in range(case["steps"]):
        f, q = torch.utils.checkpoint.checkpoint(advance, f, q, theta, use_reentrant=False)
    J = (q * observable(len(q0), seed).to(DEV)).sum()
    return [(q - q0).detach(), torch.autograd.grad(J, theta)[0]]
