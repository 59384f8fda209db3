"""What this framework is used for, as timed cases.

Each case goes through the package's public entry points only: a `Lattice`
with particles that settle, touch, are held or are moved by the caller, a
`Batch` of drag boxes, the drag gradient `AdjointDrag`, a particle-free
channel.  Box sizes, shapes, contact constants and step counts are those of
`workloads.py`, the tests and the benchmark, and odd ones around them.

`Reference` below is an independent FP64 transcription of the method for
particles that do not touch (node classification, refilling, streaming with
walls and interpolated bounce-back, collision, momentum exchange, rigid
motion), vectorised over nodes and links; `exact` returns its values.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2206_11634_gb300 as pkg
from paper_2206_11634_gb300 import adjoint as adj
from paper_2206_11634_gb300 import workloads as wl

DEVICE = "cuda"
CONTACT = dict(kn=2000.0, eta_n=20.0, kt=1000.0, eta_t=10.0, mu_s=0.3, c_tol=1e-6)


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _settle(name, nx, ny, nz, storage, particles, steps, *, lattice=19, px=0, py=0, pz=0, ncp_lo=2, ncp_hi=8,
            spread=3.0, r_lo=5.0, r_hi=8.0, rs=0.5, density=1200.0 / 927.0, gravity=-1e-3, tau=0.8, n_sub=100, dem=0,
            floor=0):
    return dict(name=name, kind="settle", nx=nx, ny=ny, nz=nz, storage=storage, particles=particles, steps=steps,
                lattice=lattice, px=px, py=py, pz=pz, ncp_lo=ncp_lo, ncp_hi=ncp_hi, spread=spread, r_lo=r_lo,
                r_hi=r_hi, rs=rs, density=density, gravity=gravity, tau=tau, n_sub=n_sub, dem=dem, floor=floor)


def listed():
    return [
        # The smallest run: one sphere settling in a small walled FP64 box
        # (the paper's §3.1 geometry), a few coupled steps between read-outs.
        _settle("sphere_f64", 32, 32, 48, "f64", 1, 4, ncp_lo=1, ncp_hi=1, spread=0.0, r_lo=6.0, r_hi=6.0, rs=0.0,
                density=2.5, gravity=-1e-4),
        # One four-control-point metaball settling in a walled box, FP32 with
        # the FP64 rigid-body integrator: the paper's §3.2 run.
        _settle("metaball_f32", 128, 128, 256, "f32", 1, 8, ncp_lo=4, ncp_hi=4, spread=4.0, r_lo=7.0, r_hi=9.0,
                density=1134.156 / 970.0, gravity=-8e-4),
        # Two metaballs settling in the paper's §4 box, whose 150 nodes are no
        # multiple of anything, with 16-bit storage.
        _settle("pair_f16", 150, 150, 250, "f16", 2, 8, ncp_lo=4, ncp_hi=4, spread=2.2, r_lo=7.0, r_hi=7.3, rs=0.1,
                gravity=-3.92e-4, tau=0.56),
        # 200 metaballs settling, the benchmark's box; nothing touches yet.
        _settle("suspension_f32", 256, 256, 256, "f32", 200, 6, px=1, py=1),
        # The same kind of run once the lowest particles have reached the
        # floor: 16 on it, 34 above, so the contact groups are what the rigid
        # bodies wait for.  A pass goes on where the last one ended.
        _settle("floor_f32", 128, 128, 256, "f32", 50, 4, px=1, py=1, floor=16),
        # The drag on one held metaball in a small periodic box, many steps
        # per read-out: a step is short, so launches and gaps count.
        dict(name="drag_f32", kind="drag", n=48, storage="f32", steps=96, lattice=19),
        # 64 boxes of drag cases of different sides stepped together, in
        # both storages that such sweeps are run in.
        dict(name="batch_f32", kind="batch", boxes=64, lo=48, hi=128, storage="f32", steps=32, sizes=2211),
        dict(name="batch_f16", kind="batch", boxes=64, lo=48, hi=128, storage="f16", steps=32, sizes=2211),
        # One step of a shape optimisation: the drag and its gradient by the
        # discrete adjoint, at the full size and at the tests' small one.
        dict(name="gradient", kind="gradient", n=96, ncp=6, T=500, W=100),
        dict(name="gradient_small", kind="gradient", n=32, ncp=3, T=80, W=20),
        # A body-force-driven channel without particles: the bare sweep, and
        # the fields written out.
        dict(name="channel_f32", kind="channel", nx=256, ny=256, nz=256, storage="f32", lattice=19, steps=8),
        # Particles moved by the caller (another code owns their motion):
        # restart from stored populations, new poses before every step, loads
        # read after it, populations stored again.  D3Q15, the exact link
        # fraction, and box sides that are no multiples of the tiles.
        dict(name="driven_d3q15", kind="driven", nx=201, ny=157, nz=99, storage="f32", lattice=15, particles=12,
             steps=3, q_exact=1),
    ]


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["settle", "settle", "settle", "floor", "drag", "batch", "gradient", "channel", "driven"])
    if kind == "settle":
        storage = rng.choice(["f64", "f32", "f32", "f16", "bf16"])
        top = 72 if storage == "f64" else 256
        nx, ny, nz = (_log_int(rng, 36, top) for _ in range(3))
        room = max(1, int(nx * ny * (nz - 28) / 60000)) if min(nx, ny) > 60 and nz > 60 else 1
        many = min(200, _log_int(rng, 1, room)) if room > 1 else 1
        r = 5.0 if storage == "f64" or min(nx, ny, nz) < 60 else rng.uniform(5.0, 7.0)
        per = rng.choice([0, 1])
        return _unnamed(_settle("", nx, ny, nz, storage, many, rng.randint(2, 8), px=per, py=per,
                                lattice=rng.choice([19, 19, 15]), ncp_hi=rng.randint(2, 8), spread=2.0, r_lo=r,
                                r_hi=r + 1.0, dem=0 if storage == "f64" else rng.choice([0, 0, 1]),
                                tau=rng.choice([0.6, 0.8, 1.0])))
    if kind == "floor":
        nx, ny, nz = _log_int(rng, 96, 200), _log_int(rng, 96, 200), _log_int(rng, 128, 256)
        low = max(2, int(nx * ny / 1500))
        return _unnamed(_settle("", nx, ny, nz, rng.choice(["f32", "f16"]), low + rng.randint(0, 20),
                                rng.randint(2, 4), px=1, py=1, floor=low))
    if kind == "drag":
        return dict(kind="drag", n=_log_int(rng, 40, 160), storage=rng.choice(["f32", "f16", "bf16"]),
                    steps=_log_int(rng, 32, 128), lattice=rng.choice([19, 19, 15]))
    if kind == "batch":
        return dict(kind="batch", boxes=_log_int(rng, 3, 64), lo=40, hi=rng.randint(64, 128),
                    storage=rng.choice(["f32", "f16", "bf16"]), steps=rng.randint(17, 32), sizes=rng.randint(1, 9999))
    if kind == "gradient":
        return dict(kind="gradient", n=_log_int(rng, 30, 96), ncp=rng.randint(1, 6), T=_log_int(rng, 40, 300),
                    W=rng.randint(10, 40))
    if kind == "channel":
        return dict(kind="channel", nx=_log_int(rng, 40, 256), ny=_log_int(rng, 40, 256), nz=_log_int(rng, 40, 256),
                    storage=rng.choice(["f64", "f32", "f16", "bf16"]), lattice=rng.choice([19, 19, 15]),
                    steps=rng.randint(2, 8))
    return dict(kind="driven", nx=_log_int(rng, 64, 220), ny=_log_int(rng, 64, 220), nz=_log_int(rng, 64, 220),
                storage=rng.choice(["f64", "f32", "f16"]), lattice=rng.choice([15, 19]), particles=rng.randint(1, 4),
                steps=rng.randint(1, 4), q_exact=rng.choice([0, 1]))


# --------------------------------------------------------------------------
# inputs, from the seed alone
# --------------------------------------------------------------------------
_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}


def _lattice_vectors(Q):
    """Directions and weights in the package's order (opposites adjacent)."""
    if Q == 19:
        half = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
        w = {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
    else:
        half = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)]
        w = {0: 2 / 9, 1: 1 / 9, 3: 1 / 72}
    e = [(0, 0, 0)]
    for v in half:
        e += [v, tuple(-c for c in v)]
    return e, [w[sum(abs(c) for c in v)] for v in e]


def _flow(Q, shape, seed, amp=0.01):
    """Populations f[i][z][y][x] in FP64 of a smooth flow: a mean drift and a
    few long waves of velocity and density, in equilibrium."""
    g = np.random.default_rng([seed, 77])
    nz, ny, nx = shape
    dev = torch.device(DEVICE)
    ax = [torch.arange(n, dtype=torch.float64, device=dev) * (2 * math.pi / n) for n in (nx, ny, nz)]
    fields = []
    for a in range(4):  # u_x, u_y, u_z, density
        v = torch.full((nz, ny, nx), 0.3 * amp * float(g.uniform(-1, 1)) if a < 3 else 1.0, dtype=torch.float64,
                       device=dev)
        for _ in range(2):
            k = g.integers(1, 3, 3)
            ph = g.uniform(0, 2 * math.pi, 3)
            s = amp * float(g.uniform(0.3, 0.6)) * (1.0 if a < 3 else 0.1)
            v += s * torch.sin(k[2] * ax[2] + ph[2])[:, None, None] * torch.sin(k[1] * ax[1] + ph[1])[None, :, None] \
                * torch.sin(k[0] * ax[0] + ph[0])[None, None, :]
        fields.append(v)
    ux, uy, uz, rho = fields
    e, w = _lattice_vectors(Q)
    f = torch.empty((Q, nz, ny, nx), dtype=torch.float64, device=dev)
    uu = 1.0 - 1.5 * (ux * ux + uy * uy + uz * uz)
    for i in range(Q):
        eu = e[i][0] * ux + e[i][1] * uy + e[i][2] * uz
        f[i] = w[i] * rho * (uu + 3.0 * eu + 4.5 * eu * eu)
    return f


def _unit_quaternion(g):
    q = g.normal(size=4)
    return q / np.linalg.norm(q)


def _lowest(cp, K, q):
    """Height of the lowest point of the surface {M = 1} below the particle's
    reference point, to about 0.01, by sampling."""
    R = _rotation(q)
    c = cp @ R.T
    b = wl.bounding_radius(cp, K)
    dev = torch.device(DEVICE)
    xy = torch.arange(-b, b, 0.4, device=dev, dtype=torch.float32)
    z = torch.arange(-b, 0.0, 0.02, device=dev, dtype=torch.float32)
    M = torch.zeros((len(z), len(xy), len(xy)), device=dev)
    for k in range(len(K)):
        M += float(K[k]) / ((z[:, None, None] - float(c[k, 2])) ** 2 + (xy[None, :, None] - float(c[k, 1])) ** 2
                            + (xy[None, None, :] - float(c[k, 0])) ** 2 + 1e-9)
    hit = (M >= 1.0).flatten(1).any(1)
    return float(z[int(hit.to(torch.int32).argmax())])


def _particles_of(case, seed):
    """Metaballs placed by rejection with bounding spheres two nodes apart;
    the first `floor` of them touch the floor lightly."""
    g = np.random.default_rng([seed, 5])
    n = np.array([case["nx"], case["ny"], case["nz"]], dtype=float)
    per = np.array([case["px"], case["py"], case["pz"]])
    out, centres, radii = [], [], []
    r_lo, r_hi, spread = case["r_lo"], case["r_hi"], case["spread"]
    tries = 0
    while len(out) < case["particles"]:
        tries += 1
        if tries > 20000:
            raise RuntimeError("could not place the particles")
        ncp = int(g.integers(case["ncp_lo"], case["ncp_hi"] + 1))
        cp, K = wl.nominal_radius_metaball(g, ncp, spread, g.uniform(r_lo, r_hi))
        q = _unit_quaternion(g)
        b = wl.bounding_radius(cp, K, case["rs"])
        low = len(out) < case["floor"]
        lo = np.where(per == 1, 0.0, b + 1.5)
        hi = np.where(per == 1, n, n - 2.5 - b)
        if case["floor"] and not low:
            lo[2] = 32.0 + b
        if np.any(hi < lo):
            lo, hi = np.minimum(lo, n / 2 - 0.5), np.maximum(hi, n / 2 - 0.5)
        x = g.uniform(lo, hi)
        if low:
            x[2] = b  # set below, once the place is taken
        if centres:
            d = np.array(centres) - x
            d -= per * n * np.round(d / n)
            gap = 0.2 if low else 2.0
            if np.any(np.linalg.norm(d, axis=1) < np.array(radii) + b + gap):
                continue
        centres.append(x.copy())
        radii.append(b)
        if low:  # the skin between 0.04 nodes inside the plane and 0.2 above it
            x[2] = -0.5 - _lowest(cp, K, q) + case["rs"] + g.uniform(-0.04, 0.2)
        v = np.zeros(3) if low else g.uniform(-0.005, 0.005, 3)
        out.append(dict(cp=cp, K=K, x=x, q=q, v=v, w=g.uniform(-0.002, 0.002, 3) * (0.0 if low else 1.0), fixed=0,
                        Rs=case["rs"], density=case["density"], mass=0.0, inertia=None))
    return out


def _make(p):
    return pkg.make_particle(p["cp"], p["K"], p["x"], q=p["q"], v=p["v"], w=p["w"], Rs=p["Rs"], density=p["density"],
                             mass=p["mass"], inertia=p["inertia"], fixed=p["fixed"])


def _held(g, n, ncp, spread, R, ctr):
    cp, K = wl.nominal_radius_metaball(g, ncp, spread, R)
    return dict(cp=cp, K=K, x=np.asarray(ctr, dtype=float), q=_unit_quaternion(g), v=np.zeros(3), w=np.zeros(3),
                fixed=1, Rs=0.0, density=1.0, mass=1.0, inertia=np.eye(3))


def _drag_inputs(case, seed):
    g = np.random.default_rng([seed, 6])
    n = case["n"]
    c = n / 2.0 - 0.5 + g.uniform(-0.3, 0.3, 3)
    return _held(g, n, 4, 2.5 * n / 48.0, n / 8.0, c)


def _batch_inputs(case, seed):
    sizes = np.random.default_rng(case["sizes"]).integers(case["lo"], case["hi"] + 1, case["boxes"])
    g = np.random.default_rng([seed, 7])
    boxes = []
    for n in (int(v) for v in sizes):
        p = _held(g, n, int(g.integers(1, 7)), 0.075 * n, 0.12 * n, n / 2.0 - 0.5 + g.uniform(-0.5, 0.5, 3))
        boxes.append((n, 2e-6 * (48.0 / n) ** 2, p))
    return boxes


def _gradient_inputs(case, seed):
    g = np.random.default_rng([seed, 8])
    n = case["n"]
    R = n / 9.6
    cp, K = wl.nominal_radius_metaball(g, case["ncp"], 0.06 * n, R)
    c = np.full(3, n / 2.0 - 0.5) + g.uniform(-0.3, 0.3, 3)
    # parameters as a torch program holds them
    cp = torch.tensor(cp + c, dtype=torch.float32)
    K = torch.tensor(K, dtype=torch.float32)
    force = 2.0 * 6.0 * math.pi * 0.1 * R * 0.02 / float(n) ** 3
    return cp, K, c, (force, 0.0, 0.0), (0.02, 0.0, 0.0)


def _driven_inputs(case, seed):
    c = dict(case, px=1, py=1, pz=0, ncp_lo=1, ncp_hi=6, spread=2.5, r_lo=5.0, r_hi=8.0, rs=0.0, density=1.2, floor=0)
    g = np.random.default_rng([seed, 9])
    poses = []
    parts = _particles_of(c, seed)
    for p in parts:
        p.update(mass=50.0, inertia=np.eye(3) * 500.0, fixed=1, v=g.uniform(-0.03, 0.03, 3),
                 w=g.uniform(-0.003, 0.003, 3))
    for k in range(case["steps"]):
        poses.append([dict(p, x=p["x"] + k * p["v"]) for p in parts])
    return poses


# --------------------------------------------------------------------------
# prepare and run
# --------------------------------------------------------------------------
def _working(case, x):
    """A result in the precision its lattice computes in: FP64 lattices give
    FP64, the others FP32 (as such a run is stored or plotted)."""
    if case["storage"] == "f64":
        return x
    return x.astype(np.float32) if isinstance(x, np.ndarray) else x.float()


_STATE = np.dtype(pkg.LbmParticle)


def prepare(case, seed):
    kind = case["kind"]
    torch.cuda.set_device(0)
    if kind == "settle":
        lat = pkg.Lattice(case["nx"], case["ny"], case["nz"], storage=case["storage"], lattice=case["lattice"],
                          periodic=(case["px"], case["py"], case["pz"]), n_sub=case["n_sub"], tau=case["tau"],
                          gravity=(0.0, 0.0, case["gravity"]), max_particles=case["particles"], dem_mode=case["dem"],
                          **CONTACT)
        lat.set_populations(_flow(lat.Q, lat.shape, seed))
        lat.set_particles([_make(p) for p in _particles_of(case, seed)])
        # the states with their mass properties, as the library returns them
        arr = (pkg.LbmParticle * case["particles"])()
        lat._ok(lat.L.lbm_get_forces(lat.h, None, None, arr), lat.h)
        return dict(case=case, lat=lat, particles=arr, out=(pkg.LbmParticle * case["particles"])())
    if kind == "drag":
        n = case["n"]
        lat = pkg.Lattice(n, n, n, storage=case["storage"], lattice=case["lattice"], periodic=(1, 1, 1), tau=0.8,
                          force=(2e-6 * (48.0 / n) ** 2, 0.0, 0.0), max_particles=1)
        lat.set_populations(_flow(lat.Q, lat.shape, seed, 1e-3))
        lat.set_particles([_make(_drag_inputs(case, seed))])
        return dict(case=case, lat=lat)
    if kind == "batch":
        boxes = _batch_inputs(case, seed)
        bt = pkg.Batch([dict(nx=n, ny=n, nz=n, storage=case["storage"], lattice=19, periodic=(1, 1, 1), tau=0.8,
                             force=(force, 0.0, 0.0), n_sub=0, max_particles=1) for n, force, _ in boxes])
        for c, (_, _, p) in enumerate(boxes):
            bt.set_particles(c, [_make(p)])
        return dict(case=case, batch=bt)
    if kind == "gradient":
        cp, K, c, force, u0 = _gradient_inputs(case, seed)
        shape = pkg.make_particle(cp.numpy().astype(np.float64) - c, K.numpy().astype(np.float64), c, fixed=1,
                                  mass=1.0, inertia=np.eye(3))
        drag = adj.AdjointDrag(case["n"], case["n"], case["n"], particle=shape, T=case["T"], W=case["W"], tau=0.8,
                               u0=u0, force=force)
        return dict(case=case, drag=drag, cp=cp, K=K)
    if kind == "channel":
        lat = pkg.Lattice(case["nx"], case["ny"], case["nz"], storage=case["storage"], lattice=case["lattice"],
                          periodic=(1, 1, 0), tau=0.8, force=(1e-6, 0.0, 0.0))
        lat.set_populations(_flow(lat.Q, lat.shape, seed))
        return dict(case=case, lat=lat)
    lat = pkg.Lattice(case["nx"], case["ny"], case["nz"], storage=case["storage"], lattice=case["lattice"],
                      periodic=(1, 1, 0), tau=0.8, max_particles=case["particles"], q_exact=case["q_exact"])
    return dict(case=case, lat=lat, f=_flow(lat.Q, lat.shape, seed),
                poses=[[_make(p) for p in pose] for pose in _driven_inputs(case, seed)])


def _fields(case, lat):
    rho, u, flags = lat.fields()
    return dict(rho=_working(case, rho), u=_working(case, u), flags=flags.view(torch.int16))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "settle":
        # the particles start from their given states (a run on the floor goes
        # on), move freely for a few coupled steps, then loads, states and
        # fields are read out
        lat, n = state["lat"], case["particles"]
        if not case["floor"]:
            lat._ok(lat.L.lbm_set_particles(lat.h, state["particles"], n), lat.h)
            lat.np = n
        lat.step(case["steps"])
        F, T = lat.forces()
        lat._ok(lat.L.lbm_get_forces(lat.h, None, None, state["out"]), lat.h)
        s = np.frombuffer(state["out"], dtype=_STATE)
        out = _fields(case, lat)
        out.update({k: _working(case, v.copy()) for k, v in
                    dict(F=F, T=T, x=s["x"], v=s["v"], q=s["q"], w=s["w"]).items()})
        return out
    if kind == "drag":
        lat = state["lat"]
        lat.step(case["steps"])
        F, T = lat.forces()
        return dict(_fields(case, lat), F=_working(case, F), T=_working(case, T))
    if kind == "batch":
        bt = state["batch"]
        bt.step(case["steps"])
        F, T = bt.all_forces()
        return dict(F=_working(case, F), T=_working(case, T), first=_working(case, bt.populations(0)),
                    last=_working(case, bt.populations(bt.n - 1)))
    if kind == "gradient":
        cp = state["cp"].clone().requires_grad_(True)
        K = state["K"].clone().requires_grad_(True)
        J = state["drag"](cp, K)
        J.backward()
        return dict(J=J.detach().to(cp.dtype), cp=cp.grad, K=K.grad)
    lat = state["lat"]
    if kind == "channel":
        lat.step(case["steps"])
        return _fields(case, lat)
    lat.set_populations(state["f"])
    loads = []
    for pose in state["poses"]:
        lat.set_particles(pose)
        lat.step(1)
        loads.append(np.concatenate(lat.forces(), axis=1))
    return dict(loads=_working(case, np.array(loads)), f=_working(case, lat.populations()))


def work(case):
    """Every population read and written once a step, every result written
    once (fields of FP64 as the library writes them); about 250 operations per
    node and step, the rigid bodies' sub-steps beside them."""
    kind = case["kind"]
    if kind == "batch":
        sizes = np.random.default_rng(case["sizes"]).integers(case["lo"], case["hi"] + 1, case["boxes"])
        N = int((sizes.astype(np.int64) ** 3).sum())
        sides = int(sizes[0]) ** 3 + int(sizes[-1]) ** 3
        return dict(bytes=float(38 * _BYTES[case["storage"]] * N * case["steps"] + 19 * 8 * sides),
                    flops=250.0 * N * case["steps"])
    if kind == "gradient":
        # forward: read and write a state; backward: read a state and the
        # adjoint, write the adjoint
        N = case["n"] ** 3
        return dict(bytes=float(case["T"] * N * 76 * 5), flops=700.0 * N * case["T"])
    N = case["n"] ** 3 if kind == "drag" else case["nx"] * case["ny"] * case["nz"]
    Q = case["lattice"]
    b = 2 * Q * _BYTES[case["storage"]] * N * case["steps"]
    fl = 250.0 * N * case["steps"]
    if kind == "driven":
        b += 2 * Q * 8 * N
    else:
        b += 34 * N
    if kind == "settle":
        fl += 300.0 * case["particles"] * case["n_sub"] * case["steps"]
    return dict(bytes=float(b), flops=fl)


# --------------------------------------------------------------------------
# the method in FP64, in plain torch
# --------------------------------------------------------------------------
def _rotation(q):
    w, x, y, z = q
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def _qmul(a, b):
    return np.array([a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3],
                     a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2],
                     a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1],
                     a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0]])


def _with_mass(p, h=0.5):
    """Volume, centroid and inertia by counting cell-centre samples of spacing
    h; the body frame then has its origin at the centroid."""
    cp, K = p["cp"], p["K"]
    B = float(np.abs(cp).max()) + math.sqrt(float(K.sum()))
    n = math.ceil(B / h)
    t = (torch.arange(-n, n, dtype=torch.float64, device=DEVICE) + 0.5) * h
    M = 0.0
    for c, k in zip(cp, K):
        M = M + float(k) / ((t[:, None, None] - c[2]) ** 2 + (t[None, :, None] - c[1]) ** 2
                            + (t[None, None, :] - c[0]) ** 2)
    z, y, x = torch.nonzero(M >= 1.0, as_tuple=True)
    r = torch.stack([t[x], t[y], t[z]], 1)
    c = r.mean(0)
    C = (r.T @ r) / len(r) - c[:, None] * c[None, :] + torch.eye(3, dtype=torch.float64, device=DEVICE) * h * h / 12
    m = p["density"] * len(r) * h ** 3
    C, c = C.cpu().numpy(), c.cpu().numpy()
    return dict(p, cp=cp - c, x=p["x"] + _rotation(p["q"]) @ c, mass=m,
                inertia=m * (np.trace(C) * np.eye(3) - C))


def _turn(p, torque, n_sub):
    """The rotational sub-steps of one step under a frozen world torque."""
    q, I = p["q"].copy(), p["inertia"]
    R = _rotation(q)
    Iinv = np.linalg.inv(I)
    w, T = R.T @ p["w"], R.T @ torque
    h = 1.0 / n_sub

    def rate(v, t):
        return Iinv @ (t - np.cross(v, I @ v))

    for _ in range(n_sub):
        wh = w + 0.5 * h * rate(w, T)
        a = float(np.linalg.norm(wh))
        s = math.sin(0.5 * h * a) / a if a > 0 else 0.5 * h
        d = np.concatenate([[math.cos(0.5 * h * a)], s * wh])
        T = _rotation(d).T @ T
        v = wh
        for _ in range(2):
            v = wh + 0.5 * h * rate(v, T)
        w = v
        q = _qmul(q, d)
    q /= np.linalg.norm(q)
    return q, _rotation(q) @ w


class Reference:
    """One lattice in FP64; particles that do not touch one another."""

    def __init__(self, shape, Q, periodic, tau, force=(0, 0, 0), q_exact=0):
        self.shape, self.Q, self.per, self.tau, self.q_exact = shape, Q, periodic, tau, q_exact
        self.n = torch.tensor([shape[2], shape[1], shape[0]], device=DEVICE)
        self.e, self.w = _lattice_vectors(Q)
        self.opp = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, Q)]
        self.F = [float(v) for v in force]
        self.own = torch.full(shape, -1, dtype=torch.int16, device=DEVICE)
        self.E = torch.tensor(self.e, dtype=torch.float64, device=DEVICE)
        self.W = torch.tensor(self.w, dtype=torch.float64, device=DEVICE)
        self.O = torch.tensor(self.opp, device=DEVICE)
        self.links = None
        self.parts = []

    def set_particles(self, parts):
        self.parts = parts
        self.links = None
        P, m = len(parts), max((len(p["K"]) for p in parts), default=1)
        cp, K = np.full((P, m, 3), 0.0), np.zeros((P, m))
        for j, p in enumerate(parts):
            k = len(p["K"])
            cp[j, :k] = p["x"] + p["cp"] @ _rotation(p["q"]).T
            cp[j, k:] = p["x"] + 1e3
            K[j, :k] = p["K"]
        t = lambda a: torch.tensor(np.array(a), dtype=torch.float64, device=DEVICE)  # noqa: E731
        self.cp, self.K = t(cp), t(K)
        self.x, self.v, self.om = (t([p[k] for p in parts]) for k in ("x", "v", "w"))

    def image(self, d):
        for a in range(3):
            if self.per[a]:
                L = float(self.shape[2 - a])
                d[..., a] -= L * torch.floor(d[..., a] / L + 0.5)
        return d

    def M(self, j, pos):
        r = self.image(pos[:, None, :] - self.cp[j])
        return (self.K[j] / (r * r).sum(-1)).sum(-1)

    def classify(self):
        nz, ny, nx = self.shape
        own = torch.full((nz * ny * nx,), -1, dtype=torch.int16, device=DEVICE)
        best = torch.zeros(nz * ny * nx, dtype=torch.float64, device=DEVICE)
        for j, p in enumerate(self.parts):
            c, R = self.cp[j, :len(p["K"])].cpu().numpy(), math.sqrt(float(p["K"].sum()))
            ax = []
            for a, n in enumerate((nx, ny, nz)):
                lo, hi = math.floor(c[:, a].min() - R), math.ceil(c[:, a].max() + R)
                if not self.per[a]:
                    lo, hi = max(lo, 0), min(hi, n - 1)
                elif hi - lo >= n:
                    hi = lo + n - 1
                ax.append(torch.arange(lo, hi + 1, device=DEVICE))
            z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
            pos = torch.stack([x, y, z], -1).reshape(-1, 3)
            M = self.M(torch.full((len(pos),), j, device=DEVICE), pos.double())
            m = pos % self.n
            n = m[:, 0] + nx * (m[:, 1] + ny * m[:, 2])
            up = (M >= 1.0) & (M > best[n])
            own[n[up]] = j
            best[n[up]] = M[up]
        return own.view(self.shape)

    def node(self, pos):
        """Index of integer positions, and whether they are inside the box."""
        ok = torch.ones(len(pos), dtype=torch.bool, device=DEVICE)
        for a in range(3):
            if not self.per[a]:
                ok &= (pos[:, a] >= 0) & (pos[:, a] < self.n[a])
        m = pos % self.n
        return m[:, 0] + self.n[0] * (m[:, 1] + self.n[1] * m[:, 2]), ok

    def position(self, n):
        return torch.stack([n % self.n[0], (n // self.n[0]) % self.n[1], n // (self.n[0] * self.n[1])], -1)

    def feq(self, i, rho, u):
        """Eq. (16) along direction i: an index, or one index per row."""
        ei, w = self.E[i], self.W[i]
        eu, uu = (u * ei).sum(-1), (u * u).sum(-1)
        return w * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu)

    def refill(self, f, new):
        n = torch.nonzero(((self.own >= 0) & (new < 0)).view(-1))[:, 0]
        if not len(n):
            return
        j = self.own.view(-1)[n].long()
        pos = self.position(n)
        u = self.v[j] + torch.linalg.cross(self.om[j], self.image(pos.double() - self.x[j]))
        flat, vals = f.view(self.Q, -1), []
        for i in range(self.Q):
            nb, ok = self.node(pos + self.E[i].long())
            known = ok & (self.own.view(-1)[nb] < 0) & (i > 0)
            g = flat[self.opp[i]][nb] + 6.0 * self.w[i] * (u @ self.E[i])
            vals.append(torch.where(known, g, self.feq(i, torch.ones_like(g), u)))
        for i in range(self.Q):
            flat[i][n] = vals[i]

    def find_links(self, own):
        """Every link (direction i, node n) whose source x - e_i is solid,
        with the geometry that does not depend on the flow."""
        fluid, found = own < 0, []
        for i in range(1, self.Q):
            e = self.e[i]
            src = torch.roll(own, (e[2], e[1], e[0]), (0, 1, 2))
            hit = fluid & (src >= 0)
            for a in range(3):
                if e[a] and not self.per[a]:
                    hit.select(2 - a, 0 if e[a] > 0 else self.shape[2 - a] - 1).fill_(False)
            n = torch.nonzero(hit.view(-1))[:, 0]
            found.append((torch.full_like(n, i), n, src.reshape(-1)[n].long()))
        i, n, j = (torch.cat(v) for v in zip(*found))
        pos, d = self.position(n), -self.E[i]
        q = self.fraction(j, pos.double(), d)
        if self.q_exact:  # the root of M(x + q d) = 1, bracketed by [0, 1]
            lo, hi = torch.zeros_like(q), torch.ones_like(q)
            for _ in range(50):
                mid = 0.5 * (lo + hi)
                out = self.M(j, pos.double() + mid[:, None] * d) < 1.0
                lo, hi = torch.where(out, mid, lo), torch.where(out, hi, mid)
            q = 0.5 * (lo + hi)
        ff, ok = self.node(pos + self.E[i].long())
        ok = ok & (own.view(-1)[ff] < 0)
        arm = self.image(pos.double() + q[:, None] * d - self.x[j])
        return i, n, j, q, torch.where(ok, ff, n), ok, arm

    def fraction(self, j, pos, d):
        """Eq. (27)."""
        Mf, Ms = self.M(j, pos), self.M(j, pos + d)
        return torch.clamp((1.0 - Mf) / (Ms - Mf), 0.0, 1.0)

    def vibb(self, flat, i, n, q, ff, ok, uw):
        """Eqs. (19)-(25): the unknown along e_i at the nodes n, and the
        population that leaves along -e_i."""
        io = self.O[i]
        F = torch.tensor(self.F, dtype=torch.float64, device=DEVICE)

        def moments(at):
            g = flat[:, at]
            rho = g.sum(0)
            return rho, (g.T @ self.E - 0.5 * F) / rho[:, None]

        rf, uf = moments(n)
        rg, ug = moments(ff)
        gf, gg = flat[io, n], flat[io, ff]
        move = 6.0 * self.W[io] * rf * (uw * self.E[i]).sum(-1)
        Q1 = q[:, None]
        neq = 2 * q * (gf - self.feq(io, rf, uf)) + (1 - 2 * q) * (gg - self.feq(io, rg, ug))
        near = q <= 0.5
        rd = torch.where(near, 2 * q * rf + (1 - 2 * q) * rg, rf)
        qs = torch.where(near, torch.ones_like(q), q)[:, None]
        us = torch.where(near[:, None], 2 * Q1 * uf + (1 - 2 * Q1) * ug, (1 - Q1) / qs * uf + (2 * Q1 - 1) / qs * uw)
        uss = (1 - Q1) / (1 + Q1) * ug + 2 * Q1 / (1 + Q1) * uw
        val = self.feq(io, rd, (us + 2 * uss) / 3.0) + neq + move
        return torch.where(ok, val, gf + move), gf

    def collide(self, fin):
        rho = fin.sum(0)
        u = [sum(self.e[i][a] * fin[i] for i in range(self.Q) if self.e[i][a]) for a in range(3)]
        u = [(u[a] + 0.5 * self.F[a]) / rho for a in range(3)]
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = sum(u[a] * self.F[a] for a in range(3))
        out, om, gf = [], 1.0 / self.tau, 1.0 - 0.5 / self.tau
        for i in range(self.Q):
            e = self.e[i]
            eu = sum((u[a] * e[a] for a in range(3) if e[a]), torch.zeros_like(rho))
            eF = sum(e[a] * self.F[a] for a in range(3))
            feq = self.w[i] * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu)
            out.append(fin[i] + om * (feq - fin[i]) + gf * self.w[i] * (3.0 * (eF - uF) + 9.0 * eu * eF))
        return out

    def pull(self, f, i):
        e = self.e[i]
        g = torch.roll(f[i], (e[2], e[1], e[0]), (0, 1, 2))
        for a in range(3):
            if e[a] and not self.per[a]:
                k = 0 if e[a] > 0 else self.shape[2 - a] - 1
                g.select(2 - a, k).copy_(f[self.opp[i]].select(2 - a, k))
        return g

    def step(self, f):
        """One step of f (changed in place); loads in self.load."""
        self.load = torch.zeros((len(self.parts), 6), dtype=torch.float64, device=DEVICE)
        if self.parts and self.links is None:
            new = self.classify()
            self.refill(f, new)
            self.own = new
            self.links = self.find_links(new)
        fin = torch.empty_like(f)
        for i in range(self.Q):
            fin[i] = self.pull(f, i)
        if self.parts:
            i, n, j, q, ff, ok, arm = self.links
            uw = self.v[j] + torch.linalg.cross(self.om[j], arm)
            val, gout = self.vibb(f.view(self.Q, -1), i, n, q, ff, ok, uw)
            d = -self.E[i]
            dP = (d - uw) * gout[:, None] + (d + uw) * val[:, None]
            self.load.index_add_(0, j, torch.cat([dP, torch.linalg.cross(arm, dP)], 1))
            fin.view(self.Q, -1)[i, n] = val
        out = self.collide(fin)
        if not self.parts:
            for i in range(self.Q):
                f[i] = out[i]
            return f
        solid = self.own >= 0
        for i in range(self.Q):
            f[i] = torch.where(solid, f[i], out[i])
        return f

    def move(self, n_sub, gravity):
        load = self.load.cpu().numpy()
        out = []
        for p, L in zip(self.parts, load):
            acc = (1.0 - 1.0 / p["density"]) * np.array([0.0, 0.0, gravity]) + L[:3] / p["mass"]
            q, w = _turn(p, L[3:], n_sub)
            out.append(dict(p, x=p["x"] + p["v"] + 0.5 * acc, v=p["v"] + acc, q=q, w=w))
        self.set_particles(out)

    def fields(self, f):
        rho = f.sum(0)
        u = torch.stack([(sum(self.e[i][a] * f[i] for i in range(self.Q) if self.e[i][a]) - 0.5 * self.F[a]) / rho
                         for a in range(3)])
        solid = self.own >= 0
        return dict(rho=torch.where(solid, 0.0, rho), u=torch.where(solid[None], 0.0, u),
                    flags=(self.own + 1).to(torch.int16))


def _gradient_exact(case, seed):
    """The drag by plain FP64 torch, flags frozen, and for the small boxes its
    gradient by autograd (None where that would take too long)."""
    cp32, K32, c, force, u0 = _gradient_inputs(case, seed)
    n, T, W = case["n"], case["T"], case["W"]
    grad = n ** 3 * T <= 4_000_000
    cp = cp32.double().to(DEVICE).requires_grad_(grad)
    K = K32.double().to(DEVICE).requires_grad_(grad)
    R = Reference((n, n, n), 19, (1, 1, 1), 0.8, force)
    with torch.no_grad():
        R.set_particles([dict(cp=cp.detach().cpu().numpy() - c, K=K.detach().cpu().numpy(), x=c, v=np.zeros(3),
                              w=np.zeros(3), q=np.array([1.0, 0.0, 0.0, 0.0]))])
        own = R.classify()
        R.own = own
        links = R.find_links(own)
    R.cp, R.K = cp[None], K[None]
    i, nn, j, _, ff, ok, arm = links
    q, still = R.fraction(j, R.position(nn).double(), -R.E[i]), torch.zeros_like(arm)
    ex = R.E[i][:, 0]
    u = torch.tensor(u0, dtype=torch.float64, device=DEVICE)
    one = torch.ones((n, n, n), dtype=torch.float64, device=DEVICE)
    f = torch.stack([R.feq(i, one, u.expand(n, n, n, 3)) for i in range(19)])
    keep = (own < 0)
    J = 0.0
    with torch.set_grad_enabled(grad):
        for t in range(T):
            flat = f.reshape(19, -1)
            val, gout = R.vibb(flat, i, nn, q, ff, ok, still)
            if t >= T - W:  # the constant 2 d w cancels over the closed surface
                J = J - (ex * (gout + val - 2.0 * R.W[i])).sum()
            fin = torch.stack([torch.roll(f[k], (R.e[k][2], R.e[k][1], R.e[k][0]), (0, 1, 2)) for k in range(19)])
            fin = fin.view(19, -1).index_put((i, nn), val).view(19, n, n, n)
            f = torch.stack([torch.where(keep, a, b) for a, b in zip(R.collide(fin), f)])
    J = J / W
    if not grad:
        return dict(J=J, cp=None, K=None)
    J.backward()
    return dict(J=J.detach(), cp=cp.grad, K=K.grad)


def exact(case, seed):
    kind = case["kind"]
    if kind == "settle" and case["floor"]:
        return None  # contacts: their stiff law amplifies the last digits of the loads
    if kind == "gradient":
        return _gradient_exact(case, seed)
    with torch.no_grad():
        if kind == "batch":
            F, ends = [], {}
            for c, (n, force, p) in enumerate(_batch_inputs(case, seed)):
                R = Reference((n, n, n), 19, (1, 1, 1), 0.8, (force, 0.0, 0.0))
                R.set_particles([p])
                f = torch.tensor(R.w, dtype=torch.float64, device=DEVICE)[:, None, None, None].repeat(1, n, n, n)
                for _ in range(case["steps"]):
                    R.step(f)
                F.append(R.load[0])
                ends[c] = (f, R.own) if c in (0, case["boxes"] - 1) else None
            F = torch.stack(F)
            # solid nodes hold what the method leaves there: no value
            return dict(F=F[:, :3], T=F[:, 3:], first=None, last=None)
        if kind == "driven":
            poses = _driven_inputs(case, seed)
            R = Reference((case["nz"], case["ny"], case["nx"]), case["lattice"], (1, 1, 0), 0.8,
                          q_exact=case["q_exact"])
            f = _flow(R.Q, R.shape, seed)
            loads = []
            for pose in poses:
                R.set_particles(pose)
                R.step(f)
                loads.append(R.load)
            return dict(loads=torch.stack(loads), f=None)
        if kind == "settle":
            parts = [_with_mass(p) for p in _particles_of(case, seed)]
            R = Reference((case["nz"], case["ny"], case["nx"]), case["lattice"],
                          (case["px"], case["py"], case["pz"]), case["tau"])
            f = _flow(R.Q, R.shape, seed)
            R.set_particles(parts)
            for k in range(case["steps"]):
                R.step(f)
                load = R.load
                own = R.own
                R.move(case["n_sub"], case["gravity"])
            s = {k: np.array([p[k] for p in R.parts]) for k in ("x", "v", "q", "w")}
            R.own = own
            return dict(R.fields(f), F=load[:, :3], T=load[:, 3:], **s)
        n = case.get("n")
        shape = (n, n, n) if kind == "drag" else (case["nz"], case["ny"], case["nx"])
        force = (2e-6 * (48.0 / n) ** 2, 0.0, 0.0) if kind == "drag" else (1e-6, 0.0, 0.0)
        R = Reference(shape, case["lattice"], (1, 1, 1 if kind == "drag" else 0), 0.8, force)
        f = _flow(R.Q, shape, seed, 1e-3 if kind == "drag" else 0.01)
        if kind == "drag":
            R.set_particles([_drag_inputs(case, seed)])
        for _ in range(case["steps"]):
            R.step(f)
        if kind == "drag":
            return dict(R.fields(f), F=R.load[:, :3], T=R.load[:, 3:])
        return R.fields(f)
