"""Performance cases: what users of this library run, through its public entry points.

Every case is one pass of a program that holds a domain (or a batch of domains) and new
inputs for it: it sets the initial state, advances it frame by frame (new inflow velocities
and the diagnostics of every frame, as a streaming smoke program does), and reads the final
state back into its own device buffers; or it resumes from a checkpoint; or it takes the
gradient of a smoke-control loss.  ``exact`` computes the same outputs in 64 bits with plain
torch operations (an implementation of its own: populations unshifted, the moments as 3-point
sums about u, the equilibrium as the textbook second-order polynomial).

Kinds
  rollout     one block: initial state, frames of steps with diagnostics, whole final state
  resume      one block: populations, velocity and scalar written from a checkpoint, steps,
              the populations read back
  multiscale  a reference block and refined blocks at non-integer spacing ratios
  batch       many small independent plumes stepped together
  adjoint     rollout of one block and the gradient of a loss of its final scalar
  adjoint_ms  the same on a continuous-scale domain, gradients of every block
"""
import math

import numpy as np
import torch

from paper_1807_02284_gb300 import autograd, lbm

SOLID, INFLOW, SOURCE = 1, 2, 4
DEV = "cuda"


# ------------------------------------------------------------------------------- the cases

def _rollout(nx, ny, nz, **kw):
    c = dict(kind="rollout", nx=nx, ny=ny, nz=nz, storage="fp32", grad="lagged", periodic=False,
             spheres=0, surface="bounce", walls=False, inflow=False, frames=4, steps=4, nu=1e-3)
    c.update(kw)
    return c


def _adjoint(nx, ny, nz, **kw):
    c = dict(kind="adjoint", nx=nx, ny=ny, nz=nz, storage="fp32", grad="lagged", periodic=True,
             spheres=0, inflow=False, steps=20, every=10, nu=1e-3)
    c.update(kw)
    return c


def listed():
    return [
        # a decaying vortex in a small periodic box: the smallest call, launches and latency
        _rollout(32, 32, 32, periodic=True, frames=4, steps=8, nu=1.6e-2, name="box32"),
        # an interactive smoke plume: new inflow velocities and diagnostics every second step
        _rollout(64, 64, 64, spheres=1, inflow=True, frames=8, steps=2, nu=1e-4, name="plume64"),
        # a duct with no-slip floor and lid and a regularized obstacle; odd, ragged extents
        _rollout(97, 61, 75, spheres=1, surface="wall", walls=True, inflow=True, frames=2,
                 steps=8, nu=2e-3, name="duct97"),
        # flow past a sphere at the resolution and viscosity of the relaxation comparison, the
        # adaptive rates from the local strain rate
        _rollout(196, 98, 98, grad="local", spheres=1, surface="wall", inflow=True, frames=2,
                 steps=8, nu=1e-4, name="sphere196"),
        # the headline workload: the 256^3 smoke plume
        _rollout(256, 256, 256, spheres=1, inflow=True, nu=1e-5, name="plume256"),
        # the same with half-precision storage
        _rollout(256, 256, 256, storage="fp16", spheres=1, inflow=True, nu=1e-5,
                 name="plume256_fp16"),
        # a run resumed from a checkpoint and checkpointed again, fixed relaxation rates
        dict(kind="resume", nx=128, ny=128, nz=128, storage="fp32", grad="fixed", periodic=False,
             steps=8, nu=1e-4, name="resume128"),
        # continuous-scale domain: 128^3 at h = 1, 96^3 at h = 1/1.5, 64^3 at h = 1/2.25
        dict(kind="multiscale", scale=1.0, blocks=3, steps=24, nu=1e-5, name="multiscale3"),
        # 64 small plumes of uneven sizes, as a training set or a parameter study takes them
        dict(kind="batch", count=64, lo=24, hi=96, storage="fp32", frames=4, steps=4, nu=1e-5,
             name="batch64"),
        # smoke control: 128^3 periodic box, gradient with respect to the initial velocity
        _adjoint(128, 128, 128, name="adjoint128"),
        # the gradient of a plume: open faces, inflow, a bounce-back sphere, uneven extents
        _adjoint(72, 60, 51, periodic=False, spheres=1, inflow=True, steps=12, every=4,
                 name="adjoint_plume"),
        # the gradient through a continuous-scale domain
        dict(kind="adjoint_ms", scale=0.5, blocks=3, steps=2, every=2, nu=1e-3,
             name="adjoint_ms"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rollout"] * 6 + ["batch"] * 2 + ["adjoint"] * 2 +
                      ["resume", "multiscale", "adjoint_ms"])
    if kind in ("rollout", "resume"):
        n = _log_int(rng, 24, 224)
        nx, ny, nz = (max(12, min(320, int(n * rng.uniform(0.7, 1.25)))) for _ in range(3))
    if kind == "rollout":
        spheres = rng.choice([0, 1, 3])
        periodic = rng.random() < 0.25
        return _rollout(nx, ny, nz, storage=rng.choice(["fp32", "fp32", "fp16"]),
                        grad=rng.choice(["lagged", "lagged", "local", "fixed"]),
                        periodic=periodic, spheres=spheres,
                        surface=rng.choice(["bounce", "bounce", "wall"]) if spheres else "bounce",
                        walls=not periodic and rng.random() < 0.25,
                        inflow=not periodic and rng.random() < 0.8,
                        frames=rng.choice([2, 4]), steps=rng.choice([1, 2, 3, 4]),
                        nu=10.0 ** rng.uniform(-4, -2))
    if kind == "resume":
        return dict(kind="resume", nx=nx, ny=ny, nz=nz, storage=rng.choice(["fp32", "fp16"]),
                    grad=rng.choice(["lagged", "local", "fixed"]), periodic=rng.random() < 0.5,
                    steps=rng.randint(1, 8), nu=10.0 ** rng.uniform(-4, -2))
    if kind == "multiscale":
        return dict(kind="multiscale", scale=rng.uniform(0.3, 1.0), blocks=rng.choice([2, 3]),
                    steps=rng.randint(4, 24), nu=10.0 ** rng.uniform(-5, -3))
    if kind == "batch":
        lo = rng.randint(16, 40)
        return dict(kind="batch", count=_log_int(rng, 4, 64), lo=lo, hi=rng.randint(lo + 8, 96),
                    storage=rng.choice(["fp32", "fp32", "fp16"]), frames=rng.choice([2, 4]),
                    steps=rng.choice([1, 2, 3, 4]), nu=10.0 ** rng.uniform(-5, -3))
    if kind == "adjoint_ms":
        return dict(kind="adjoint_ms", scale=rng.uniform(0.25, 0.5), blocks=rng.choice([2, 3]),
                    steps=rng.randint(1, 3), every=rng.randint(1, 3),
                    nu=10.0 ** rng.uniform(-3, -2))
    n = _log_int(rng, 16, 104)
    nx, ny, nz = (max(12, int(n * rng.uniform(0.75, 1.25))) for _ in range(3))
    periodic = rng.random() < 0.5
    return _adjoint(nx, ny, nz, storage=rng.choice(["fp32", "fp32", "fp16"]) if periodic else "fp32",
                    grad=rng.choice(["lagged", "lagged", "local", "fixed"]), periodic=periodic,
                    spheres=0 if periodic else rng.choice([0, 1]), inflow=not periodic,
                    steps=rng.randint(4, 20), every=rng.randint(2, 10),
                    nu=10.0 ** rng.uniform(-3, -2))


# -------------------------------------------------------------------------------- inputs

def _coords(dims, origin=(0.0, 0.0, 0.0), h=1.0):
    """Node positions (reference units) along x, y, z, broadcastable to [z][y][x]."""
    ax = [torch.arange(n, device=DEV, dtype=torch.float64) * h + o for n, o in zip(dims, origin)]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _fields(rng, dims, box, periodic, amp=0.05, origin=(0.0, 0.0, 0.0), h=1.0):
    """A smooth flow: seeded low Fourier modes of `box`, velocity at most `amp`, density within
    half a percent of 1, scalar in [0, 1]; float32 on the device."""
    X, Y, Z = _coords(dims, origin, h)
    top = 4

    def modes(n):
        s = 0.0
        for _ in range(n):
            k = [int(rng.integers(-top, top + 1)) for _ in range(3)]
            w = [2 * math.pi * k[a] / box[a] * (1.0 if periodic else 0.83) for a in range(3)]
            s = s + float(rng.standard_normal()) * torch.cos(w[0] * X + w[1] * Y + w[2] * Z +
                                                             float(rng.uniform(0, 2 * math.pi)))
        return s.expand(dims[2], dims[1], dims[0])

    u = torch.stack([modes(4) for _ in range(3)])
    u = u * (amp / 7.0)
    u = u.clamp(-amp, amp)
    rho = 1.0 + 0.005 * torch.sin(modes(3))
    c = 0.5 + 0.5 * torch.sin(modes(3))
    return u.float().contiguous(), rho.float().contiguous(), c.float().contiguous()


def _spheres(rng, n, dims, origin=(0.0, 0.0, 0.0)):
    m = min(dims)
    out = []
    for _ in range(n):
        r = float(rng.uniform(0.06, 0.1)) * m
        out.append(tuple(origin[a] + float(rng.uniform(0.3, 0.7)) * dims[a] for a in range(3)) + (r,))
    return out


def _flags(dims, spheres, inflow, origin=(0.0, 0.0, 0.0), h=1.0):
    """Obstacle voxels of the spheres, and a disk of inflow and smoke-source nodes on the face
    x = 0 (radius an eighth of the smaller extent)."""
    X, Y, Z = _coords(dims, origin, h)
    fl = torch.zeros((dims[2], dims[1], dims[0]), dtype=torch.uint8, device=DEV)
    for x, y, z, r in spheres:
        fl[(X - x) ** 2 + (Y - y) ** 2 + (Z - z) ** 2 <= r * r] = SOLID
    if inflow:
        r = max(2.0, min(dims[1], dims[2]) / 8.0)
        disk = ((Y - dims[1] / 2.0) ** 2 + (Z - dims[2] / 2.0) ** 2 <= r * r)[:, :, 0]
        fl[:, :, 0] = torch.where(disk, torch.full_like(fl[:, :, 0], INFLOW | SOURCE), fl[:, :, 0])
    return fl


def _records(rng, fl, u_in, noise=0.01):
    """Inflow records of every inflow node: u_in along x with +/- noise."""
    z, y = np.nonzero(fl[:, :, 0].cpu().numpy() & INFLOW)
    rec = np.zeros(z.size, dtype=lbm.INFLOW_RECORD)
    rec["y"], rec["z"] = y, z
    j = noise * u_in * (2.0 * rng.random((3, z.size)) - 1.0)
    rec["ux"], rec["uy"], rec["uz"] = u_in + j[0], j[1], j[2]
    return rec


def _block_inputs(rng, dims, spheres, inflow, periodic, frames, u_in=0.1):
    fl = _flags(dims, spheres, inflow)
    u, rho, c = _fields(rng, dims, dims, periodic)
    recs = [_records(rng, fl, u_in) for _ in range(frames)] if inflow else None
    if inflow:
        r = _records(rng, fl, u_in)
        u[:, torch.from_numpy(r["z"].astype(np.int64)), torch.from_numpy(r["y"].astype(np.int64)),
          torch.from_numpy(r["x"].astype(np.int64))] = torch.from_numpy(
              np.stack([r["ux"], r["uy"], r["uz"]])).to(DEV)
    return dict(flags=fl, u=u, rho=rho, c=c, recs=recs)


def _ms_blocks(scale, blocks):
    """(dims, origin, h) of the continuous-scale domain's blocks."""
    n = [max(10, int(round(v * scale))) for v in (128, 96, 64)]
    spec = [((0.0, 0.0, 0.0), 1.0), ((24.0, 32.0, 32.0), 1 / 1.5), ((36.0, 50.0, 50.0), 1 / 2.25)]
    return [((n[b],) * 3, tuple(scale * v for v in spec[b][0]), spec[b][1]) for b in range(blocks)]


def _inputs(case, seed):
    """Everything the seed decides: geometry, fields, inflow records."""
    rng = np.random.default_rng([seed, 1807])
    k = case["kind"]
    if k in ("rollout", "adjoint"):
        dims = (case["nx"], case["ny"], case["nz"])
        b = _block_inputs(rng, dims, _spheres(rng, case["spheres"], dims), case["inflow"],
                          case["periodic"], case.get("frames", 0))
        if k == "adjoint":
            X, Y, Z = _coords(dims)
            s, off = min(dims) / 8.0, rng.uniform(-0.06, 0.06, 3)
            blob = lambda o: torch.exp(-sum((V - dims[a] * (0.5 + o[a])) ** 2  # noqa: E731
                                            for a, V in enumerate((X, Y, Z))) / (2 * s * s))
            b["c"] = blob((0, 0, 0)).float().contiguous()
            b["target"] = blob(off).float().reshape(-1).contiguous()
        return b
    if k == "resume":
        dims = (case["nx"], case["ny"], case["nz"])
        u, rho, c = _fields(rng, dims, dims, case["periodic"])
        g = torch.Generator(device=DEV).manual_seed(int(rng.integers(1 << 31)))
        f = torch.empty((27,) + u.shape[1:], device=DEV)
        w = _weights()
        for q in range(27):     # near equilibrium, with a non-equilibrium part of one percent
            k3 = _PAPER[q]
            cu = sum(float(e) * u[a] for a, e in enumerate(k3))
            f[q] = w[_slot(k3)] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))
            f[q] *= 1.0 + 0.01 * (2.0 * torch.rand(u.shape[1:], device=DEV, generator=g) - 1.0)
        return dict(f=f.contiguous(), u=u, c=c)
    if k in ("multiscale", "adjoint_ms"):
        spec = _ms_blocks(case["scale"], case["blocks"])
        span = spec[1]
        sph = _spheres(rng, 4, tuple(int(n * span[2]) for n in span[0]), span[1])
        mode_seed = int(rng.integers(1 << 31))
        out = []
        for i, (dims, org, h) in enumerate(spec):
            fl = _flags(dims, sph, i == 0, org, h)
            u, rho, c = _fields(np.random.default_rng(mode_seed), dims, spec[0][0], False, 0.05, org, h)
            if i == 0:
                r = _records(rng, fl, 0.08)
                z, y, x = (torch.from_numpy(r[a].astype(np.int64)) for a in "zyx")
                u[:, z, y, x] = torch.from_numpy(np.stack([r["ux"], r["uy"], r["uz"]])).to(DEV)
            out.append(dict(flags=fl, u=u, rho=rho, c=c))
        n0 = spec[0][0][0]
        target = 0.5 + 0.5 * torch.sin(2 * math.pi * _coords(spec[0][0])[0] / n0 +
                                       float(rng.uniform(0, 6)))
        return dict(blocks=out, spec=spec,
                    target=target.expand(n0, n0, n0).float().reshape(-1).contiguous())
    members = []
    sizes = np.random.default_rng(case["count"])      # the set of sizes is the case's, not the seed's
    for _ in range(case["count"]):
        L = int(sizes.integers(case["lo"], case["hi"] + 1))
        members.append(_block_inputs(rng, (L, L, L), _spheres(rng, int(rng.integers(1, 4)), (L,) * 3),
                                     True, False, case["frames"], float(rng.uniform(0.03, 0.1))))
    return dict(members=members)


# ------------------------------------------------------------------------------- passes

def _domain(case, dims, stream=None):
    return lbm.Domain(dims, case["nu"], periodic=(bool(case.get("periodic")),) * 3,
                      storage=case.get("storage", "fp32"), adaptive=case.get("grad") != "fixed",
                      grad_mode="local" if case.get("grad") == "local" else "lagged", stream=stream)


def _buffers(dims, f=True):
    n = dims[0] * dims[1] * dims[2]
    return {"u": torch.empty(3 * n, device=DEV), "c": torch.empty(n, device=DEV),
            **({"f": torch.empty(27 * n, device=DEV)} if f else {})}


def prepare(case, seed):
    k = case["kind"]
    s = dict(case=case, **_inputs(case, seed))
    if k in ("rollout", "adjoint", "resume"):
        dims = (case["nx"], case["ny"], case["nz"])
        s["dom"] = _domain(case, dims)
        if k != "resume":
            s["dom"].set_flags(s["flags"])
            if case.get("walls") or case.get("surface") == "wall":
                s["dom"].set_walls([0, 0, 0, 0] + [case["walls"]] * 2, obstacles=case["surface"] == "wall")
        if k == "adjoint":
            s["u"] = s["u"].requires_grad_(True)
        else:
            s["out"] = _buffers(dims)
        if k == "rollout":
            s["diag"] = torch.empty((case["frames"], 5), dtype=torch.float64).pin_memory()
    elif k in ("multiscale", "adjoint_ms"):
        d = s["dom"] = _domain(case, s["spec"][0][0])
        for dims, org, h in s["spec"][1:]:
            d.add_scale_block(org, h, dims)
        for i, b in enumerate(s["blocks"]):
            d.set_flags(b["flags"], block=i)
        if k == "multiscale":
            s["out"] = [_buffers(dims) for dims, _, _ in s["spec"]]
        else:
            s["c_end"] = torch.empty(s["spec"][0][0][0] ** 3, device=DEV)
            s["grads"] = [torch.empty(3 * dims[0] ** 3, device=DEV) for dims, _, _ in s["spec"]]
    else:
        stream = torch.cuda.Stream()
        s["doms"] = []
        n = 0
        for m in s["members"]:
            L = m["flags"].shape[0]
            d = _domain(case, (L, L, L), stream)
            d.set_flags(m["flags"])
            s["doms"].append(d)
            n += L ** 3
        s["out"] = {"u": torch.empty(3 * n, device=DEV), "c": torch.empty(n, device=DEV),
                    "f": torch.empty(27 * n, device=DEV)}
        s["diag"] = torch.empty((case["frames"], len(s["doms"]), 5), dtype=torch.float64).pin_memory()
        s["recs"] = [[m["recs"][i] for m in s["members"]] for i in range(case["frames"])]
    return s


def _read(dom, out, block=0):
    dom.read_field(lbm.LBM_FIELD_U, lbm.LBM_F32, block=block, out=out["u"])
    dom.read_field(lbm.LBM_FIELD_SCALAR, lbm.LBM_F32, block=block, out=out["c"])
    if "f" in out:
        dom.read_field(lbm.LBM_FIELD_F, lbm.LBM_F32, block=block, out=out["f"])


def run(state):
    s, case = state, state["case"]
    k = case["kind"]
    if k == "rollout":
        d = s["dom"]
        d.init_macro(s["u"], rho=s["rho"], c=s["c"])
        ticket = 0
        for i in range(case["frames"]):
            if s["recs"]:
                d.set_inflow(s["recs"][i])
            ticket = d.step_reduce_async(case["steps"], s["diag"][i])
        d.wait_results(ticket)
        _read(d, s["out"])
        # the diagnostics are sums of per-node FP32 values: accurate to FP32 rounding
        return {**s["out"], "diag": s["diag"].float()}
    if k == "resume":
        d = s["dom"]
        d.write_field(lbm.LBM_FIELD_F, s["f"])
        d.write_field(lbm.LBM_FIELD_U, s["u"])
        d.write_field(lbm.LBM_FIELD_SCALAR, s["c"])
        d.step(case["steps"])
        _read(d, s["out"])
        return s["out"]
    if k == "multiscale":
        d = s["dom"]
        for i, b in enumerate(s["blocks"]):
            d.init_macro(b["u"], rho=b["rho"], c=b["c"], block=i)
        d.step(case["steps"])
        for i, o in enumerate(s["out"]):
            _read(d, o, block=i)
        return s["out"]
    if k == "batch":
        doms = s["doms"]
        for d, m in zip(doms, s["members"]):
            d.init_macro(m["u"], rho=m["rho"], c=m["c"])
        ticket = 0
        for i in range(case["frames"]):
            lbm.set_inflow_batch(doms, s["recs"][i])
            ticket = lbm.step_batch_reduce_async(doms, case["steps"], s["diag"][i])
        doms[0].wait_results(ticket)
        at = 0
        for d, m in zip(doms, s["members"]):
            n = m["flags"].numel()
            _read(d, {"u": s["out"]["u"][3 * at:3 * (at + n)], "c": s["out"]["c"][at:at + n],
                      "f": s["out"]["f"][27 * at:27 * (at + n)]})
            at += n
        return {**s["out"], "diag": s["diag"].float()}
    if k == "adjoint":
        s["u"].grad = None
        with torch.cuda.stream(s["dom"].torch_stream):
            c = autograd.smoke_rollout(s["u"], s["dom"], case["steps"], case["every"], s["rho"], s["c"])
            loss = 0.5 * ((c - s["target"]) ** 2).sum()
            loss.backward()
        return {"c": c.detach(), "grad": s["u"].grad}
    d = s["dom"]
    for i, b in enumerate(s["blocks"]):
        d.init_macro(b["u"], rho=b["rho"], c=b["c"], block=i)
    d.set_tape(case["every"])
    d.step(case["steps"])
    d.read_field(lbm.LBM_FIELD_SCALAR, lbm.LBM_F32, out=s["c_end"])
    with torch.cuda.stream(d.torch_stream):
        d.adjoint_step(case["steps"], s["c_end"] - s["target"], s["grads"][0])
    for i in range(1, case["blocks"]):
        d.adjoint_block_grad(i, s["grads"][i])
    d.sync()
    return {"c": s["c_end"], "grads": s["grads"]}


# --------------------------------------------------------------------------------- work

def work(case):
    """Bytes: every step reads and writes each node's populations (27), velocity (3) and scalar
    once (the local-strain and fixed modes read no velocity) and its flag byte; the initial
    state is read (5 values) and stored, the final state is read and handed over.  A reverse
    step reads the step's input state (after the replay of the forward step), the adjoints of
    its result and writes those of its input.  Flops: about 700 per node update, 1600 per
    reversed update."""
    k = case["kind"]
    e = 2 if case.get("storage") == "fp16" else 4
    node = 2 * 27 * e + (24 if case.get("grad", "lagged") == "lagged" else 12) + 8 + 1
    state = 27 * e + 16
    io = (20 + state) + (state + 124)
    if k in ("rollout", "resume"):
        n = case["nx"] * case["ny"] * case["nz"]
        steps = case["steps"] * case.get("frames", 1)
        return {"bytes": n * (steps * node + (io if k == "rollout" else 2 * (state + 124))),
                "flops": n * steps * 700}
    if k == "batch":
        sizes = np.random.default_rng(case["count"])
        n = sum(int(sizes.integers(case["lo"], case["hi"] + 1)) ** 3 for _ in range(case["count"]))
        steps = case["steps"] * case["frames"]
        return {"bytes": n * (steps * node + io), "flops": n * steps * 700}
    back = 249 + 373
    if k == "adjoint":
        n = case["nx"] * case["ny"] * case["nz"]
        fwd = n * case["steps"] * node
        return {"bytes": fwd + n * (case["steps"] * back + state + 20 + 16),
                "flops": n * case["steps"] * (700 + 700 + 1600)}
    b, fl = 0, 0
    for dims, _, h in _ms_blocks(case["scale"], case["blocks"]):
        n, sub = dims[0] ** 3, max(1, math.ceil(1 / h - 1e-9)) * case["steps"]
        b += n * (sub * node + io)
        fl += n * sub * 700
        if k == "adjoint_ms":
            b += n * sub * back
            fl += n * sub * 2300
    return {"bytes": b, "flops": fl}


# -------------------------------------------------------------- the same in 64-bit torch

# velocities in the order of the populations that the library reads and writes
_PAPER = [(k % 3 - 1, k // 3 % 3 - 1, k // 9 - 1) for k in
          (13, 14, 12, 16, 10, 22, 4, 17, 15, 11, 9, 23, 21, 5, 3, 25, 19, 7, 1, 26, 24, 20, 18,
           8, 6, 2, 0)]
# working order: slot (cx + 1) + 3 (cy + 1) + 9 (cz + 1), so the opposite of k is 26 - k
_C = [(k % 3 - 1, k // 3 % 3 - 1, k // 9 - 1) for k in range(27)]
_NU_HI = (0.005, 0.007, 0.009, 0.01)


def _slot(c):
    return (c[0] + 1) + 3 * (c[1] + 1) + 9 * (c[2] + 1)


def _weights():
    return [(8 / 27, 2 / 27, 1 / 54, 1 / 216)[sum(v != 0 for v in c)] for c in _C]


def _equilibrium(rho, u):
    usq = 1.5 * (u * u).sum(0)
    w = _weights()
    out = []
    for k in range(27):
        cu = sum(e * u[a] for a, e in enumerate(_C[k]) if e)
        out.append(w[k] * rho * (1 + 3 * cu + 4.5 * cu * cu - usq) if any(_C[k]) else w[k] * rho * (1 - usq))
    return torch.stack(out)


def _central(f, u):
    """Central moments sum f (cx - ux)^a (cy - uy)^b (cz - uz)^c, index [c][b][a]."""
    v = f.reshape((3, 3, 3) + f.shape[1:])
    for a, dim in ((0, 2), (1, 1), (2, 0)):
        m, z, p = v.unbind(dim)
        x = [-1 - u[a], -u[a], 1 - u[a]]
        v = torch.stack([m + z + p, x[0] * m + x[1] * z + x[2] * p,
                         x[0] * x[0] * m + x[1] * x[1] * z + x[2] * x[2] * p], dim)
    return v


def _populations(v, u):
    """The inverse of _central."""
    for a, dim in ((0, 2), (1, 1), (2, 0)):
        k0, k1, k2 = v.unbind(dim)
        r1 = k1 + u[a] * k0
        r2 = k2 + u[a] * (2 * k1 + u[a] * k0)
        v = torch.stack([0.5 * (r2 - r1), k0 - r2, 0.5 * (r2 + r1)], dim)
    return v.reshape((27,) + v.shape[3:])


def _macro(f):
    rho = f.sum(0)
    j = [sum((1 if _C[k][a] > 0 else -1) * f[k] for k in range(27) if _C[k][a]) for a in range(3)]
    return rho, torch.stack(j) / rho


def _scaled(f, u, rho, keep_of):
    """Equilibrium plus the non-equilibrium part with its central moments scaled by
    keep_of(K) = (shear, trace, third.. sixth-order factors)."""
    eq = _equilibrium(rho, u)
    K = _central(f - eq, u)
    shear, tr, hi = keep_of(K)
    rows = []
    for c in range(3):
        for b in range(3):
            for a in range(3):
                n = a + b + c
                x = K[c, b, a]
                if n == 2 and max(a, b, c) == 1:
                    x = shear * x
                elif n == 2:
                    s = (K[0, 0, 2] + K[0, 2, 0] + K[2, 0, 0]) / 3
                    x = tr * s + shear * (x - s)
                elif n > 2:
                    x = hi[n - 3] * x
                rows.append(x)
    return eq + _populations(torch.stack(rows).reshape(K.shape), u)


def _pad(x, periodic):
    """One more node on each side of the last three axes: the wrapped, or the nearest one."""
    for d in (-3, -2, -1):
        n = x.shape[d]
        lo, hi = x.narrow(d, 0, 1), x.narrow(d, n - 1, 1)
        x = torch.cat([hi, x, lo] if periodic else [lo, x, hi], d)
    return x


def _shifted(p, c, shape):
    """The values at x - c of an array padded by _pad."""
    return p[..., 1 - c[2]:1 - c[2] + shape[0], 1 - c[1]:1 - c[1] + shape[1],
             1 - c[0]:1 - c[0] + shape[2]]


def _norm(s):
    pos = s > 0
    return torch.where(pos, torch.sqrt(torch.where(pos, s, torch.ones_like(s))), torch.zeros_like(s))


def _sample(c, u, periodic):
    """Trilinear sample of c at x - u, the displacement at most one node per axis."""
    shape = c.shape
    at = []
    for a in range(3):
        n = shape[2 - a]
        x = torch.arange(n, device=c.device)
        x = x.reshape([-1 if 2 - a == d else 1 for d in range(3)])
        d = (-u[a]).clamp(-1.0, 1.0)
        fl = torch.floor(d.detach())
        t, i0 = d - fl, x + fl.long()
        if periodic:
            i0 = i0 % n
            i1 = (i0 + 1) % n
        else:
            t = torch.where(i0 < 0, torch.zeros_like(t), t)
            i0 = i0.clamp(0, n - 1)
            i1 = (i0 + 1).clamp(max=n - 1)
        at.append((i0, i1, t))
    flat, out = c.reshape(-1), 0.0
    for m in range(8):
        idx, w = 0, 1.0
        for a, stride in ((0, 1), (1, shape[2]), (2, shape[1] * shape[2])):
            i0, i1, t = at[a]
            idx = idx + (i1 if m >> a & 1 else i0) * stride
            w = w * (t if m >> a & 1 else 1 - t)
        out = out + w * flat[idx]
    return out


class _Exact:
    """One block in 64 bits."""

    def __init__(self, flags, periodic, nu, grad, walls=(False,) * 6, surface=False):
        fl = flags.cpu().numpy() if not flags.is_cuda else flags
        self.periodic, self.grad, self.s_nu = periodic, grad, 1.0 / (3.0 * nu + 0.5)
        solid = (fl & SOLID) != 0
        self.shape = solid.shape
        self.any_solid = bool(solid.any())
        self.obstacle = solid
        self.inflow = ((fl & INFLOW) != 0) & ~solid
        self.source = (fl & SOURCE) != 0
        wall = torch.zeros_like(solid)
        if surface:
            p = _pad(solid, periodic)
            outer = torch.zeros_like(solid)
            for c in _C:
                outer |= ~_shifted(p, c, self.shape)
            wall |= solid & outer
            solid = solid & ~outer
        self.solid = solid
        p = _pad(solid, periodic)
        self.behind = [_shifted(p, c, self.shape) for c in _C] if self.any_solid else None
        faces = torch.zeros_like(solid)
        n = self.shape[::-1]
        self.through = [torch.zeros_like(solid) for _ in range(27)]
        for f in range(6):
            if not walls[f]:
                continue
            sl = [slice(None)] * 3
            sl[2 - f // 2] = 0 if f % 2 == 0 else n[f // 2] - 1
            faces[tuple(sl)] = True
            for k in range(27):
                if _C[k][f // 2] == (1 if f % 2 == 0 else -1):
                    self.through[k][tuple(sl)] = True
        self.wall = (wall | faces) & ~solid & ~self.inflow
        if bool(self.wall.any()):
            self.unknown = [t | (wall & b) if self.behind else t
                            for t, b in zip(self.through, self.behind or [None] * 27)]
        else:
            self.unknown = None
        self.obst_wall = wall

    def start(self, rho, u, c):
        z = self.obstacle
        rho = torch.where(z, torch.ones_like(rho), rho)
        u = torch.where(z, torch.zeros_like(u), u)
        return _equilibrium(rho, u), u, torch.where(z, torch.zeros_like(c), c)

    def _regularized(self, f):
        """Wall nodes: unknown populations from their opposites, then every population from the
        density and the non-equilibrium stress of the completed set."""
        w = torch.tensor(_weights(), dtype=f.dtype, device=f.device)[:, None]
        at = self.wall
        d = torch.stack([f[k][at] for k in range(27)]) - w
        unk = torch.stack([m[at] for m in self.unknown])
        both = unk & unk.flip(0)
        d = torch.where(unk, d.flip(0), d)
        d = torch.where(both, torch.zeros_like(d), d)
        drho = d.sum(0) / (1.0 - (both * w).sum(0))
        neq = torch.where(both, torch.zeros_like(d), d - w * drho)
        cc = torch.tensor(_C, dtype=f.dtype, device=f.device)
        P = torch.einsum("ka,kb,kn->abn", cc, cc, neq)
        q = torch.einsum("ka,kb,abn->kn", cc, cc, P) - (P[0, 0] + P[1, 1] + P[2, 2]) / 3
        out = w + w * (drho + 4.5 * q)
        res = f.clone()
        res[:, at] = out
        return res

    def step(self, state):
        f, u, c = state
        p = _pad(f, self.periodic)
        g = torch.stack([_shifted(p[k], _C[k], self.shape) for k in range(27)])
        del p
        if self.any_solid:
            bounced = torch.stack([torch.where(self.behind[k] & ~self.obst_wall, f[26 - k], g[k])
                                   for k in range(27)])
            g = bounced
        if self.unknown is not None:
            g = self._regularized(g)
        rho, un = _macro(g)
        lagged = None
        if self.grad == "lagged":
            p = _pad(u, self.periodic)
            s = 0.0
            for a in range(3):
                e = [0, 0, 0]
                e[a] = 1
                d = _shifted(p, [-v for v in e], self.shape) - _shifted(p, e, self.shape)
                s = s + (d * d).sum(0)
            lagged = 0.5 * _norm(s)

        def keep(K):
            if self.grad == "fixed":
                phi = torch.ones_like(rho)
            else:
                n = lagged
                if n is None:
                    ss = (K[0, 0, 2] ** 2 + K[0, 2, 0] ** 2 + K[2, 0, 0] ** 2 +
                          2 * (K[0, 1, 1] ** 2 + K[1, 0, 1] ** 2 + K[1, 1, 0] ** 2))
                    n = 1.5 * self.s_nu / rho * _norm(2 * ss)
                phi = 5.0 - 4.0 * (n / 0.1).clamp(max=1.0)
            k = [1.0 - 1.0 / (3.0 * phi * v + 0.5) for v in _NU_HI]
            return 1.0 - self.s_nu, k[0], k

        fn = _scaled(g, un, rho, keep)
        del g
        if bool(self.inflow.any()):
            un = torch.where(self.inflow, u, un)
            at = self.inflow
            fn = fn.clone()
            fn[:, at] = _equilibrium(torch.ones_like(rho[at]), u[:, at])
        cn = _sample(c, un, self.periodic)
        cn = torch.where(self.source, torch.ones_like(cn), cn)
        if self.any_solid:
            w = torch.tensor(_weights(), dtype=f.dtype, device=f.device)[:, None, None, None]
            fn = torch.where(self.solid, w, fn)
            un = torch.where(self.solid, torch.zeros_like(un), un)
            cn = torch.where(self.solid, torch.zeros_like(cn), cn)
        return fn, un, cn

    def diagnostics(self, state):
        rho, u = _macro(state[0])
        on = ~self.solid
        rho = rho * on
        j = rho * u
        return torch.stack([rho.sum(), j[0].sum(), j[1].sum(), j[2].sum(),
                            0.5 * (rho * (u * u).sum(0)).sum()])


def _set_inflow(state, rec):
    f, u, c = state
    u = u.clone()
    z, y, x = (torch.from_numpy(rec[a].astype(np.int64)).to(DEV) for a in "zyx")
    u[:, z, y, x] = torch.from_numpy(np.stack([rec["ux"], rec["uy"], rec["uz"]])).double().to(DEV)
    return f, u, c


def _outputs(state):
    f, u, c = state
    return {"u": u.reshape(-1), "c": c.reshape(-1),
            "f": torch.stack([f[_slot(e)].reshape(-1) for e in _PAPER]).reshape(-1)}


def _exact_rollout(case, b):
    e = _Exact(b["flags"], bool(case.get("periodic")), case["nu"], case.get("grad", "lagged"),
               [False] * 4 + [bool(case.get("walls"))] * 2, case.get("surface") == "wall")
    st = e.start(b["rho"].double(), b["u"].double(), b["c"].double())
    diag = []
    for i in range(case["frames"]):
        if b["recs"]:
            st = _set_inflow(st, b["recs"][i])
        for _ in range(case["steps"]):
            st = e.step(st)
        diag.append(e.diagnostics(st))
    return st, torch.stack(diag)


class _ExactScales:
    """A reference block and refined blocks: per reference step the reference block advances
    once, then every refined block, coarse to fine, takes its sub-steps with its outer layer
    mapped from the finest coarser block around it, is interpolated to the end of the step and
    mapped into every coarser block."""

    def __init__(self, case, inp):
        self.spec = inp["spec"]
        self.nu = [case["nu"] / h for _, _, h in self.spec]
        self.e = [_Exact(b["flags"], False, nu, "lagged") for b, nu in zip(inp["blocks"], self.nu)]
        nb = len(self.spec)
        self.parent = [0] * nb
        for b in range(1, nb):
            for p in range(1, b):
                if self._inside(p, b):
                    self.parent[b] = p
        self.ghost, self.prior, self.post = [None] * nb, [None] * nb, {}
        for b in range(1, nb):
            dims = self.spec[b][0]
            edge = torch.zeros(dims[::-1], dtype=torch.bool, device=DEV)
            for d in range(3):
                edge.select(d, 0).fill_(True)
                edge.select(d, dims[2 - d] - 1).fill_(True)
            at = edge.nonzero()
            at = at[~self.e[b].obstacle[at[:, 0], at[:, 1], at[:, 2]]]
            self.ghost[b] = edge
            self.prior[b] = self._table(self.parent[b], b, at)
            for t in range(b):
                o, h = self.spec[b][1], self.spec[b][2]
                td, to, th = self.spec[t]
                ok = torch.ones(td[::-1], dtype=torch.bool, device=DEV)
                for a, V in enumerate(_coords(td, to, th)):
                    ok &= (V >= o[a] + h - 1e-9) & (V <= o[a] + (self.spec[b][0][a] - 2) * h + 1e-9)
                ok &= ~self.e[t].obstacle
                if t:
                    ok &= ~self.ghost[t]
                self.post[b, t] = self._table(b, t, ok.nonzero())

    def _inside(self, p, b):
        (pd, po, ph), (bd, bo, bh) = self.spec[p], self.spec[b]
        return all(bo[a] >= po[a] - 1e-9 and bo[a] + (bd[a] - 1) * bh <= po[a] + (pd[a] - 1) * ph + 1e-9
                   for a in range(3))

    def _table(self, src, dst, at):
        (sd, so, sh), (_, do, dh) = self.spec[src], self.spec[dst]
        i0, t = [], []
        for a in range(3):
            q = (at[:, 2 - a].double() * dh + do[a] - so[a]) / sh
            i = torch.floor(q).clamp(0, sd[a] - 2)
            i0.append(i.long())
            t.append(q - i)
        corner, weight = [], []
        for m in range(8):
            idx, w = 0, 1.0
            for a, stride in ((0, 1), (1, sd[0]), (2, sd[0] * sd[1])):
                idx = idx + (i0[a] + (m >> a & 1)) * stride
                w = w * (t[a] if m >> a & 1 else 1 - t[a])
            corner.append(idx)
            weight.append(torch.where(self.e[src].obstacle.reshape(-1)[idx], torch.zeros_like(w), w))
        s = sum(weight)
        some = s > 0
        weight = [w / torch.where(some, s, torch.ones_like(s)) for w in weight]
        Ss, Sd = (1.0 / (3.0 * self.nu[b] + 0.5) for b in (src, dst))
        khat = (1 - Sd) * (Ss / (sh / dh * Sd)) / (1 - Ss)
        return at, corner, weight, some, khat

    def _mapped(self, table, state, into, rest):
        at, corner, weight, some, khat = table
        f, u, c = state
        ff, cf = f.reshape(27, -1), c.reshape(-1)
        v = sum(w * ff[:, i] for w, i in zip(weight, corner))
        cv = sum(w * cf[i] for w, i in zip(weight, corner))
        w27 = torch.tensor(_weights(), dtype=f.dtype, device=f.device)[:, None]
        v = torch.where(some, v, w27)
        rho, un = _macro(v)
        v = _scaled(v, un, rho, lambda K: (khat, 1.0, (1.0,) * 4))
        if not rest:                   # a node without a source keeps its own value
            at, v, un, cv = at[some], v[:, some], un[:, some], cv[some]
        f, u, c = (x.clone() for x in into)
        z, y, x = at.unbind(1)
        f[:, z, y, x], u[:, z, y, x], c[z, y, x] = v, un, cv
        return f, u, c

    def step(self, states):
        old, cur = list(states), list(states)
        nb = len(old)
        for b in range(1, nb):         # the outer layers at the start of the step
            old[b] = self._mapped(self.prior[b], old[self.parent[b]], old[b], True)
        cur[0] = self.e[0].step(old[0])
        for b in range(1, nb):
            h = self.spec[b][2]
            n, p = max(1, math.ceil(1 / h - 1e-9)), self.parent[b]
            exact = abs(n * h - 1) < 1e-9
            now = old[b]
            for j in range(1, n + 1):
                th = j * h if j < n else 1.0
                new = self.e[b].step(now)
                if j == n and not exact:
                    t1, t2 = (n - 1) * h, n * h
                    a0 = (1 - t1) * (1 - t2) / (t1 * t2)
                    a1 = (1 - t2) / (t1 * (t1 - t2))
                    a2 = (1 - t1) / (t2 * (t2 - t1))
                    f = a0 * old[b][0] + a1 * now[0] + a2 * new[0]
                    c = a0 * old[b][2] + a1 * now[2] + a2 * new[2]
                    u = _macro(f)[1]
                    u = torch.where(self.e[b].solid, torch.zeros_like(u), u)
                    new = (f, u, c)
                src = tuple((1 - th) * x + th * y for x, y in zip(old[p], cur[p]))
                now = self._mapped(self.prior[b], src, new, True)
            cur[b] = now
            for t in range(b):
                cur[t] = self._mapped(self.post[b, t], cur[b], cur[t], False)
        return cur


def _exact_scales(case, inp):
    """(start, step) of the domain as functions of the blocks' initial velocities."""
    ms = _ExactScales(case, inp)

    def start(us):
        return [e.start(b["rho"].double(), u, b["c"].double())
                for e, b, u in zip(ms.e, inp["blocks"], us)]

    return start, ms.step


def _checkpointed(step, state, n):
    """n steps whose intermediate values are computed again in the backward pass."""
    from torch.utils.checkpoint import checkpoint
    for _ in range(n):
        state = checkpoint(step, state, use_reentrant=False)
    return state


def exact(case, seed):
    k = case["kind"]
    inp = _inputs(case, seed)
    if k in ("adjoint", "adjoint_ms"):
        blocks = inp["blocks"] if k == "adjoint_ms" else [inp]
        us = [b["u"].double().requires_grad_(True) for b in blocks]
        if k == "adjoint_ms":
            start, step = _exact_scales(case, inp)
            c = _checkpointed(step, start(us), case["steps"])[0][2].reshape(-1)
        else:
            e = _Exact(inp["flags"], case["periodic"], case["nu"], case["grad"])
            c = _checkpointed(e.step, e.start(inp["rho"].double(), us[0], inp["c"].double()),
                              case["steps"])[2].reshape(-1)
        loss = 0.5 * ((c - inp["target"].double()) ** 2).sum()
        g = torch.autograd.grad(loss, us)
        if k == "adjoint":
            return {"c": c.detach(), "grad": g[0]}
        return {"c": c.detach(), "grads": [x.reshape(-1) for x in g]}
    with torch.no_grad():
        if k == "rollout":
            st, diag = _exact_rollout(case, inp)
            return {**_outputs(st), "diag": diag}
        if k == "resume":
            e = _Exact(torch.zeros(inp["c"].shape, dtype=torch.uint8, device=DEV), case["periodic"],
                       case["nu"], case["grad"])
            f = torch.empty(inp["f"].shape, dtype=torch.float64, device=DEV)
            for q, c in enumerate(_PAPER):
                f[_slot(c)] = inp["f"][q].double()
            st = (f, inp["u"].double(), inp["c"].double())
            for _ in range(case["steps"]):
                st = e.step(st)
            return _outputs(st)
        if k == "multiscale":
            start, step = _exact_scales(case, inp)
            st = start([b["u"].double() for b in inp["blocks"]])
            for _ in range(case["steps"]):
                st = step(st)
            return [_outputs(s) for s in st]
        parts, diags = [], []
        for m in inp["members"]:
            st, diag = _exact_rollout(dict(case, grad="lagged"), m)
            parts.append(_outputs(st))
            diags.append(diag)
        return {**{n: torch.cat([p[n] for p in parts]) for n in ("u", "c", "f")},
                "diag": torch.stack(diags, 1)}
