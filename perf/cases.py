"""Performance cases of the library's main path: the solves its users run, timed through its entry points.

Every case is one call sequence of a user's program on a handle that it keeps (``prepare``): advance the
solve by a number of steps, sample forces and probes where that flow is sampled, and read the fields
(``run``).  The flows are the repository's own workloads: the D2Q9 acoustic pulse, the D2Q9 cylinder on one
level and on a coarse / fine pair, the round jet (D3Q19 / D3Q27, every storage format, both streaming
patterns, one level and refined), periodic boxes of any size, and the solve server.

``exact`` advances the same inputs with a plain torch FP64 restatement of the method (no code of the
package's kernels): collision, boundary rules, sponges, inlet noise, bounce-back and the 2:1 coupling.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1710_02065_gb300 import lbm

CS = 1.0 / math.sqrt(3.0)
LATTICES = {"d2q9": lbm.LBM_D2Q9, "d3q19": lbm.LBM_D3Q19, "d3q27": lbm.LBM_D3Q27}
Q = {"d2q9": 9, "d3q19": 19, "d3q27": 27}
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
# floating-point operations of one collision (multiply-adds as two), counted from the moment sums, the
# Hermite coefficients and the rebuild
FLOPS = {"d2q9": 120, "d3q19": 227, "d3q27": 420}
MEAN_FLOW = 0.05  # uniform flow the acoustic pulse travels on
SAMPLE_EVERY = 10  # steps between force / probe samples of the cylinder


def listed():
    def c(name, flow, lattice, nx, ny, nz, precision, steps, streaming="pull", shift=False):
        return dict(name=name, flow=flow, lattice=lattice, nx=nx, ny=ny, nz=nz, precision=precision, steps=steps,
                    streaming=streaming, shift=shift)

    return [
        # validation run: the periodic acoustic pulse in FP64, the smallest solve (launches and latency)
        c("pulse_fp64", "pulse", "d2q9", 128, 128, 1, "fp64", 200),
        # an acoustic field on a mean flow, 16-bit storage shifted by the mean-flow equilibrium
        c("pulse_fp16_shift", "pulse", "d2q9", 1024, 1024, 1, "fp16", 200, shift=True),
        # laminar cylinder with lift, drag and far-field pressure sampled every 10 steps
        c("cylinder_fp32", "cylinder", "d2q9", 1600, 800, 1, "fp32", 200),
        # the same flow on a coarse grid with a fine patch around the cylinder (small dependent kernels)
        c("cylinder_two_level_fp32", "cylinder2", "d2q9", 800, 400, 1, "fp32", 100),
        # the production solve: round jet in single precision, and with 16-bit storage
        c("jet_fp32", "jet", "d3q19", 384, 256, 256, "fp32", 48),
        c("jet_fp16", "jet", "d3q19", 384, 256, 256, "fp16", 48),
        # the jet where memory binds: one lattice updated in place
        c("jet_bf16_in_place", "jet", "d3q19", 384, 256, 256, "bf16", 48, streaming="aa"),
        # the jet on the tensor-product lattice at half the resolution
        c("jet_d3q27_fp16", "jet", "d3q27", 192, 128, 128, "fp16", 64),
        # double-precision reference of the jet (error studies)
        c("jet_fp64", "jet", "d3q19", 96, 64, 64, "fp64", 100),
        # the jet with a refined near-nozzle region
        c("jet_two_level_fp32", "jet2", "d3q19", 384, 256, 256, "fp32", 40),
        # a decaying vortex in a box of odd extents: initial state uploaded, advanced, all moments read
        c("box_odd_fp16", "box", "d3q19", 161, 129, 97, "fp16", 100),
        # the solve server: a mixed batch of requests (both lattices, both storages) run to completion;
        # nx / ny: the sides of its largest 2D / 3D requests
        c("serving_mix", "serve", "mixed", 512, 96, 8, "mixed", 400),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a flow, its lattice, storage and options, and sizes over the range of the listed ones."""
    flow = rng.choice(["pulse", "pulse", "cylinder", "cylinder2", "jet", "jet", "jet", "jet2", "box", "box", "serve"])
    lattice, streaming, shift, nz = "d2q9", "pull", False, 1
    if flow == "pulse":
        precision = rng.choice(["fp64", "fp32", "fp16", "bf16"])
        nx, ny = _log_int(rng, 64, 1024), _log_int(rng, 64, 1024)
        if precision in ("fp16", "bf16"):
            shift = rng.random() < 0.5
        if not shift:
            streaming = rng.choice(["pull", "pull", "aa"])
        steps = rng.randint(40, 200)
    elif flow == "cylinder":
        precision = rng.choice(["fp32", "fp32", "fp16", "bf16"])
        nx = _log_int(rng, 400, 1600)
        ny = nx // 2 + rng.randint(0, 3)
        steps = 10 * rng.randint(4, 20)
    elif flow == "cylinder2":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        nx = _log_int(rng, 200, 800)
        ny = nx // 2 + rng.randint(0, 3)
        steps = 10 * rng.randint(2, 10)
    elif flow == "jet":
        lattice = rng.choice(["d3q19", "d3q19", "d3q27"])
        precision = rng.choice(["fp32", "fp32", "fp16", "bf16"])
        k = math.exp(rng.uniform(math.log(0.25), math.log(0.9)))
        nx, ny, nz = (int(round(k * e)) for e in (384, 256, 256))
        if rng.random() < 0.5:  # rows of whole 16-byte groups, as a user rounds them
            nx = (nx + 7) // 8 * 8
        streaming = rng.choice(["pull", "pull", "aa"])
        steps = rng.randint(16, 48)
    elif flow == "jet2":
        lattice = rng.choice(["d3q19", "d3q19", "d3q27"])
        precision = rng.choice(["fp32", "fp32", "fp16"])
        k = math.exp(rng.uniform(math.log(0.3), math.log(0.7)))
        nx, ny, nz = (int(round(k * e)) for e in (384, 256, 256))
        steps = rng.randint(10, 32)
    elif flow == "box":
        lattice = rng.choice(["d3q19", "d3q19", "d3q27"])
        precision = rng.choice(["fp32", "fp16", "bf16"])
        nx, ny, nz = (_log_int(rng, 32, 192) for _ in range(3))
        steps = rng.randint(20, 100)
    else:
        lattice, precision = "mixed", "mixed"
        nx, ny, nz = _log_int(rng, 128, 512), _log_int(rng, 32, 96), rng.randint(4, 8)
        steps = rng.randint(100, 400)
    return dict(flow=flow, lattice=lattice, nx=nx, ny=ny, nz=nz, precision=precision, steps=steps, streaming=streaming,
                shift=shift)


# ---------------------------------------------------------------------------
# The flows: geometry, boundary rules and relaxation times
# ---------------------------------------------------------------------------
def _cylinder_params(case):
    """Diameter D = nx / 40 at (nx / 4, ny / 2), Ma 0.2, Re 150, sponge of nx / 16 cells at the outflow."""
    nx, ny = case["nx"], case["ny"]
    two = case["flow"] == "cylinder2"
    D, U = nx / 40.0, 0.2 * CS
    p = dict(D=D, U=U, sponge=nx // 16, xc=nx // 4, yc=ny // 2)
    if two:
        p["tau_f"] = 3 * U * 2 * D / 150.0 + 0.5
        p["tau"] = (p["tau_f"] + 0.5) / 2
        w, h = 2 * (nx // 5), 2 * (ny // 5)
        p["patch"] = (p["xc"] - w // 8, p["yc"] - h // 2, 0), (w, h, 1)
    else:
        p["tau"] = 3 * U * D / 150.0 + 0.5
    return p


def _disc(nx, ny, xc, yc, D):
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    return ((x - xc) ** 2 + (y - yc) ** 2 <= (D / 2.0) ** 2).astype(np.uint8)


def _jet_params(case, seed):
    """Inlet disc of diameter ny / 10.67 on -x, Ma 0.3, Re_D 2500, tanh shear layer, sponges of ny / 8 cells
    and zero-gradient outflow on the other faces, 1 % seeded inlet noise."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    D, U = ny * 24.0 / 256.0, 0.3 * CS
    z, y = np.meshgrid(np.arange(nz), np.arange(ny), indexing="ij")
    r = np.sqrt((y - ny / 2) ** 2 + (z - nz / 2) ** 2)
    prof = np.zeros((nz, ny, 3))
    prof[..., 0] = 0.5 * U * (1.0 - np.tanh((r - D / 2) / (2.0 * D / 40.0)))
    p = dict(D=D, U=U, tau=3 * U * D / 2500.0 + 0.5, prof=prof, sponge=ny // 8, chi=0.5, noise=(seed % 100000, 0.01))
    if case["flow"] == "jet2":
        w = ny // 4
        p["patch"] = (2, ny // 2 - w // 2, nz // 2 - w // 2), (w, w, min(w, nz - 8 - (nz // 2 - w // 2)))
        p["tau_f"] = 2 * p["tau"] - 0.5
    return p


def _tau(case, seed):
    if case["flow"] == "pulse":
        return 0.6
    if case["flow"] == "box":
        return 0.55
    return (_cylinder_params(case) if case["flow"].startswith("cyl") else _jet_params(case, seed))["tau"]


def _initial(case, seed, level=0):
    """rho [nz, ny, nx] and u [nz, ny, nx, 3] in FP32 on the GPU: the flow's base field with seeded perturbations."""
    gen = torch.Generator(device="cuda").manual_seed(2 * seed + level)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if level:
        _, ext = (_cylinder_params(case) if case["flow"] == "cylinder2" else _jet_params(case, seed))["patch"]
        nx, ny, nz = 2 * ext[0] + 1, 2 * ext[1] + 1, (2 * ext[2] + 1 if case["nz"] > 1 else 1)
    dev, f32 = "cuda", torch.float32
    rho = torch.ones((nz, ny, nx), device=dev, dtype=f32)
    u = torch.zeros((nz, ny, nx, 3), device=dev, dtype=f32)
    z, y, x = (torch.arange(n, device=dev, dtype=f32) for n in (nz, ny, nx))
    z, y, x = z[:, None, None], y[None, :, None], x[None, None, :]

    def rnd():
        return 2 * torch.rand((nz, ny, nx), generator=gen, device=dev, dtype=f32) - 1

    if case["flow"] == "pulse":  # Gaussian density pulse off the centre on a uniform flow
        a = torch.rand(3, generator=gen, device=dev, dtype=f32) * 0.2 + 0.4
        r2 = (x - a[0] * nx) ** 2 + (y - a[1] * ny) ** 2
        rho += 2e-3 * a[2] * torch.exp(-math.log(2.0) * r2 / max(4.0, ny / 20.0) ** 2)
        u[..., 0] = MEAN_FLOW
    elif case["flow"].startswith("cyl"):
        p = _cylinder_params(case)
        u[..., 0] = p["U"]
        u[..., 1] = 0.01 * p["U"] * rnd()
        solid = _solid(case, level)
        if solid is not None:
            u[torch.from_numpy(solid.astype(bool)).to(dev)[None]] = 0.0
    elif case["flow"].startswith("jet"):  # a developed column with 1 % noise in the sheared region
        p = _jet_params(case, seed)
        prof = torch.from_numpy(p["prof"][..., 0]).to(dev, f32)
        if level:
            (_, Y0, Z0), _ = p["patch"]
            iz = (torch.arange(nz, device=dev) // 2 + Z0).clamp(max=case["nz"] - 1)
            iy = (torch.arange(ny, device=dev) // 2 + Y0).clamp(max=case["ny"] - 1)
            prof = prof[iz][:, iy]
        u[..., 0] = prof[..., None] * (1 + 0.01 * rnd())
        for b in (1, 2):
            u[..., b] = 0.01 * prof[..., None] * rnd()
        rho += 1e-4 * rnd()
    else:  # Taylor-Green vortex with seeded phases
        a = 2 * math.pi * torch.rand(3, generator=gen, device=dev, dtype=f32)
        X, Y, Z = 2 * math.pi * x / nx + a[0], 2 * math.pi * y / ny + a[1], 2 * math.pi * z / nz + a[2]
        u[..., 0] = 0.05 * torch.sin(X) * torch.cos(Y) * torch.cos(Z)
        u[..., 1] = -0.05 * torch.cos(X) * torch.sin(Y) * torch.cos(Z)
        rho += 1e-3 * torch.cos(X) * torch.cos(Z) * torch.ones_like(Y)
    return rho, u


def _solid(case, level=0):
    p = _cylinder_params(case)
    if case["flow"] == "cylinder":
        return _disc(case["nx"], case["ny"], p["xc"], p["yc"], p["D"])
    if case["flow"] == "cylinder2" and level:
        (X0, Y0, _), (w, h, _) = p["patch"]
        return _disc(2 * w + 1, 2 * h + 1, 2 * (p["xc"] - X0), 2 * (p["yc"] - Y0), 2 * p["D"])
    return None


def _probes(case):
    nx, ny = case["nx"], case["ny"]
    return [nx // 4 + nx * (7 * ny // 8), 3 * nx // 4 + nx * (ny // 2)]


def _requests(case, seed):
    """Half D2Q9 pulses (side from nx / 8), half D3Q19 vortices (side from ny / 2), storage FP32 / FP16 in turn."""
    out = []
    for k in range(case["nz"]):
        two_d = k % 2 == 0
        frac = (k // 2 + 1) / ((case["nz"] + 1) // 2)
        side = max(16, int(case["nx"] * (1 / 8 + 7 / 8 * frac)) if two_d else int(case["ny"] * (1 / 2 + 1 / 2 * frac)))
        out.append(dict(flow="pulse" if two_d else "box", lattice="d2q9" if two_d else "d3q19", nx=side, ny=side,
                        nz=1 if two_d else side, precision="fp32" if (k // 2) % 2 == 0 else "fp16",
                        tau=0.55 + 0.04 * (k % 5), steps=case["steps"] - 17 * k, seed=seed * 64 + k))
    return out


# ---------------------------------------------------------------------------
# The program's state and one pass
# ---------------------------------------------------------------------------
def _pinned(*shape):
    return torch.empty(shape, dtype=torch.float32, pin_memory=True)


class _State:
    """A handle (or server), its stream, and the host and device buffers the program reads into."""

    def __del__(self):
        if getattr(self, "server", None):
            lbm.lbm_server_destroy(self.server)


def prepare(case, seed):
    s = _State()
    s.case, s.server = case, None
    if case["flow"] == "serve":
        s.requests = []
        for r in _requests(case, seed):
            rho, u = _initial(r, r["seed"])
            s.requests.append((r, rho.double().reshape(-1).cpu().numpy(), u.double().reshape(-1, 3).cpu().numpy(),
                               torch.empty(rho.numel()), torch.empty(rho.numel(), 3),
                               np.empty(rho.numel()), np.empty((rho.numel(), 3))))
        s.stream = torch.cuda.Stream()
        s.server = lbm.lbm_server_create(8 << 30, 64, s.stream.cuda_stream)
        return s
    n = (case["nx"], case["ny"], case["nz"])
    s.stream = torch.cuda.Stream()
    s.solver = lbm.Solver(LATTICES[case["lattice"]], n, _tau(case, seed), lbm.PRECISIONS[case["precision"]],
                          stream=s.stream.cuda_stream)
    h, N = s.solver.h, s.solver.ncell
    fp64 = case["precision"] == "fp64"
    s.rho = torch.empty(N, dtype=torch.float64, pin_memory=True) if fp64 else _pinned(N)
    s.u = torch.empty((N, 3), dtype=torch.float64, pin_memory=True) if fp64 else _pinned(N, 3)
    s.pi = _pinned(N, 6) if case["flow"] == "box" else None
    if case["flow"].startswith("cyl"):
        p = _cylinder_params(case)
        lbm.lbm_set_boundary(h, lbm.LBM_FACE_XM, lbm.LBM_BC_VELOCITY, (p["U"], 0.0, 0.0))
        lbm.lbm_set_boundary(h, lbm.LBM_FACE_XP, lbm.LBM_BC_OUTFLOW)
        lbm.lbm_set_sponge(h, lbm.LBM_FACE_XP, p["sponge"], 0.5, 1.0, (p["U"], 0.0, 0.0))
        samples = case["steps"] // SAMPLE_EVERY
        s.force = torch.zeros((samples, 3), dtype=torch.float64, device="cuda")
        s.probe = torch.zeros((samples, 2), dtype=torch.float64, device="cuda")
        s.cells = torch.tensor(_probes(case), dtype=torch.int64, device="cuda")
    elif case["flow"].startswith("jet"):
        p = _jet_params(case, seed)
        lbm.lbm_set_boundary(h, lbm.LBM_FACE_XM, lbm.LBM_BC_VELOCITY, None, p["prof"])
        for face in range(1, 6):
            lbm.lbm_set_boundary(h, face, lbm.LBM_BC_OUTFLOW)
            lbm.lbm_set_sponge(h, face, p["sponge"], p["chi"])
        lbm.lbm_set_inlet_noise(h, *p["noise"])
    if case["streaming"] == "aa":
        lbm.lbm_set_streaming(h, lbm.LBM_STREAM_AA)
    if case["shift"]:
        lbm.lbm_set_storage_shift(h, (MEAN_FLOW, 0.0, 0.0))
    if case["flow"] in ("cylinder2", "jet2"):
        lbm.lbm_add_refinement_patch(h, *p["patch"])
        ext, _ = lbm.lbm_level_info(h, 1)
        nf = int(np.prod(ext))
        rho, u = _initial(case, seed, 1)
        solid = _solid(case, 1) if case["flow"] == "cylinder2" else None
        if solid is not None:
            lbm.lbm_set_geometry_level(h, 1, solid)
        lbm.lbm_set_state_level(h, 1, rho.double().reshape(-1).cpu().numpy(), u.double().reshape(-1, 3).cpu().numpy())
        s.rho1 = torch.empty(nf, dtype=torch.float64, pin_memory=True)
        s.u1 = torch.empty((nf, 3), dtype=torch.float64, pin_memory=True)
    elif case["flow"] == "cylinder":
        lbm.lbm_set_geometry(h, _solid(case))
    rho, u = _initial(case, seed)
    s.rho.copy_(rho.reshape(-1))
    s.u.copy_(u.reshape(-1, 3))
    torch.cuda.synchronize()
    if case["flow"] == "box":  # the pass uploads its initial state
        s.rho0, s.u0 = s.rho.clone().pin_memory(), s.u.clone().pin_memory()
    elif fp64:
        lbm.lbm_set_state(h, s.rho.numpy(), s.u.numpy())
    else:
        lbm.lbm_set_state_f32(h, s.rho.numpy(), s.u.numpy())
    return s


def _serve(s):
    ids = [lbm.lbm_server_submit(s.server, LATTICES[r["lattice"]], lbm.PRECISIONS[r["precision"]],
                                 (r["nx"], r["ny"], r["nz"]), r["tau"], r["steps"], rho, u)
           for r, rho, u, *_ in s.requests]
    done = 0
    while done < len(ids):
        done += lbm.lbm_server_run(s.server, 100)
    out = []
    for rid, (_, _, _, rho32, u32, rho, u) in zip(ids, s.requests):
        lbm.lbm_server_result(s.server, rid, rho, u)
        rho32.copy_(torch.from_numpy(rho))  # fields are kept in single precision
        u32.copy_(torch.from_numpy(u))
        out += [rho32, u32]
    return out


def run(s):
    """One pass of the user's program; returns everything it reads."""
    case = s.case
    if s.server:
        return _serve(s)
    h, out = s.solver.h, []
    if case["flow"] == "box":
        lbm.lbm_set_state_f32(h, s.rho0.numpy(), s.u0.numpy())
    if case["flow"].startswith("cyl"):
        level = 1 if case["flow"] == "cylinder2" else 0
        for k in range(case["steps"] // SAMPLE_EVERY):
            lbm.lbm_step(h, SAMPLE_EVERY)
            lbm.lbm_force_async(h, level, s.force[k].data_ptr())
            lbm.lbm_probe_async(h, 2, s.cells.data_ptr(), s.probe[k].data_ptr())
    else:
        lbm.lbm_step(h, case["steps"])
    if case["precision"] == "fp64":
        lbm.lbm_moments(h, s.rho.numpy(), s.u.numpy())
    else:
        lbm.lbm_moments_f32(h, s.rho.numpy(), s.u.numpy(), None if s.pi is None else s.pi.numpy())
    out += [s.rho, s.u] + ([] if s.pi is None else [s.pi])
    real = s.rho.dtype
    if case["flow"] in ("cylinder2", "jet2"):
        lbm.lbm_moments_level(h, 1, s.rho1.numpy(), s.u1.numpy())
        out += [s.rho1.to(real), s.u1.to(real)]
    if case["flow"].startswith("cyl"):  # the series are kept in the fields' precision
        out += [s.force.to(real), s.probe.to(real)]
    return out


def work(case):
    """Populations read once and written once per cell and step, the fields written at the end, and the
    collision's operations."""
    if case["flow"] == "serve":
        parts = [work(dict(r, streaming="pull", shift=False)) for r in _requests(case, 0)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    cells = case["nx"] * case["ny"] * case["nz"]
    updates = cells * case["steps"]
    if case["flow"] in ("cylinder2", "jet2"):
        _, ext = (_cylinder_params(case) if case["flow"] == "cylinder2" else _jet_params(case, 0))["patch"]
        fine = (2 * ext[0] + 1) * (2 * ext[1] + 1) * (2 * ext[2] + 1 if case["nz"] > 1 else 1)
        updates += 2 * fine * case["steps"]
        cells += fine
    per = 2 * Q[case["lattice"]] * BYTES[case["precision"]]
    field = 16 if case["flow"] != "box" else 16 + 40
    if case["precision"] == "fp64":
        field *= 2
    return {"bytes": updates * per + cells * field, "flops": updates * FLOPS[case["lattice"]]}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
class _Lattice64:
    """Velocities, weights and the matrices of the moment sums and of the Hermite reconstruction
    w_i [a0 + 3 xi.a1 + 4.5 H2:A2 + third order], coefficients (a0, a1 x y z, A2 xx yy zz xy xz yz,
    A3 xxy xyy xxz xzz yyz yzz xyz)."""

    def __init__(self, name):
        d3, full = name != "d2q9", name == "d3q27"
        rng = (-1, 0, 1)
        xi = [(x, y, z) for z in (rng if d3 else (0,)) for y in rng for x in rng
              if full or abs(x) + abs(y) + abs(z) <= 2]
        self.xi, self.d = xi, 3 if d3 else 2
        one = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if not d3 else (
            {0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216} if full else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36})
        self.opp = [xi.index((-x, -y, -z)) for x, y, z in xi]
        M, R = [], []
        for x, y, z in xi:
            M.append([1, x, y, z, x * x, y * y, z * z, x * y, x * z, y * z])
            hx, hy, hz = x * x - 1 / 3, y * y - 1 / 3, (z * z - 1 / 3 if d3 else 0.0)
            H = dict(xxy=hx * y, xyy=hy * x, xxz=hx * z, xzz=hz * x, yyz=hy * z, yzz=hz * y)
            names = ["xxy", "xyy", "xxz", "xzz", "yyz", "yzz"]
            if not d3 or full:
                third = [13.5 * H[k] for k in names] + [27.0 * x * y * z if full else 0.0]
            else:  # pair sums and differences over their lattice norms
                third = dict.fromkeys(names, 0.0)
                for p, q in (("xxy", "yzz"), ("xzz", "xyy"), ("yyz", "xxz")):
                    a, b = 13.5 * (H[p] + H[q]), 4.5 * (H[p] - H[q])
                    third[p], third[q] = a + b, a - b
                third = [third[k] for k in names] + [0.0]
            w = one[x * x + y * y + z * z]
            row = [1.0, 3 * x, 3 * y, 3 * z, 4.5 * hx, 4.5 * hy, 4.5 * hz, 9 * x * y, 9 * x * z, 9 * y * z] + third
            R.append([w * v for v in row])
        self.M = torch.tensor(M, dtype=torch.float64, device="cuda").T.contiguous()
        self.R = torch.tensor(R, dtype=torch.float64, device="cuda")


def _pi_neq(m, dr, rho, u):
    """Pi^neq (xx, yy, zz, xy, xz, yz) about rho = 1 + dr and u from the shifted moments m."""
    pairs = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
    return [m[4 + k] - (dr / 3 if a == b else 0.0) - rho * u[a] * u[b] for k, (a, b) in enumerate(pairs)]


def _coefficients(eqs, neq, d):
    """Sum of s * equilibrium(dr, rho, u) over eqs and of omega * non-equilibrium (u, P)."""
    k = [0.0] * 17
    third = ((0, 0, 1), (0, 1, 1), (0, 0, 2), (0, 2, 2), (1, 1, 2), (1, 2, 2), (0, 1, 2))
    for s, dr, rho, u in eqs:
        r = s * rho
        terms = [s * dr] + [r * u[a] for a in range(3)]
        terms += [r * u[a] * u[b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
        terms += [r * u[a] * u[b] * u[c] for a, b, c in third]
        k = [x + y for x, y in zip(k, terms)]
    if neq is not None:
        om, u, P = neq
        at = {(0, 0): 0, (1, 1): 1, (2, 2): 2, (0, 1): 3, (0, 2): 4, (1, 2): 5}
        for i in range(6):
            k[4 + i] = k[4 + i] + om * P[i]
        for i, (a, b, c) in enumerate(third):
            k[10 + i] = k[10 + i] + om * (u[a] * P[at[b, c]] + u[b] * P[at[a, c]] + u[c] * P[at[a, b]])
    if d == 2:
        for i in (3, 6, 8, 9, 12, 13, 14, 15, 16):
            k[i] = k[i] * 0.0
    return k


class _Grid64:
    """One level in FP64: shifted populations f_i - w_i as [q, nz, ny, nx]."""

    def __init__(self, L, n, tau, periodic=(True, True, True)):
        self.L, self.n, self.om, self.periodic = L, n, 1.0 - 1.0 / tau, periodic
        self.solid = self.keep = self.chi = self.inlet = self.noise = None
        self.ref = (1.0, (0.0, 0.0, 0.0))

    def rebuild(self, k):
        shape = torch.broadcast_shapes(*(torch.as_tensor(x).shape for x in k))
        C = torch.stack([torch.as_tensor(x, dtype=torch.float64, device="cuda").expand(shape) for x in k])
        return (self.L.R @ C.reshape(17, -1)).reshape(len(self.L.xi), *shape)

    def equilibrium(self, rho, u):
        rho, u = rho.double(), u.double()
        return self.rebuild(_coefficients([(1.0, rho - 1.0, rho, [u[..., a] for a in range(3)])], None, self.L.d))

    def sums(self, g):
        return (self.L.M @ g.reshape(len(self.L.xi), -1)).reshape(10, *g.shape[1:])

    def streamed(self, f):
        g = torch.empty_like(f)
        for i, (x, y, z) in enumerate(self.L.xi):
            g[i] = torch.roll(f[i], (z, y, x), (0, 1, 2))
            if self.solid is not None and i != self.L.xi.index((0, 0, 0)):
                # the weights of an opposite pair agree, so the shifted values bounce as they are
                g[i] = torch.where(torch.roll(self.solid, (z, y, x), (0, 1, 2)), f[self.L.opp[i]], g[i])
        return g

    def step(self, f, t):
        m = self.sums(self.streamed(f))
        for a, dim in ((0, 3), (1, 2), (2, 1)):  # nodes of open faces take their inward neighbour's populations
            if not self.periodic[a]:
                n = m.shape[dim]
                m = m.index_select(dim, torch.arange(n, device="cuda").clamp(1, n - 2))
        dr, om = m[0], self.om
        if self.chi is None:
            rho = 1.0 + dr
            u = [m[1 + a] / rho for a in range(3)]
            P = _pi_neq(m, dr, rho, u)
            if self.inlet is not None:
                u = self.at_inlet(u, t)
            out = self.rebuild(_coefficients([(1.0, dr, rho, u)], (om, u, P), self.L.d))
        else:
            chi, (rr, ur) = self.chi, self.ref
            h = 1.0 / (1.0 + 0.5 * chi)
            drs = (dr + 0.5 * chi * (rr - 1.0)) * h
            rho = 1.0 + drs
            u = [(m[1 + a] + 0.5 * chi * rr * ur[a]) * h / rho for a in range(3)]
            P = _pi_neq(m, drs, rho, u)
            if self.inlet is not None:
                u = self.at_inlet(u, t)
            rv = [torch.tensor(v, dtype=torch.float64, device="cuda") for v in ur]
            out = self.rebuild(_coefficients([(1.0 - chi, drs, rho, u), (chi, rr - 1.0, rr, rv)], (om, u, P), self.L.d))
        return out if self.keep is None else torch.where(self.keep, f, out)

    def at_inlet(self, u, t):
        """The imposed velocity on the -x face (chi is zero there), with the seeded noise."""
        ub = self.inlet.clone()  # [nz, ny, 3]
        if self.noise is not None and self.noise[1] > 0:
            seed, amp = self.noise
            nz, ny, _ = ub.shape
            mag = ub.norm(dim=-1)
            c = torch.arange(nz * ny, device="cuda", dtype=torch.int64).reshape(nz, ny)
            for b in range(3):
                v = (seed << 32) + (t * nz * ny + c) * 3 + b
                ub[..., b] += torch.where(mag > 0, amp * mag * (2.0 * _u01(v) - 1.0), 0.0)
        u = [x.clone() for x in u]
        for a in range(3):
            u[a][:, :, 0] = ub[..., a]
        return u

    def fields(self, f, pi=False):
        m = self.sums(f)
        rho = 1.0 + m[0]
        u = [m[1 + a] / rho for a in range(3)]
        out = [rho.reshape(-1), torch.stack(u, -1).reshape(-1, 3)]
        if pi:
            P = _pi_neq(m, m[0], rho, u)
            out.append(torch.stack([P[0], P[3], P[4], P[1], P[5], P[2]], -1).reshape(-1, 6))
        return out

    def force(self, f):
        F = torch.zeros(3, dtype=torch.float64, device="cuda")
        fluid = ~(self.solid if self.keep is None else self.solid | self.keep)
        for i, (x, y, z) in enumerate(self.L.xi):
            link = torch.roll(self.solid, (-z, -y, -x), (0, 1, 2)) & fluid
            w = float(self.L.R[i, 0])
            F += 2.0 * ((f[i] + w) * link).sum() * torch.tensor([x, y, z], dtype=torch.float64, device="cuda")
        return F


def _i64(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _u01(x):
    """splitmix64 (Steele, Lea, Flood 2014) of int64 counters, scaled to [0, 1)."""
    def shr(v, k):
        return (v >> k) & ((1 << (64 - k)) - 1)
    z = x + _i64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * _i64(0x94D049BB133111EB)
    return shr(z ^ shr(z, 31), 11).double() * 2.0 ** -53


def _sigma(d, W):
    return torch.where(d >= 0, 3125.0 * (W - d) * d ** 4 / (256.0 * W ** 5), 0.0)


def _layers(n, widths, chi):
    """chi of face layers: widths {face: W}; larger value where layers overlap; [nz, ny, nx]."""
    out = torch.zeros((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    for face, W in widths.items():
        a = face // 2
        c = torch.arange(n[a], dtype=torch.float64, device="cuda")
        v = chi * _sigma(c - (n[a] - W) if face & 1 else W - 1 - c, float(W))
        out = torch.maximum(out, v.reshape([-1 if k == 2 - a else 1 for k in range(3)]))
    return out


class _Pair64:
    """A coarse level and its fine patch (vertex-based 2:1 coupling)."""

    def __init__(self, C, F, origin, extent, tau_c, tau_f):
        self.C, self.F = C, F
        self.o, self.e, self.three = origin, extent, C.n[2] > 1
        self.down = tau_f / (2 * tau_c), 1 - 1 / tau_f
        self.up = 2 * tau_c / tau_f, 1 - 1 / tau_c
        self.shell = self._shell(F.n, self.three)
        F.keep = self.shell if F.solid is None else self.shell | F.solid
        covered = torch.zeros((C.n[2], C.n[1], C.n[0]), dtype=torch.bool, device="cuda")
        covered[self.inner()] = True
        C.keep = covered

    @staticmethod
    def _shell(n, three):
        s = torch.ones((n[2], n[1], n[0]), dtype=torch.bool, device="cuda")
        s[(slice(1, -1) if three else slice(None)), 1:-1, 1:-1] = False
        return s

    def inner(self, grow=0):
        ax = []
        for a in (2, 1, 0):
            flat = a == 2 and not self.three
            ax.append(slice(0, 1) if flat else slice(self.o[a] + 1 - grow, self.o[a] + self.e[a] + grow))
        return tuple(ax)

    def moments(self, G, g):
        m = G.sums(g)
        rho = 1.0 + m[0]
        u = [m[1 + a] / rho for a in range(3)]
        return torch.stack([m[0]] + u + _pi_neq(m, m[0], rho, u))

    def node(self, G, m, alpha, om):
        u = [m[1], m[2], m[3]]
        return G.rebuild(_coefficients([(1.0, m[0], 1.0 + m[0], u)], (om, u, [alpha * m[4 + k] for k in range(6)]), G.L.d))

    def box(self, m):
        return m[(slice(None),) + self.inner(2)]

    def refine(self, M):
        """Coarse box moments (one node past each side) on the fine nodes."""
        for a, dim in ((0, 3), (1, 2), (2, 1)):
            if a == 2 and not self.three:
                continue
            n = self.e[a]
            c = M.narrow(dim, 1, n + 1)
            mid = (9 * (M.narrow(dim, 1, n) + M.narrow(dim, 2, n)) - M.narrow(dim, 0, n) - M.narrow(dim, 3, n)) / 16
            shape = list(M.shape)
            shape[dim] = 2 * n + 1
            out = torch.empty(shape, dtype=M.dtype, device=M.device)
            idx = [slice(None)] * 4
            idx[dim] = slice(0, None, 2)
            out[tuple(idx)] = c
            idx[dim] = slice(1, None, 2)
            out[tuple(idx)] = mid
            M = out
        return M

    def fill(self, f, M):
        m = self.refine(M)[:, self.shell]
        f[:, self.shell] = self.node(self.F, m, *self.down)
        return f

    def start(self, fc):
        return self.box(self.moments(self.C, fc))

    def step(self, fc, ff, M0, t):
        M1 = self.box(self.moments(self.C, self.C.streamed(fc)))
        new = self.C.step(fc, t)
        half = self.fill(self.F.step(ff, 2 * t), 0.5 * (M0 + M1))
        full = self.fill(self.F.step(half, 2 * t + 1), M1)
        m = self.moments(self.F, self.F.streamed(half))
        P = m[4:]
        for a, dim in ((0, 3), (1, 2), (2, 1)):
            if a == 2 and not self.three:
                continue
            P = 0.25 * (torch.roll(P, 1, dim) + 2 * P + torch.roll(P, -1, dim))
        m = torch.cat([m[:4], P])
        even = (slice(None), slice(2, -2, 2) if self.three else slice(None), slice(2, -2, 2), slice(2, -2, 2))
        m = m[even]  # coincident fine nodes of the covered coarse nodes
        ring = self._shell((m.shape[3], m.shape[2], m.shape[1]), self.three)
        sub = new[(slice(None),) + self.inner()]
        sub[:, ring] = self.node(self.C, m[:, ring], *self.up)
        return new, full, M1


def _cell_steps(case):
    c = case["nx"] * case["ny"] * case["nz"] * Q.get(case["lattice"], 19) * case["steps"]
    return c * (2 if case["flow"] == "jet2" else 1)


def _exact_solve(case, seed, steps=None, tau=None):
    L = _Lattice64(case["lattice"])
    n = (case["nx"], case["ny"], case["nz"])
    G = _Grid64(L, n, tau or _tau(case, seed), (case["flow"] in ("pulse", "box"),
                                                not case["flow"].startswith("jet"), not case["flow"].startswith("jet")))
    rho, u = _initial(case, seed)
    pair = p = None
    if case["flow"].startswith("cyl"):
        p = _cylinder_params(case)
        G.chi = _layers(n, {1: p["sponge"]}, 0.5)
        G.ref = (1.0, (p["U"], 0.0, 0.0))
        G.inlet = torch.zeros((1, n[1], 3), dtype=torch.float64, device="cuda")
        G.inlet[..., 0] = p["U"]
    elif case["flow"].startswith("jet"):
        p = _jet_params(case, seed)
        G.chi = _layers(n, {face: p["sponge"] for face in range(1, 6)}, p["chi"])
        G.chi[:, :, 0] = 0.0
        G.inlet = torch.from_numpy(p["prof"]).to("cuda")
        G.noise = p["noise"]
    if case["flow"] == "cylinder":
        G.solid = torch.from_numpy(_solid(case).astype(bool)).to("cuda")[None]
        G.keep = G.solid
    f = G.equilibrium(rho, u)
    if case["flow"] in ("cylinder2", "jet2"):
        o, e = p["patch"]
        nf = tuple(2 * v + 1 if (a < 2 or n[2] > 1) else 1 for a, v in enumerate(e))
        F = _Grid64(L, nf, p["tau_f"])
        if case["flow"] == "cylinder2":
            F.solid = torch.from_numpy(_solid(case, 1).astype(bool)).to("cuda")[None]
        ff = F.equilibrium(*_initial(case, seed, 1))
        pair = _Pair64(G, F, o, e, p["tau"], p["tau_f"])
        M0 = pair.start(f)
    force, probe = [], []
    for t in range(steps or case["steps"]):
        if pair:
            f, ff, M0 = pair.step(f, ff, M0, t)
        else:
            f = G.step(f, t)
        if case["flow"].startswith("cyl") and (t + 1) % SAMPLE_EVERY == 0:
            force.append(pair.F.force(ff) if pair else G.force(f))
            probe.append(f.sum(0).reshape(-1)[_probes(case)] / 3)
    out = G.fields(f, case["flow"] == "box")
    if pair:
        out += pair.F.fields(ff)
    if force:
        out += [torch.stack(force), torch.stack(probe)]
    return out


def exact(case, seed):
    if case["flow"] == "serve":
        out = []
        for r in _requests(case, seed):
            out += _exact_solve(dict(r, streaming="pull", shift=False), r["seed"], r["steps"], r["tau"])[:2]
        return out
    return _exact_solve(case, seed) if _cell_steps(case) < 5e10 else None
