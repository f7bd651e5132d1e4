"""What users of the framework have it do, as measurable cases.

Every case goes through the public entry points (the C ABI's binding
``lbfluct`` and the autograd wrapper ``adjoint``) on device buffers the caller
owns, in steady state: a state is prepared once and each ``run`` is the next
piece of the same simulation.  The kinds:

  step      lb_step: fluctuating or deterministic boxes, periodic or between
            walls, three storage formats, both equilibria, with or without a
            caller's force field, one or several steps a call
  chains    lb_couple_particles + lb_step: FENE / WCA bead-spring chains
  free      the same with free point particles between walls
  adjoint   one training step on the force field: forward, loss, reverse
  coupled   the same through particles, differentiable in their initial state
  batch     lb_batch_step: replica boxes of different sizes in one launch
  moments   lb_moments: the hydrodynamic fields of a state
  spheres   lb_step_spheres: moving solid spheres

``exact`` restates the method in 64 bits with plain torch (the moment basis of
Duenweg & Ladd's Table 1, Philox4x32-10 as in its paper) and shares no code
with the framework.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0803_2826_gb300 import adjoint as ADJ
from paper_0803_2826_gb300 import inputs
from paper_0803_2826_gb300 import lbfluct as L

KT = 1e-4
DT, NSUB = 0.1, 10                             # particle steps of one LB step
MASS, GAMMA = 1.0, 2.0
EPS, SIGMA, K_FENE, R0 = 0.01, 1.0, 0.3, 1.5   # chains, in lattice units
DTYPES = {"f32": (L.LB_F32, torch.float32), "f16": (L.LB_F16, torch.float16), "bf16": (L.LB_BF16, torch.bfloat16)}
L2_BYTES = 129e6
BATCH_CONFIG = (512, 2048, 1)                  # threads, nodes per tile, blocks per SM


def _step(name, shape, steps=1, dtype="f32", walls=False, kT=KT, relax=False, field=False, g=0.0, exponential=False):
    return {"name": name, "kind": "step", "nx": shape[0], "ny": shape[1], "nz": shape[2], "steps": steps, "dtype": dtype,
            "walls": walls, "kT": kT, "relax": relax, "field": field, "g": g, "exponential": exponential}


def listed():
    return [
        # the decaying shear wave that every validation run advances, many steps a call
        _step("wave_32", (32, 32, 32), steps=20),
        # a small ragged channel stepped one call at a time from a host loop
        _step("channel_small_ragged", (61, 47, 53), walls=True, relax=True, g=1e-5),
        # a large ragged channel in the narrowest storage
        _step("channel_bf16_ragged", (257, 131, 129), dtype="bf16", walls=True, g=1e-6),
        # a deterministic flow driven by the caller's force field
        _step("driven_field", (192, 160, 144), kT=0.0, relax=True, field=True),
        # entropic equilibrium at a visible flow speed
        _step("exponential_128", (128, 128, 128), exponential=True),
        # the headline run: a 256^3 bath with 64 chains of 256 monomers, coupling beside the fluid update
        {"name": "chains_256", "kind": "chains", "nx": 256, "ny": 256, "nz": 256, "chains": 64, "length": 256, "phi": 2,
         "overlap": True},
        # a small polymer box with the smoothest interpolation, in the plain order
        {"name": "chains_small_phi4", "kind": "chains", "nx": 72, "ny": 64, "nz": 60, "chains": 12, "length": 64, "phi": 4,
         "overlap": False},
        # tracers in a half-precision Poiseuille channel, the largest box that is run
        {"name": "channel_f16_tracers", "kind": "free", "nx": 512, "ny": 512, "nz": 512, "n": 100000, "dtype": "f16", "phi": 2,
         "overlap": False},
        # learning a force field: 50 steps, a checkpoint every 25
        {"name": "adjoint_64", "kind": "adjoint", "nx": 64, "ny": 64, "nz": 64, "steps": 50, "every": 25},
        # 512 replicas of mixed edges, ten steps of the ensemble a call
        {"name": "batch_512", "kind": "batch", "n": 512, "draw": 7, "ragged": False, "steps": 10},
        # reading the density, momentum and stress fields of a large box
        {"name": "moments_256", "kind": "moments", "nx": 256, "ny": 256, "nz": 256, "dtype": "f32", "walls": False},
        # a suspension of neutrally buoyant spheres
        {"name": "spheres_128", "kind": "spheres", "nx": 128, "ny": 128, "nz": 128, "n": 64, "radius": 4.0},
    ]


def _edge(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "chains", "free", "adjoint", "coupled", "batch", "moments", "spheres"])
    box = lambda lo, hi: (_edge(rng, lo, hi), _edge(rng, lo, hi), _edge(rng, lo, hi))  # noqa: E731
    if kind == "step":
        s = box(12, 300)
        exponential = rng.random() < 0.15
        c = _step("", s, steps=rng.choice([1, 1, 2, 5, 20]) if s[0] * s[1] * s[2] < 2e6 else 1, dtype=rng.choice(list(DTYPES)),
                  walls=rng.random() < 0.4, kT=rng.choice([0.0, KT, KT]), relax=rng.random() < 0.5,
                  field=rng.random() < 0.25, g=rng.choice([0.0, 1e-6]), exponential=exponential)
        del c["name"]
        return c
    if kind == "chains":
        s = box(40, 240)
        room = s[0] * s[1] * s[2] / 400
        length = _edge(rng, 16, 256)
        return {"kind": kind, "nx": s[0], "ny": s[1], "nz": s[2], "chains": max(1, min(_edge(rng, 1, 64), int(room / length))),
                "length": length, "phi": rng.choice([2, 2, 3, 4]), "overlap": rng.random() < 0.5}
    if kind == "free":
        s = box(24, 400)
        return {"kind": kind, "nx": s[0], "ny": s[1], "nz": s[2], "n": _edge(rng, 50, 100000), "dtype": rng.choice(list(DTYPES)),
                "phi": rng.choice([2, 2, 3, 4]), "overlap": rng.random() < 0.5}
    if kind == "adjoint":
        s = box(16, 80)
        return {"kind": kind, "nx": s[0], "ny": s[1], "nz": s[2], "steps": rng.randint(10, 50), "every": rng.choice([10, 25, 50])}
    if kind == "coupled":
        s = box(12, 48)
        return {"kind": kind, "nx": s[0], "ny": s[1], "nz": s[2], "n": _edge(rng, 10, 2000), "steps": rng.randint(3, 12),
                "every": rng.choice([4, 10])}
    if kind == "batch":
        return {"kind": kind, "n": _edge(rng, 8, 512), "draw": rng.randrange(1000), "ragged": rng.random() < 0.4,
                "steps": rng.choice([2, 5, 10])}
    if kind == "moments":
        s = box(24, 280)
        return {"kind": kind, "nx": s[0], "ny": s[1], "nz": s[2], "dtype": rng.choice(list(DTYPES)), "walls": rng.random() < 0.3}
    s = box(48, 200)
    return {"kind": "spheres", "nx": s[0], "ny": s[1], "nz": s[2],
            "n": max(1, min(_edge(rng, 1, 256), int(s[0] * s[1] * s[2] / 12000))), "radius": rng.choice([2.5, 3.0, 4.0, 4.7])}


# ---- inputs -------------------------------------------------------------------

def _shape(case):
    return case["nx"], case["ny"], case["nz"]


def _physics(case):
    """Keyword arguments of the box, as make_params takes them."""
    kw = {"kT": case.get("kT", 0.0 if case["kind"] in ("adjoint", "coupled") else KT),
          "walls": bool(case.get("walls", case["kind"] == "free")), "dtype": DTYPES[case.get("dtype", "f32")][0],
          "body_force": (case.get("g", 1e-6 if case["kind"] == "free" else 0.0), 0.0, 0.0),
          "equilibrium": int(case.get("exponential", False))}
    if case.get("relax"):
        kw.update(gamma_shear=0.2, gamma_bulk=-0.1, gamma_odd=0.1, gamma_even=0.05)
    return kw


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + 17)


def _flow(shape, kT, gen, amplitude=0.01):
    """rho [N] and u [3][N] (FP64): a shear wave with thermal density and velocity fluctuations."""
    nx, ny, nz = shape
    new = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    rho = 1.0 + math.sqrt(3.0 * max(kT, 1e-6)) * new(nz, ny, nx)
    u = math.sqrt(max(kT, 1e-6)) * new(3, nz, ny, nx)
    z = torch.arange(nz, device="cuda", dtype=torch.float64)
    phase = 2.0 * math.pi * torch.rand(1, generator=gen, device="cuda", dtype=torch.float64)
    u[0] += amplitude * torch.sin(2.0 * math.pi * z / nz + phase)[:, None, None]
    return rho, u


def _amplitude(case):
    return 0.05 if case.get("exponential") else 0.01


def _momenta(n, kT, gen):
    return math.sqrt(MASS * max(kT, 1e-6)) * torch.randn(n, 3, generator=gen, device="cuda", dtype=torch.float32)


def _chain_positions(case, gen):
    """Random walks of bond length 0.97, all chains grown side by side, each
    bead the first of 32 trial directions that is 1.0 away from every bead
    but its own predecessor; drawn again if two beads still came too close."""
    box = torch.tensor(_shape(case), device="cuda", dtype=torch.float64)
    nc, ln = case["chains"], case["length"]
    for _ in range(50):
        pos = torch.empty(nc, ln, 3, device="cuda", dtype=torch.float64)
        pos[:, 0] = torch.rand(nc, 3, generator=gen, device="cuda", dtype=torch.float64) * box
        for b in range(1, ln):
            v = torch.randn(nc, 32, 3, generator=gen, device="cuda", dtype=torch.float64)
            trial = pos[:, b - 1, None] + 0.97 * v / v.norm(dim=-1, keepdim=True)
            d = (trial.reshape(-1, 1, 3) - pos[:, :b].reshape(1, -1, 3)).float()
            d -= box.float() * torch.round(d / box.float())
            r2 = (d * d).sum(-1).view(nc, 32, nc, b)
            own = torch.arange(nc, device="cuda")
            r2[own, :, own, b - 1] = 9.0
            ok = r2.amin((2, 3)) >= 1.0
            best = torch.where(ok.any(1), ok.to(torch.float32).argmax(1), r2.amin((2, 3)).argmax(1))
            pos[:, b] = trial[own, best]
        flat = pos.view(-1, 3)
        worst = 9.0
        for k in range(0, flat.shape[0], 2048):
            d = (flat[k:k + 2048, None] - flat[None]).float()
            d -= box.float() * torch.round(d / box.float())
            r2 = (d * d).sum(-1)
            i = torch.arange(k, min(k + 2048, flat.shape[0]), device="cuda")
            r2[i - k, i] = 9.0
            worst = min(worst, r2.min().item())
        if worst > 0.85 ** 2:
            break
    return flat - box * torch.floor(flat / box)


def _free_positions(case, gen, walls):
    lo = torch.tensor([0.0, 0.0, 2.0 if walls else 0.0], device="cuda", dtype=torch.float64)
    hi = torch.tensor([case["nx"], case["ny"], case["nz"] - 3.0 if walls else case["nz"]], device="cuda", dtype=torch.float64)
    return lo + (hi - lo) * torch.rand(case["n"], 3, generator=gen, device="cuda", dtype=torch.float64)


def _batch_shapes(case):
    edges = inputs.replica_edges(case["n"], case["draw"])
    if not case["ragged"]:
        return [(e, e, e) for e in edges]
    rng = np.random.default_rng(case["draw"])
    return [tuple(int(e - v) for v in rng.integers(0, 6, 3)) for e in edges]


def _sub_box(shape):
    return tuple(3 * s // 8 for s in shape), tuple(max(3 * s // 8 + 1, 5 * s // 8) for s in shape)


class Box:
    """A box over two population buffers the program owns (typed, planes of lb_plane_pitch elements)."""

    def __init__(self, shape, seed, force=None, **kw):
        self.params = L.make_params(shape, seed=seed, **kw)
        self.shape, self.n = shape, shape[0] * shape[1] * shape[2]
        kind = {code: t for code, t in DTYPES.values()}[self.params.dtype]
        self.pops = [torch.zeros(19, L.lb_plane_pitch(self.params), dtype=kind, device="cuda") for _ in range(2)]
        self.force = force
        self.h = L.lb_create(self.params, self.pops[0], self.pops[1], force)

    def state(self):
        """The current populations of the fluid nodes, [19][...]."""
        cur, _ = L.lb_state_buffers(self.h)
        p = self.pops[0] if cur == self.pops[0].data_ptr() else self.pops[1]
        wall = self.shape[0] * self.shape[1] if self.params.walls else 0
        return p[:, wall:self.n - wall]

    def __del__(self):
        if getattr(self, "h", None) is not None:
            L.lb_destroy(self.h)
            self.h = None


def prepare(case, seed):
    kind = case["kind"]
    gen = _generator(seed)
    if kind == "batch":
        shapes = _batch_shapes(case)
        plist = [L.make_params(s, kT=KT, seed=seed + r, replica=r) for r, s in enumerate(shapes)]
        bufs = [torch.zeros(L.lb_batch_population_bytes(plist) // 4, dtype=torch.float32, device="cuda") for _ in range(2)]
        b = L.lb_batch_create(plist, bufs[0], bufs[1])
        L.lb_batch_set_config(b, *BATCH_CONFIG)
        for r, s in enumerate(shapes):
            rho, u = _flow(s, KT, gen)
            L.lb_batch_init_equilibrium(b, r, rho, u)
        return {"case": case, "b": _BatchOwner(b), "bufs": bufs, "cur": 0}
    shape, kw = _shape(case), _physics(case)
    force = None
    if case.get("field") or kind in ("adjoint", "coupled"):
        force = (1e-5 * torch.randn(3, *shape[::-1], generator=gen, device="cuda", dtype=torch.float32)).contiguous()
    if kind in ("adjoint", "coupled"):
        state = {"case": case, "theta": force.clone().requires_grad_(True), "lo_hi": _sub_box(shape)}
        lat = L.Lattice(shape, force=torch.empty_like(force), **kw)
        state["lat"] = lat
        if kind == "coupled":
            state["pos"], state["mom"] = _free_positions(case, gen, False), _momenta(case["n"], 0.0, gen)
            state["cp"] = L.couple_params(n_substeps=NSUB, dt=DT)
        return state
    box = Box(shape, seed, force, **kw)
    rho, u = _flow(shape, kw["kT"], gen, _amplitude(case))
    L.lb_init_equilibrium(box.h, rho, u)
    state = {"case": case, "box": box}
    if kind in ("chains", "free"):
        walls = kw["walls"]
        pos = _chain_positions(case, gen) if kind == "chains" else _free_positions(case, gen, walls)
        pos = pos.contiguous()
        mom = _momenta(pos.shape[0], kw["kT"], gen)
        more = {"chain_len": case["length"], "use_wca": True, "eps": EPS, "sigma": SIGMA, "k_fene": K_FENE, "r0": R0} if kind == "chains" else {}
        state.update(pos=pos, mom=mom, parts=L.particles(pos.shape[0], pos, mom, mass0=MASS, gamma0=GAMMA), t=0,
                     cp=L.couple_params(n_substeps=NSUB, dt=DT, seed=seed + 5, kernel=case["phi"], overlap=case["overlap"], **more))
    if kind == "spheres":
        centres, vel, mass = _sphere_inputs(case, seed)
        state.update(pos=centres, vel=vel, sph=L.spheres(case["n"], centres, vel, case["radius"], mass0=mass))
        L.lb_spheres_place(box.h, state["sph"])
    if kind == "moments":
        L.lb_step(box.h, 2)  # a state with stresses in it
        r = shape[::-1]
        state["out"] = [torch.zeros(*s, dtype=torch.float32, device="cuda") for s in (r, (3,) + r, (6,) + r)]
    torch.cuda.synchronize()  # rho and u may go
    return state


class _BatchOwner:
    def __init__(self, b):
        self.b = b

    def __del__(self):
        L.lb_batch_destroy(self.b)


def _sphere_inputs(case, seed):
    rad = case["radius"]
    centres = inputs.sphere_centres(case["n"], _shape(case), rad, seed=seed % (1 << 31))
    vel = np.random.default_rng(seed + 1).normal(0.0, 0.01, (case["n"], 3))
    return torch.as_tensor(centres).cuda(), torch.as_tensor(vel).cuda(), 4.0 / 3.0 * math.pi * rad ** 3


# ---- one pass --------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        L.lb_step(state["box"].h, case["steps"])
        return state["box"].state()
    if kind in ("chains", "free"):
        state["cp"].md_step0 = (NSUB * state["t"]) & 0xffffffff
        state["t"] += 1
        L.lb_couple_particles(state["box"].h, state["parts"], state["cp"])
        L.lb_step(state["box"].h, 1)
        return {"populations": state["box"].state(), "positions": state["pos"], "momenta": state["mom"]}
    if kind == "adjoint":
        state["lat"].init_equilibrium()
        theta, (lo, hi) = state["theta"], state["lo_hi"]
        theta.grad = None
        loss = ADJ.kinetic_energy(theta, state["lat"], case["steps"], lo, hi, case["every"]).to(theta.dtype)
        loss.backward()
        return {"loss": loss.detach(), "gradient": theta.grad}
    if kind == "coupled":
        state["lat"].init_equilibrium()
        theta, (lo, hi) = state["theta"], state["lo_hi"]
        theta.grad = None
        pos, mom = state["pos"].clone().requires_grad_(True), state["mom"].clone().requires_grad_(True)
        loss = ADJ.coupled_kinetic_energy(theta, pos, mom, state["lat"], state["cp"], case["steps"], lo, hi, mass0=MASS,
                                          gamma0=GAMMA, checkpoint_every=case["every"]).to(theta.dtype)
        loss.backward()
        return {"loss": loss.detach(), "gradient": theta.grad, "positions": pos.grad.float(), "momenta": mom.grad}
    if kind == "batch":
        L.lb_batch_step(state["b"].b, case["steps"], True)
        state["cur"] ^= case["steps"] & 1
        return state["bufs"][state["cur"]]
    if kind == "moments":
        rho, j, pi = state["out"]
        L.lb_moments(state["box"].h, rho, j, pi)
        return {"rho": rho, "j": j, "pi": pi}
    L.lb_step_spheres(state["box"].h, state["sph"])
    return {"populations": state["box"].state(), "centres": state["pos"], "velocities": state["vel"]}


def work(case):
    """Bytes: the state read and written in every step where two copies of it
    exceed the L2 (smaller ones could stay on the chip: once a pass), plus the
    other inputs and outputs once.  Flops: per node and step 190 for the two
    moment transforms, 110 for the relaxation and, with noise, 350 for the
    counter generator and the Gaussians."""
    kind = case["kind"]
    steps = case.get("steps", 1)
    es = {"f32": 4, "f16": 2, "bf16": 2}[case.get("dtype", "f32")]
    if kind == "batch":
        nodes = sum(a * b * c for a, b, c in _batch_shapes(case))
    else:
        nx, ny, nz = _shape(case)
        nodes = nx * ny * (nz - 2 * int(_physics(case)["walls"]))
    state = 2 * 19 * es * nodes
    times = steps if state > L2_BYTES else 1
    noisy = kind in ("batch",) or _physics(case)["kT"] > 0
    flops = nodes * steps * (300 + (350 if noisy else 0) + (600 if case.get("exponential") else 0))
    if kind == "moments":
        return {"bytes": nodes * (19 * es + 40), "flops": nodes * 150}
    if kind in ("adjoint", "coupled"):  # the field in, its gradient out; forward, recompute, reverse
        more = 48 * case.get("n", 0)
        return {"bytes": 24 * nodes + more, "flops": 3 * flops}
    n = case.get("n", 0) if kind == "free" else case.get("chains", 0) * case.get("length", 0)
    return {"bytes": state * times + (12 * nodes if case.get("field") else 0) + 72 * n, "flops": flops + 2000 * n * NSUB}


# ---- the method in 64 bits ---------------------------------------------------------

_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (1, -1, 0), (-1, 1, 0), (-1, -1, 0), (0, 1, 1), (0, 1, -1), (0, -1, 1), (0, -1, -1),
      (1, 0, 1), (1, 0, -1), (-1, 0, 1), (-1, 0, -1)]
_A = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
_OPP = [_C.index((-a, -b, -c)) for a, b, c in _C]


def _basis():
    rows = []
    for x, y, z in _C:
        c2 = x * x + y * y + z * z
        rows.append([1, x, y, z, c2 - 1, 3 * x * x - c2, y * y - z * z, x * y, y * z, z * x,
                     (3 * c2 - 5) * x, (3 * c2 - 5) * y, (3 * c2 - 5) * z,
                     (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z,
                     3 * c2 * c2 - 6 * c2 + 1, (2 * c2 - 3) * (3 * x * x - c2), (2 * c2 - 3) * (y * y - z * z)])
    return np.array(rows, dtype=np.float64).T  # [k][i]


_E = _basis()
_W = (_E ** 2) @ np.array(_A)


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors / ints holding 32-bit words."""
    m = 0xffffffff
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # wraps modulo 2^64
        c0, c1, c2, c3 = ((p1 >> 32) & m) ^ c1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ c3 ^ k1, p0 & m
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1, c2, c3


def _normal_pair(a, b):
    v1 = (2.0 * (a >> 9).double() + 1.0) / 16777216.0
    v2 = (2.0 * (b >> 9).double() + 1.0) / 16777216.0
    r = torch.sqrt(-2.0 * torch.log(v1))
    return r * torch.cos(2.0 * math.pi * v2), r * torch.sin(2.0 * math.pi * v2)


class Exact:
    """Boxes [..., nz, ny, nx] in FP64: populations as deviations n_i - a_i
    rho0 (rho0 = 1), [19][...]; a leading replica axis may stand before nz."""

    def __init__(self, shape, kw, seed, replica=0):
        self.nx, self.ny, self.nz = shape
        self.kT, self.walls = kw["kT"], kw["walls"]
        self.body, self.exponential = kw["body_force"], kw["equilibrium"]
        g = [kw.get("gamma_" + k, 0.0) for k in ("bulk", "shear", "odd", "even")]
        self.gamma = [1.0] * 4 + [g[0]] + [g[1]] * 5 + [g[2]] * 6 + [g[3]] * 3
        self.seed, self.replica = seed, replica

    def equilibrium(self, rho, u):
        out = []
        u2 = (u * u).sum(0)
        for i, c in enumerate(_C):
            cu = u[0] * c[0] + u[1] * c[1] + u[2] * c[2]
            out.append(_A[i] * (rho - 1.0) + _A[i] * rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * u2))
        return torch.stack(out)

    def equilibrium_exp(self, rho, u):
        c = torch.tensor(_C, dtype=torch.float64, device=u.device)
        a = torch.tensor(_A, dtype=torch.float64, device=u.device)
        uf = u.reshape(3, -1)
        lam = 3.0 * uf
        for _ in range(8):
            w = a[:, None] * torch.exp(c @ lam)
            w = w / w.sum(0)
            m = c.T @ w
            cov = torch.einsum("ia,ib,is->sab", c, c, w) - torch.einsum("as,bs->sab", m, m)
            lam = lam + torch.linalg.solve(cov, (uf - m).T).T
        w = a[:, None] * torch.exp(c @ lam)
        w = w / w.sum(0)
        return (rho.reshape(-1) * w - a[:, None]).reshape((19,) + rho.shape)

    def pull(self, dev, z0, z1):
        zs = torch.arange(z0, z1, device=dev.device)
        out = []
        for i, c in enumerate(_C):
            v = dev[i].index_select(-3, (zs - c[2]) % self.nz)
            v = torch.roll(v, (c[1], c[0]), (-2, -1))
            if self.walls and c[2]:
                solid = (zs - c[2] == 0) | (zs - c[2] == self.nz - 1)
                v = torch.where(solid[:, None, None], dev[_OPP[i]].index_select(-3, zs), v)
            out.append(v)
        return torch.stack(out)

    def _force(self, field, like, z0, z1):
        f = torch.zeros((3,) + like.shape, dtype=torch.float64, device=like.device)
        f = f + torch.tensor(self.body, dtype=torch.float64, device=like.device).view(3, *([1] * like.dim()))
        return f if field is None else f + field[..., z0:z1, :, :]

    def moments(self, dev, field, z0, z1):
        """rho, j (with the half force), the pulled deviations and the force."""
        n = self.pull(dev, z0, z1)
        f = self._force(field, n[0], z0, z1)
        rho = 1.0 + n.sum(0)
        j = torch.stack([sum(n[i] * c[d] for i, c in enumerate(_C) if c[d]) for d in range(3)]) + 0.5 * f
        return rho, j, n, f

    def noise(self, step, z0, z1, device):
        node = torch.arange(z0 * self.ny * self.nx, z1 * self.ny * self.nx, device=device).view(z1 - z0, self.ny, self.nx)
        k0, k1 = self.seed & 0xffffffff, self.seed >> 32
        g = []
        for b in range(4):
            w = _philox(node, step, b, self.replica, k0, k1)
            g += [*_normal_pair(w[0], w[1]), *_normal_pair(w[2], w[3])]
        return g[:15]

    def collide(self, rho, j, n, f, r):
        u = j / rho
        eq = self.equilibrium_exp(rho, u) if self.exponential else self.equilibrium(rho, u)
        neq = n - eq
        uf = (u * f).sum(0)
        gs, gb = self.gamma[5], self.gamma[4]
        sig = {}
        for a in range(3):
            for b in range(3):
                s = 0.5 * (1.0 + gs) * (u[a] * f[b] + u[b] * f[a])
                if a == b:
                    s = s - (1.0 + gs) * uf / 3.0 + (1.0 + gb) * uf / 3.0
                sig[a, b] = s
        amp = torch.sqrt(3.0 * self.kT * rho) if r is not None else None
        ms = []
        for k in range(19):
            m = 0.0
            if self.gamma[k]:
                m = self.gamma[k] * sum(float(_E[k, i]) * neq[i] for i in range(19) if _E[k, i])
            if r is not None and k >= 4:
                m = m + math.sqrt((1.0 - self.gamma[k] ** 2) * _W[k]) * amp * r[k - 4]
            ms.append(m)
        out = []
        for i, c in enumerate(_C):
            s = eq[i]
            t = sum((float(_E[k, i] / _W[k]) * ms[k] for k in range(19) if _E[k, i] and not isinstance(ms[k], float)), 0.0)
            fc = f[0] * c[0] + f[1] * c[1] + f[2] * c[2]
            sc = sum(sig[a, b] * (c[a] * c[b] - (1 / 3 if a == b else 0.0)) for a in range(3) for b in range(3))
            out.append(s + _A[i] * (t + 3.0 * fc + 4.5 * sc))
        return torch.stack(out)

    def step(self, dev, step, field=None, slab=None):
        lo, hi = (1, self.nz - 1) if self.walls else (0, self.nz)
        slab = slab or max(1, int(3e6 * self.nz / (dev[0].numel())))
        parts = []
        for z0 in range(lo, hi, slab):
            z1 = min(hi, z0 + slab)
            rho, j, n, f = self.moments(dev, field, z0, z1)
            r = self.noise(step, z0, z1, dev.device) if self.kT > 0 else None
            parts.append(self.collide(rho, j, n, f, r))
        if self.walls:
            parts = [dev[..., :1, :, :]] + parts + [dev[..., -1:, :, :]]
        return parts[0] if len(parts) == 1 else torch.cat(parts, -3)

    def velocity(self, dev, field=None):
        slab = max(1, int(6e6 / (self.ny * self.nx)))
        out = []
        for z0 in range(0, self.nz, slab):
            z1 = min(self.nz, z0 + slab)
            rho, j, _, _ = self.moments(dev, field, z0, z1)
            u = j / rho
            if self.walls:
                zs = torch.arange(z0, z1, device=dev.device)
                u = torch.where(((zs == 0) | (zs == self.nz - 1))[:, None, None], torch.zeros_like(u), u)
            out.append(u)
        return torch.cat(out, -3).reshape(3, -1)

    # -- particles ----------------------------------------------------------------

    def stencil(self, pos, phi):
        dims = (self.nx, self.ny, self.nz)
        first = torch.floor(pos + 0.5) - 1 if phi == 3 else torch.floor(pos) - (1 if phi == 4 else 0)
        w, idx = [], []
        for d in range(3):
            wd, jd = [], []
            for q in range(phi):
                jq = first[:, d].detach() + q
                v = jq - pos[:, d]
                a = v.abs()
                if phi == 2:
                    t = 1.0 - a
                elif phi == 3:
                    near = (1.0 + torch.sqrt((1.0 - 3.0 * v * v).clamp(min=0.0))) / 3.0
                    far = (5.0 - 3.0 * a - torch.sqrt((-2.0 + 6.0 * a - 3.0 * v * v).clamp(min=0.0))) / 6.0
                    t = torch.where(a <= 0.5, near, far)
                else:
                    near = (3.0 - 2.0 * a + torch.sqrt((1.0 + 4.0 * a - 4.0 * v * v).clamp(min=0.0))) / 8.0
                    far = (5.0 - 2.0 * a - torch.sqrt((-7.0 + 12.0 * a - 4.0 * v * v).clamp(min=0.0))) / 8.0
                    t = torch.where(a <= 1.0, near, far)
                wd.append(t)
                jd.append(jq.long() % dims[d])
            w.append(wd)
            idx.append(jd)
        wt, node = [], []
        for z in range(phi):
            for y in range(phi):
                for x in range(phi):
                    wt.append(w[0][x] * w[1][y] * w[2][z])
                    node.append((idx[2][z] * self.ny + idx[1][y]) * self.nx + idx[0][x])
        return torch.stack(wt), torch.stack(node)

    def confine(self, pos, mom, phi):
        cols, mz = [], mom[:, 2]
        for d, size in enumerate((self.nx, self.ny, self.nz)):
            p = pos[:, d]
            if d == 2 and self.walls:
                for edge, out in ((0.5 * phi, lambda v, e: v < e), (self.nz - 1 - 0.5 * phi, lambda v, e: v > e)):
                    hit = out(p, edge)
                    p, mz = torch.where(hit, 2.0 * edge - p, p), torch.where(hit, -mz, mz)
            else:
                p = p - size * torch.floor(p.detach() / size)
            cols.append(p)
        return torch.stack(cols, 1), torch.cat([mom[:, :2], mz[:, None]], 1)

    def chain_forces(self, pos, length):
        box = torch.tensor([self.nx, self.ny, self.nz], dtype=torch.float64, device=pos.device)
        force = torch.zeros_like(pos)
        for k in range(0, pos.shape[0], 2048):
            d = pos[k:k + 2048, None] - pos[None]
            d -= box * torch.floor(d / box + 0.5)
            r2 = (d * d).sum(-1)
            i = torch.arange(k, k + r2.shape[0], device=pos.device)
            r2[i - k, i] = 1e9
            s6 = (SIGMA * SIGMA / r2) ** 3
            mag = torch.where(r2 < 2.0 ** (1 / 3) * SIGMA ** 2, 24.0 * EPS * (2.0 * s6 * s6 - s6) / r2, torch.zeros_like(r2))
            force[k:k + 2048] = (mag[..., None] * d).sum(1)
        d = pos[1:] - pos[:-1]
        d -= box * torch.floor(d / box + 0.5)
        bond = (-K_FENE / (1.0 - (d * d).sum(-1, keepdim=True) / R0 ** 2)) * d
        bond[length - 1::length] = 0.0
        force[1:] += bond
        force[:-1] -= bond
        return force

    def couple(self, dev, pos, mom, phi, seed, md_step0, field=None, length=0):
        u = self.velocity(dev, field)
        n = pos.shape[0]
        c1 = math.exp(-GAMMA * DT / MASS)
        c2 = MASS / GAMMA * (1.0 - c1)
        c3 = math.sqrt(MASS * self.kT * (1.0 - math.exp(-2.0 * GAMMA * DT / MASS)))
        acc = torch.zeros(3, u.shape[1], dtype=torch.float64, device=pos.device)
        for s in range(NSUB):
            pos, mom = self.confine(pos + 0.5 * DT / MASS * mom, mom, phi)
            fc = self.chain_forces(pos, length) if length > 1 else 0.0
            wt, node = self.stencil(pos, phi)
            up = (wt * u[:, node]).sum(1).T
            new = c1 * mom + c2 * (fc + GAMMA * up)
            if self.kT > 0:
                w = _philox(torch.arange(n, device=pos.device), md_step0 + s, 1 << 8, 0, seed & 0xffffffff, seed >> 32)
                g0, g1 = _normal_pair(w[0], w[1])
                g2, _ = _normal_pair(w[2], w[3])
                new = new + c3 * torch.stack([g0, g1, g2], 1)
            jmp = new - mom - DT * fc
            acc = torch.stack([acc[d].index_add(0, node.reshape(-1), -(wt * jmp[:, d]).reshape(-1)) for d in range(3)])
            mom = new
            pos, mom = self.confine(pos + 0.5 * DT / MASS * mom, mom, phi)
        return pos, mom, acc.view(3, self.nz, self.ny, self.nx)


def _initial(ref, case, gen):
    rho, u = _flow(_shape(case), ref.kT, gen, _amplitude(case))
    return ref.equilibrium(rho, u)


def _trim(ref, dev):
    """As the buffers hold it: FP16 / BF16 deviations are stored times 1024."""
    return (dev[:, 1:-1] if ref.walls else dev).reshape(19, -1)


def _field(case, gen):
    return 1e-5 * torch.randn(3, *_shape(case)[::-1], generator=gen, device="cuda", dtype=torch.float32)


def _kinetic(ref, dev, field, lo, hi):
    rho, j, _, _ = ref.moments(dev, field, 0, ref.nz)
    e = 0.5 * (j * j).sum(0) / rho
    return e[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]].sum()


def exact(case, seed):
    kind = case["kind"]
    gen = _generator(seed)
    if kind in ("adjoint", "coupled"):
        return _exact_gradient(case, gen)
    with torch.no_grad():
        if kind == "batch":
            return _exact_batch(case, seed, gen)
        ref = Exact(_shape(case), _physics(case), seed)
        scale = 1.0 if case.get("dtype", "f32") == "f32" else 1024.0
        if kind == "spheres":
            return _exact_spheres(case, seed, ref, gen)
        field = _field(case, gen).double() if case.get("field") else None
        dev = _initial(ref, case, gen)
        if kind == "step":
            for t in range(case["steps"]):
                dev = ref.step(dev, t, field)
            return scale * _trim(ref, dev)
        if kind == "moments":
            for t in range(2):
                dev = ref.step(dev, t)
            return _exact_moments(ref, dev)
        walls = ref.walls
        pos = _chain_positions(case, gen) if kind == "chains" else _free_positions(case, gen, walls)
        mom = _momenta(pos.shape[0], ref.kT, gen).double()
        pos, mom, acc = ref.couple(dev, pos, mom, case["phi"], seed + 5, 0, None, case.get("length", 0))
        dev = ref.step(dev, 0, acc)
        return {"populations": scale * _trim(ref, dev), "positions": pos, "momenta": mom}


def _exact_moments(ref, dev):
    rhos, js, pis = [], [], []
    slab = max(1, int(6e6 / (ref.ny * ref.nx)))
    for z0 in range(0, ref.nz, slab):
        z1 = min(ref.nz, z0 + slab)
        rho, j, n, _ = ref.moments(dev, None, z0, z1)
        pi = []
        for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (2, 0)):
            base = 1 / 3 if a == b else 0.0
            pi.append(base + sum(n[i] * (c[a] * c[b]) for i, c in enumerate(_C) if c[a] * c[b]))
        if ref.walls:
            zs = torch.arange(z0, z1, device=dev.device)
            solid = ((zs == 0) | (zs == ref.nz - 1))[:, None, None]
            rho = torch.where(solid, torch.ones_like(rho), rho)
            j = torch.where(solid, torch.zeros_like(j), j)
            pi = [torch.where(solid, torch.zeros_like(p), p) for p in pi]
        rhos.append(rho)
        js.append(j)
        pis.append(torch.stack(pi))
    return {"rho": torch.cat(rhos, -3), "j": torch.cat(js, -3), "pi": torch.cat(pis, -3)}


def _exact_batch(case, seed, gen):
    shapes = _batch_shapes(case)
    kw = {"kT": KT, "walls": False, "body_force": (0.0, 0.0, 0.0), "equilibrium": 0}
    pitch = [(a * b * c + 63) // 64 * 64 for a, b, c in shapes]
    out = torch.zeros(19 * sum(pitch), dtype=torch.float64, device="cuda")
    flows = [_flow(s, KT, gen) for s in shapes]
    off = np.concatenate([[0], np.cumsum([19 * p for p in pitch])])
    for s in sorted(set(shapes)):
        reps = [r for r, t in enumerate(shapes) if t == s]
        many = lambda v: torch.tensor(v, device="cuda").view(-1, 1, 1, 1)  # noqa: E731
        ref = Exact(s, kw, many([seed + r for r in reps]), many(reps))
        rho, u = torch.stack([flows[r][0] for r in reps]), torch.stack([flows[r][1] for r in reps], 1)
        dev = ref.equilibrium(rho, u)
        for t in range(case["steps"]):
            dev = ref.step(dev, t)
        for q, r in enumerate(reps):
            nodes = s[0] * s[1] * s[2]
            out[off[r]:off[r + 1]].view(19, pitch[r])[:, :nodes] = dev[:, q].reshape(19, -1)
    return out


def _exact_gradient(case, gen):
    from torch.utils.checkpoint import checkpoint
    nx, ny, nz = _shape(case)
    ref = Exact((nx, ny, nz), _physics(case), 0)
    field = _field(case, gen).double().requires_grad_(True)
    lo, hi = _sub_box((nx, ny, nz))
    dev = torch.zeros(19, nz, ny, nx, dtype=torch.float64, device="cuda")
    if case["kind"] == "adjoint":
        for t in range(case["steps"]):
            dev = checkpoint(lambda d, f: ref.step(d, 0, f, slab=nz), dev, field, use_reentrant=False)
        loss = _kinetic(ref, dev, field, lo, hi)
        return {"loss": loss.detach(), "gradient": torch.autograd.grad(loss, field)[0]}
    pos0 = _free_positions(case, gen, False).requires_grad_(True)
    mom0 = _momenta(case["n"], 0.0, gen).double().requires_grad_(True)
    pos, mom = pos0, mom0

    def advance(d, f, p, m):
        p, m, acc = ref.couple(d, p, m, 2, 0, 0, f)
        return ref.step(d, 0, f + acc, slab=nz), p, m

    for t in range(case["steps"]):
        dev, pos, mom = checkpoint(advance, dev, field, pos, mom, use_reentrant=False)
    loss = _kinetic(ref, dev, field, lo, hi)
    g = torch.autograd.grad(loss, (field, pos0, mom0))
    return {"loss": loss.detach(), "gradient": g[0], "positions": g[1], "momenta": g[2]}


def _exact_spheres(case, seed, ref, gen):
    """The spheres' motion; the populations come without a value (those of solid nodes mean nothing)."""
    dev = _initial(ref, case, gen)
    pos, vel, mass = _sphere_inputs(case, seed)
    n, a = case["n"], case["radius"]
    dims = torch.tensor(_shape(case), dtype=torch.float64, device="cuda")
    half = pos + 0.5 * vel
    half = half - dims * torch.floor(half / dims)
    reach = int(math.ceil(a)) + 2

    def near(centre):
        """Nodes around each centre: linear index [n][...], offset from the centre [n][...][3]."""
        k = torch.arange(-reach, reach + 1, device="cuda", dtype=torch.float64)
        cube = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).view(1, -1, 3)
        at = torch.floor(centre)[:, None] + cube
        d = at - centre[:, None]
        w = (at % dims).long()
        return (w[..., 2] * ref.ny + w[..., 1]) * ref.nx + w[..., 0], d

    def solid_map(centre):
        idx, d = near(centre)
        m = torch.full((ref.nz * ref.ny * ref.nx,), -1, dtype=torch.long, device="cuda")
        inside = (d * d).sum(-1) < a * a
        owner = torch.arange(n, device="cuda")[:, None].expand_as(idx)
        m[idx[inside]] = owner[inside]
        return m

    old, new = solid_map(pos), solid_map(half)
    flat = dev.reshape(19, -1)
    c = torch.tensor(_C, dtype=torch.float64, device="cuda")
    w = torch.tensor(_A, dtype=torch.float64, device="cuda")
    dp = torch.zeros(n, 3, dtype=torch.float64, device="cuda")
    covered = ((old < 0) & (new >= 0)).nonzero()[:, 0]
    dp.index_add_(0, new[covered], (c.T @ flat[:, covered]).T)
    bare = ((old >= 0) & (new < 0)).nonzero()[:, 0]
    ub = vel[old[bare]]
    flat[:, bare] = ref.equilibrium(torch.ones(bare.numel(), dtype=torch.float64, device="cuda"), ub.T)
    dp.index_add_(0, old[bare], -ub)
    vel = vel + dp / mass
    box = new.view(ref.nz, ref.ny, ref.nx)
    f0 = torch.zeros(n, 3, dtype=torch.float64, device="cuda")
    zeta = torch.zeros(n, 3, 3, dtype=torch.float64, device="cuda")
    for i in range(1, 19):
        to = torch.roll(box, (-_C[i][2], -_C[i][1], -_C[i][0]), (0, 1, 2)).reshape(-1)
        s = ((new < 0) & (to >= 0)).nonzero()[:, 0]
        f0.index_add_(0, to[s], 2.0 * (flat[i, s] + w[i])[:, None] * c[i])
        zeta.index_add_(0, to[s], (6.0 * w[i] * c[i][:, None] * c[i]).expand(s.numel(), 3, 3))
    lam, q = torch.linalg.eigh(zeta)
    ue, fe = (q.mT @ vel[..., None])[..., 0], (q.mT @ f0[..., None])[..., 0]
    e1 = -torch.expm1(-lam / mass)
    vel = (q @ ((1.0 - e1) * ue + e1 * fe / lam)[..., None])[..., 0]
    end = half + 0.5 * vel
    return {"populations": None, "centres": end - dims * torch.floor(end / dims), "velocities": vel}
