"""Timed cases of the library: the work its users have it do, through its
public entry points.

Four kinds of program are covered:

* ``steps``: a program advances a lattice that is already running and keeps
  the populations on the device.  It owns the device memory (the library's
  allocator callbacks hand out its tensors), so the populations are at hand
  without a copy.  FP32 populations lie in the pull layout that
  ``elbm_step_static`` documents: entry [i][x] is the post-collision f_i(x)
  minus W_i rho0.
* ``static``: one step of a latency-critical loop on the caller's buffers
  (``elbm_step_static``).
* ``batch``: many lattices of mixed type and size advanced together, as the
  server does between admissions.
* ``run``: a whole request: host fields in, steps with their diagnostics read
  back on the way, density and velocity out, kept in single precision.

``exact`` restates the method in torch with 64-bit arithmetic: entropic
product-form equilibrium, alpha by the formula, the bisection or the secant
iteration, relaxation, periodic streaming.
"""
import ctypes
import math
import random

import numpy as np
import torch

import paper_1904_00866_gb300 as elbm

DEV = "cuda"
DIM = {"D2Q9": 2, "D3Q27": 3}


def _velocities(lattice):
    """Velocity set in the library's order: rest, faces, edges, corners, each
    followed by its opposite."""
    if lattice == "D2Q9":
        half = [(1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0)]
    else:
        half = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0),
                (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1), (1, 1, 1),
                (1, 1, -1), (1, -1, 1), (-1, 1, 1)]
    out = [(0, 0, 0)]
    for c in half:
        out += [c, tuple(-a for a in c)]
    return out


def _weights(lattice):
    d = DIM[lattice]
    return [(2 / 3) ** (d - k) * (1 / 6) ** k
            for k in (sum(map(abs, c)) for c in _velocities(lattice))]


# --------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------
def _case(name, kind, lattice, n, dtype, flow, nu, **more):
    nx, ny, nz = (tuple(n) + (1,))[:3]
    case = {"kind": kind, "lattice": lattice, "nx": nx, "ny": ny, "nz": nz,
            "dtype": dtype, "mode": "formula", "decision": "exact",
            "flow": flow, "nu": nu, "warm": 4, "steps": 1, "diag_every": 1,
            "alpha_map": False}
    case.update(more)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # The plain method at the size a CPU run can check: 1000-step
        # Taylor-Green decay in FP64, statistics on every step (the default
        # schedule).  Smallest call: launches and latency.
        _case("d2q9_64_fp64", "steps", "D2Q9", (64, 64), "fp64", "tgv", 0.01,
              steps=50),
        # The smallest 3D lattice the server admits, stepped on its own.
        _case("d3q27_32_fp32", "steps", "D3Q27", (32, 32, 32), "fp32_shifted",
              "modes", 1e-3, steps=50),
        # Thin double shear layer at Re 30,000: FP32 populations, the alpha
        # map dumped now and then.  Most nodes lie within FP32 rounding of
        # equilibrium.
        _case("d2q9_shear_1024_fp32", "steps", "D2Q9", (1024, 1024),
              "fp32_shifted", "shear", 0.04 * 1024 / 3e4, steps=50,
              diag_every=10, alpha_map=True),
        # Its FP64 reference run.
        _case("d2q9_shear_1024_fp64", "steps", "D2Q9", (1024, 1024), "fp64",
              "shear", 0.04 * 1024 / 3e4, steps=4, diag_every=10),
        # The same flow with alpha from the bisection root, the method the
        # formula is compared with.
        _case("d2q9_shear_1024_fp32_root", "steps", "D2Q9", (1024, 1024),
              "fp32_shifted", "shear", 0.04 * 1024 / 3e4, mode="root",
              steps=2, diag_every=10),
        # The headline: Taylor-Green vortex at Re 1600 on 512^3.
        _case("d3q27_tgv_512_fp32", "steps", "D3Q27", (512, 512, 512),
              "fp32_shifted", "tgv", 0.05 * 512 / (2 * math.pi) / 1600,
              steps=8, warm=2, diag_every=10),
        # A ragged box of ordinary size with the default schedule.
        _case("d3q27_ragged_fp32", "steps", "D3Q27", (189, 107, 83),
              "fp32_shifted", "modes", 5e-4, steps=20),
        # Binary16 storage, for lattices FP32 could not hold.
        _case("d3q27_tgv_256_fp16", "steps", "D3Q27", (256, 256, 256),
              "fp16_shifted", "tgv", 0.05 * 256 / (2 * math.pi) / 1600,
              steps=8, diag_every=10),
        # FP64 reference run of a 3D flow.
        _case("d3q27_tgv_128_fp64", "steps", "D3Q27", (128, 128, 128), "fp64",
              "tgv", 0.05 * 128 / (2 * math.pi) / 1600, steps=4,
              diag_every=10),
        # Twelve mixed lattices between two admissions of the server: two
        # bursts of sixteen steps.
        _case("batch_mix_12", "batch", "mixed", (512, 96, 1), "fp32_shifted",
              "modes", 1e-3, members=12, steps=32, warm=16, diag_every=0),
        # One step of a loop that owns its buffers and may not allocate.
        _case("static_d3q27_step", "static", "D3Q27", (121, 64, 70),
              "fp32_shifted", "modes", 1e-3, warm=2, alpha_map=True),
        # A whole request: fields from the host, 60 steps with statistics
        # read every 20, density and velocity back.
        _case("run_d3q27_96", "run", "D3Q27", (96, 96, 96), "fp32_shifted",
              "modes", 1e-3, warm=0, steps=60, diag_every=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lattice, lo, hi):
    """A ragged box of lo..hi nodes (log-uniform) with edges within a factor
    of two of each other."""
    d = DIM[lattice]
    edge = math.exp(rng.uniform(math.log(lo), math.log(hi)) / d)
    return tuple(max(8, int(edge * 2 ** rng.uniform(-0.5, 0.5) / 1.2))
                 for _ in range(d))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["fp32", "fp32", "fp16", "fp64", "fp64mode", "batch",
                       "static", "run"])
    lattice = rng.choice(["D2Q9", "D3Q27"])
    nu = 10 ** rng.uniform(-5, -2)
    flow = "modes"
    if lattice == "D2Q9" and rng.random() < 0.3:
        flow = "shear"
    elif rng.random() < 0.3:
        flow = "tgv"
    more = {"diag_every": rng.choice([1, 1, 10, 0])}
    if kind in ("fp32", "fp16"):
        n = _box(rng, lattice, 4e3, 4e6 if lattice == "D2Q9" else 4e7)
        nodes = math.prod(n)
        dtype = "fp16_shifted" if kind == "fp16" else rng.choice(
            ["fp32_shifted", "fp32_shifted", "fp32"])
        return _case(None, "steps", lattice, n, dtype, flow, nu,
                     steps=max(3, min(50, int(4e8 / nodes))),
                     decision=rng.choice(["exact", "exact", "certified"]),
                     alpha_map=rng.random() < 0.25, **more)
    if kind == "fp64":
        n = _box(rng, lattice, 2e3, 2e6)
        return _case(None, "steps", lattice, n, "fp64", flow, nu,
                     steps=max(2, min(50, int(4e6 / math.prod(n)))), **more)
    if kind == "fp64mode":   # root / secant on any storage
        n = _box(rng, lattice, 2e3, 1e6 if lattice == "D2Q9" else 2e5)
        return _case(None, "steps", lattice, n,
                     rng.choice(["fp64", "fp32_shifted", "fp16_shifted"]),
                     flow, nu, mode=rng.choice(["root", "secant"]),
                     steps=max(2, min(20, int(1e6 / math.prod(n)))), **more)
    if kind == "batch":
        return _case(None, "batch", "mixed",
                     (_log_int(rng, 128, 700), _log_int(rng, 40, 110), 1),
                     "fp32_shifted", "modes", nu,
                     members=rng.randint(2, 16), steps=16 * rng.randint(1, 2),
                     warm=16, diag_every=0)
    if kind == "static":
        n = _box(rng, lattice, 4e3, 1.2e6)
        return _case(None, "static", lattice, n, "fp32_shifted", flow, nu,
                     warm=2, alpha_map=rng.random() < 0.5)
    n = _box(rng, lattice, 4e3, 1.5e6)
    every = rng.choice([5, 10, 20])
    return _case(None, "run", lattice, n,
                 rng.choice(["fp32_shifted", "fp32_shifted", "fp16_shifted"]),
                 flow, nu, warm=0, steps=every * rng.randint(2, 4),
                 diag_every=every)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _fields(flow, lattice, shape, seed):
    """Density (nz, ny, nx) and velocity (d, nz, ny, nx), FP64, on the GPU."""
    rng = random.Random(seed)
    nz, ny, nx = shape
    d = DIM[lattice]
    axis = [2 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n
            for n in (nx, ny, nz)]
    X = axis[0].view(1, 1, nx) + rng.uniform(0, 2 * math.pi)
    Y = axis[1].view(1, ny, 1) + rng.uniform(0, 2 * math.pi)
    Z = axis[2].view(nz, 1, 1) + rng.uniform(0, 2 * math.pi)
    u = torch.empty((d,) + tuple(shape), device=DEV, dtype=torch.float64)
    rho = torch.ones(tuple(shape), device=DEV, dtype=torch.float64)
    u0 = 0.05 * rng.uniform(0.9, 1.0)
    if flow == "shear":
        # double shear layer: width parameter 80, velocity 0.04, transverse
        # perturbation 2e-3
        y = (axis[1] / (2 * math.pi)).view(1, ny, 1)
        u0 = 0.04 * rng.uniform(0.95, 1.05)
        u[0] = torch.where(y <= 0.5, u0 * torch.tanh(80 * (y - 0.25)),
                           u0 * torch.tanh(80 * (0.75 - y)))
        u[1] = 2e-3 * torch.sin(X)
        if d == 3:
            u[2] = 0.0
    elif flow == "tgv" and d == 2:
        u[0] = -u0 * torch.cos(X) * torch.sin(Y)
        u[1] = u0 * torch.sin(X) * torch.cos(Y)
        rho -= 0.75 * u0 ** 2 * (torch.cos(2 * X) + torch.cos(2 * Y))
    elif flow == "tgv":
        u[0] = u0 * torch.sin(X) * torch.cos(Y) * torch.cos(Z)
        u[1] = -u0 * torch.cos(X) * torch.sin(Y) * torch.cos(Z)
        u[2] = 0.0
        rho += 3 * u0 ** 2 / 16 * (torch.cos(2 * X) + torch.cos(2 * Y)) * (
            torch.cos(2 * Z) + 2)
    else:
        # low-mode flow: shear waves along each axis, modes 1..4
        a = [rng.uniform(0.5, 1.5) for _ in range(3)]
        k = [rng.randint(1, 4) for _ in range(3)]
        if d == 2:
            u[0] = (a[0] * torch.sin(k[0] * Y)
                    + a[2] * torch.cos(k[2] * Y)).expand(shape)
            u[1] = (a[1] * torch.sin(k[1] * X)).expand(shape)
        else:
            u[0] = a[0] * torch.sin(k[0] * Z) + a[2] * torch.cos(k[2] * Y)
            u[1] = a[1] * torch.sin(k[1] * X) + a[0] * torch.cos(k[0] * Z)
            u[2] = a[2] * torch.sin(k[2] * Y) + a[1] * torch.cos(k[1] * X)
        u *= 0.05 / u.square().sum(0).max().sqrt()
    return rho, u


def _members(case, seed):
    """The batch's members: alternately D2Q9 with edge 64..nx and D3Q27 with
    edge 32..ny, viscosity log-uniform in [1e-5, 1e-2].  Their shapes belong
    to the case, their flows to the seed."""
    rng = random.Random(case["members"] * 1009 + case["nx"] + case["ny"])
    out = []
    for k in range(case["members"]):
        lattice = "D2Q9" if k % 2 == 0 else "D3Q27"
        lo, hi = (64, case["nx"]) if k % 2 == 0 else (32, case["ny"])
        n = rng.randint(lo, max(lo, hi))
        shape = (1, n, n) if lattice == "D2Q9" else (n, n, n)
        out.append((lattice, shape, 10 ** rng.uniform(-5, -2),
                    seed * 1000 + k))
    return out


# --------------------------------------------------------------------------
# programs
# --------------------------------------------------------------------------
class _Pool:
    """A program's device memory: the library's buffers are its tensors."""

    def __init__(self):
        self.live = {}
        self.sizes = []   # (bytes, tensor) in order of allocation

        def alloc(size, ctx):
            try:
                t = torch.empty(max(int(size), 1), dtype=torch.uint8,
                                device=DEV)
            except Exception:   # no exception crosses the C ABI
                return None
            self.live[t.data_ptr()] = t
            self.sizes.append((int(size), t))
            return t.data_ptr()

        def free(ptr, ctx):
            t = self.live.pop(int(ptr), None)
            self.sizes = [s for s in self.sizes if s[1] is not t]

        self.callbacks = (elbm.ALLOC_FN(alloc), elbm.FREE_FN(free))

    def pair(self, size):
        """The first two live buffers of `size` bytes not yet handed out."""
        got = [t for s, t in self.sizes if s == size][:2]
        self.sizes = [s for s in self.sizes
                      if all(s[1] is not t for t in got)]
        return got


TYPES = {"fp64": torch.float64, "fp32": torch.float32,
         "fp32_shifted": torch.float32, "fp16_shifted": torch.float16}


def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


def _lattice(case, pool=None):
    lat = elbm.Lattice(case["lattice"], case["nx"], case["ny"], case["nz"],
                       nu=case["nu"], dtype=case["dtype"],
                       allocator="cuda" if pool else None)
    if pool:
        if elbm.lib().elbm_set_allocator(lat._h, *pool.callbacks, None):
            raise RuntimeError("elbm_set_allocator")
        lat.pool = pool   # outlives the handle
    lat.set_decision(case["decision"])
    lat.set_diagnostics(
        diag_every=case["diag_every"],
        alpha_map_every=case["steps"] if case["alpha_map"] else 0)
    return lat


def _stored(lattice, dtype, shape, buffer):
    """The populations of a buffer as [Q][nz][ny][nx]."""
    q, n = len(_velocities(lattice)), math.prod(shape)
    t = buffer.view(TYPES[dtype])
    return t.view(q, t.numel() // q)[:, :n].view((q,) + tuple(shape))


def prepare(case, seed):
    shape = _shape(case)
    if case["kind"] == "static":
        # the populations a running lattice holds
        f, rho0 = _reference(case, seed, case["warm"], True)
        f_in = f.to(torch.float32)
        return {"case": case, "f_in": f_in, "f_out": torch.empty_like(f_in),
                "rho0": rho0, "alpha": torch.empty(
                    shape, device=DEV, dtype=torch.float32)
                if case["alpha_map"] else None}
    if case["kind"] == "batch":
        pool = _Pool()
        batch = elbm.Batch(allocator="cuda", diag_every=case["diag_every"])
        if elbm.lib().elbm_batch_set_allocator(batch._h, *pool.callbacks,
                                               None):
            raise RuntimeError("elbm_batch_set_allocator")
        batch.pool = pool
        members = []
        for lattice, sh, nu, s in _members(case, seed):
            rho, u = _fields("modes", lattice, sh, s)
            mid = batch.add(lattice, sh[2], sh[1], sh[0], nu,
                            rho.cpu().numpy(), u.cpu().numpy())
            size = 4 * len(_velocities(lattice)) * math.prod(sh)
            members.append((mid, lattice, sh, pool.pair(size)))
        batch.step(case["warm"])
        batch.sync()
        return {"case": case, "batch": batch, "members": members}
    rho, u = _fields(case["flow"], case["lattice"], shape, seed)
    if case["kind"] == "run":
        return {"case": case, "lat": _lattice(case),
                "rho": rho.cpu().numpy(), "u": u.cpu().numpy()}
    pool = _Pool()
    lat = _lattice(case, pool)
    lat.init_fields(rho, u)
    q, n = len(_velocities(case["lattice"])), math.prod(shape)
    if case["dtype"] == "fp16_shifted":
        n = (n + 63) // 64 * 64
    size = TYPES[case["dtype"]].itemsize * q * n
    lat.step(case["warm"], case["mode"])
    lat.sync()
    return {"case": case, "lat": lat, "buffers": pool.pair(size)}


def run(state):
    case = state["case"]
    if case["kind"] == "static":
        alpha = state["alpha"]
        st = elbm.lib().elbm_step_static(
            elbm.LATTICES[case["lattice"]], case["nx"], case["ny"],
            case["nz"], case["nu"], state["rho0"],
            state["f_in"].data_ptr(), state["f_out"].data_ptr(),
            alpha.data_ptr() if alpha is not None else None,
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), None)
        if st:
            raise elbm.ElbmError(st, "elbm_step_static")
        return [state["f_out"]] + ([alpha] if alpha is not None else [])
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.step(case["steps"])
        return [_stored(lattice, "fp32_shifted", sh,
                        buffers[batch.info(mid)[0] & 1])
                for mid, lattice, sh, buffers in state["members"]]
    lat = state["lat"]
    if case["kind"] == "run":
        lat.init_fields(state["rho"], state["u"])
        history = []
        for _ in range(case["steps"] // case["diag_every"]):
            lat.step(case["diag_every"], case["mode"])
            s = lat.entropy_stats()
            history.append([s["mass"], *s["momentum"], s["kinetic_energy"]])
        rho, u = lat.moments()
        # the record a run keeps: fields and history in single precision
        return [torch.from_numpy(rho).float(), torch.from_numpy(u).float(),
                torch.tensor(history, dtype=torch.float32)]
    lat.step(case["steps"], case["mode"])
    out = [_stored(case["lattice"], case["dtype"], _shape(case),
                   state["buffers"][lat.step_count & 1])]
    if case["alpha_map"]:
        out.append(lat.alpha_map())
    return out


def work(case):
    """Bytes and operations of one pass.  Each step reads and writes every
    population once; per population about 30 operations for the moments,
    equilibrium and relaxation and two logarithms (about 20 each) for the
    entropy test."""
    if case["kind"] == "batch":
        nodes = [(len(_velocities(lat)), math.prod(sh))
                 for lat, sh, _, _ in _members(case, 0)]
    else:
        nodes = [(len(_velocities(case["lattice"])), math.prod(_shape(case)))]
    esz = TYPES[case["dtype"]].itemsize
    pops = sum(q * n for q, n in nodes)
    total = {"bytes": 2 * esz * pops * case["steps"],
             "flops": 70 * pops * case["steps"]}
    if case["alpha_map"]:
        total["bytes"] += 4 * sum(n for _, n in nodes)
    if case["kind"] == "run":   # FP64 fields in and out
        total["bytes"] += 16 * (1 + DIM[case["lattice"]]) * nodes[0][1]
    return total


# --------------------------------------------------------------------------
# the method in 64 bits
# --------------------------------------------------------------------------
def _equilibrium(lattice, rho, u):
    """f^eq_i = rho W_i prod_a psi_a(c_ia), psi(0) = 1 - s,
    psi(+-1) = 1 +- 3u + 2s, s = 3u^2 / (1 + sqrt(1 + 3u^2))."""
    cs, ws = _velocities(lattice), _weights(lattice)
    psi = []
    for v in u:
        s = 3 * v * v / (1 + torch.sqrt(1 + 3 * v * v))
        psi.append({0: 1 - s, 1: 1 + 3 * v + 2 * s, -1: 1 - 3 * v + 2 * s})
    out = torch.empty((len(cs),) + tuple(rho.shape), device=rho.device,
                      dtype=torch.float64)
    for i, c in enumerate(cs):
        p = rho * ws[i]
        for a in range(len(u)):
            p = p * psi[a][c[a]]
        out[i] = p
    return out


def _moments(lattice, f):
    rho = f.sum(0)
    u = []
    for a in range(DIM[lattice]):
        m = torch.zeros_like(rho)
        for i, c in enumerate(_velocities(lattice)):
            if c[a]:
                m += c[a] * f[i]
        u.append(m / rho)
    return rho, u


def _phi(y):
    """(1 + y) ln(1 + y) - y, by its series where |y| < 0.1."""
    p = torch.full_like(y, -1.0 / 272)
    for k in range(16, 1, -1):
        p.mul_(y).add_((-1.0) ** k / (k * (k - 1)))
    z = torch.clamp(1 + y, min=1e-300)
    return torch.where(y.abs() < 0.1, y * y * p, z * torch.log(z) - y)


def _alpha(f, x, mode):
    inf = torch.full_like(x, math.inf)
    amax = torch.where(x < 0, -1 / x, inf).amin(0)
    rest = torch.isinf(amax)   # equilibrium: alpha is free, 2
    L = torch.log1p(x)
    B = (f * x * L).sum(0)
    D1 = (f * (L - x)).sum(0)

    def dH(a):
        return (f * _phi(a * x)).sum(0) - a * B

    if mode == "root":
        lo, hi = torch.ones_like(amax), torch.where(rest, 2.0, amax)
        alpha = hi.clone()
        todo = ~rest & (dH(hi) > 0)
        for _ in range(64):
            mid = 0.5 * (lo + hi)
            d = dH(mid)
            done = todo & (d >= -1e-13) & (d <= 0)
            alpha = torch.where(done, mid, alpha)
            todo = todo & ~done
            hi = torch.where(todo & (d > 0), mid, hi)
            lo = torch.where(todo & ~(d > 0), mid, lo)
            done = todo & (hi - lo < 1e-15 * hi)
            alpha = torch.where(done, lo, alpha)
            todo = todo & ~done
        return torch.where(todo, lo, alpha)
    astar = torch.clamp(amax, max=2.0)
    Ds = dH(astar)
    if mode == "secant":
        a, da = torch.ones_like(astar), D1
        go = torch.ones_like(rest)
        for _ in range(4):
            an = astar + Ds / (Ds - da) * (a - astar)
            dn = dH(an)
            go = go & ~(dn > 0)
            a, da = torch.where(go, an, a), torch.where(go, dn, da)
            go = go & ~(da >= -1e-13)
    else:
        a = astar + Ds / (Ds - D1) * (1 - astar)
    a = torch.where(Ds - D1 > 0, a, torch.ones_like(a))
    a = torch.where(Ds <= 0, astar, a)
    return torch.where(rest, torch.full_like(a, 2.0), a)


def _collide(lattice, f, beta, mode):
    """Post-collision populations, in place."""
    flat = f.view(f.shape[0], -1)
    chunk = 1 << 21
    for k in range(0, flat.shape[1], chunk):
        g = flat[:, k:k + chunk]
        rho, u = _moments(lattice, g)
        x = _equilibrium(lattice, rho, u).sub_(g).div_(g)
        g += _alpha(g, x, mode) * beta * g * x


def _stream(lattice, f):
    for i, c in enumerate(_velocities(lattice)):
        if i:
            f[i] = torch.roll(f[i], (c[2], c[1], c[0]), (0, 1, 2))


def _reference(case, seed, steps, shifted):
    """Post-collision populations after `steps` steps (minus W_i rho0 when
    `shifted`) and rho0."""
    lattice = case["lattice"]
    rho, u = _fields(case["flow"], lattice, _shape(case), seed)
    rho0 = float(np.float32(rho.mean().item()))
    f = _equilibrium(lattice, rho, u)
    del rho, u
    beta = 1 / (6 * case["nu"] + 1)
    for s in range(steps):
        if s:
            _stream(lattice, f)
        _collide(lattice, f, beta, case["mode"])
    if shifted:
        for i, w in enumerate(_weights(lattice)):
            f[i] -= w * rho0
    return f, rho0


def exact(case, seed):
    """What run() returns, in 64 bits; None for the alpha map (where f is
    within rounding of f^eq any alpha is right) and for the history."""
    if case["kind"] == "static":
        s = prepare(case, seed)
        f = s["f_in"].double()
        ws = _weights(case["lattice"])
        for i, w in enumerate(ws):
            f[i] += w * s["rho0"]
        _stream(case["lattice"], f)
        _collide(case["lattice"], f, 1 / (6 * case["nu"] + 1), case["mode"])
        for i, w in enumerate(ws):
            f[i] -= w * s["rho0"]
        return [f] + ([None] if case["alpha_map"] else [])
    steps = case["warm"] + case["steps"]
    if case["kind"] == "batch":
        out = []
        for lattice, sh, nu, s in _members(case, seed):
            one = dict(case, lattice=lattice, nz=sh[0], ny=sh[1], nx=sh[2],
                       nu=nu, flow="modes")
            out.append(_reference(one, s, steps, True)[0])
        return out
    shifted = case["dtype"].endswith("shifted") and case["kind"] == "steps"
    f, _ = _reference(case, seed, steps, shifted)
    if case["kind"] == "run":
        _stream(case["lattice"], f)
        rho, u = _moments(case["lattice"], f)
        return [rho, torch.stack(u), None]
    if case["dtype"] == "fp16_shifted":
        # stored as the deviation times 2^round(log2(1 / W_i))
        for i, w in enumerate(_weights(case["lattice"])):
            f[i] *= 2.0 ** round(-math.log2(w))
    return [f] + ([None] if case["alpha_map"] else [])
