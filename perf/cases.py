"""Cases by which this library's speed is followed, each one pass of work that a program using it
does through its public calls (the Grid, Batch and Server classes of the binding, and
rmt_extrapolate_noalloc), over the range of sizes, precisions and options it is used with.

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  what a program holds before the pass: grids, batches, servers, buffers
  run(state)           one pass, and the state it leaves behind
  work(case)           the bytes and operations a pass cannot do without
  exact(case, seed)    the pass in plain 64-bit torch, where the method has a closed form there

Kinds of case:
  steps    a simulation advances `steps` timesteps and its whole state is read (u, p, rho and every
           body's reference map), as a program does between output frames; `io` says whether the
           fields stay on the device or u also comes from and goes to page-locked host memory
  batch    independent simulations advanced together, one graph launch per step
  serve    a queue of simulation jobs through the server, from submission to release
  extrap   the reference map of one body extrapolated on caller-owned buffers
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2104_00095_gb300 import rmt, scenes

# the solver schedule the benchmark times and the serving runtime uses
SCHEDULE = {"fe_inner": 4, "mac_inner": 5, "mac_pre": 2, "mac_post": 2, "mac_omega": 1.15, "mac_coarse_pre": 2,
            "mac_coarse_post": 2, "fe_pre": 2, "fe_post": 1, "fe_omega": 1.0}
CYCLES = {"mg_fixed_cycles": 5, "mg_fixed_cycles_fe": 4}
FIXED, ADAPTIVE = "fixed", "adaptive"


def _steps(name, scene, nx, ny, nz, bodies, precision, solver, steps, io="device"):
    c = {"kind": "steps", "scene": scene, "nx": nx, "ny": ny, "nz": nz, "bodies": bodies, "precision": precision,
         "solver": solver, "steps": steps, "io": io}
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest simulation a user starts with: the lid-driven cavity with one soft sphere in
        # plain FP64 with the default (adaptive, 1e-12) solves.  Latency and launches.
        _steps("cavity32_fp64", "cavity", 32, 32, 32, 1, "fp64", ADAPTIVE, 2),
        # The smallest grid of the serving mix, FP32 with fixed cycles and step graphs.
        _steps("settling48_fp32", "settling", 48, 48, 48, 3, "fp32", FIXED, 4),
        # Unequal sides between walls, partial tiles on every axis, adaptive FP32 solves to 1e-9: a
        # program that asks for a residual instead of a cycle count.
        _steps("ragged136x120x128_fp32", "ragged", 136, 120, 128, 1, "fp32", ADAPTIVE, 2),
        # A periodic size whose multigrid hierarchy ends on an odd side (112 -> 7).
        _steps("swimmers112_fp32", "swimmers", 112, 112, 112, 2, "fp32", FIXED, 4),
        # The settling mixture (20 ellipsoids, walls, gravity), the ordinary production size, FP32.
        _steps("settling128_fp32", "settling", 128, 128, 128, 20, "fp32", FIXED, 4),
        # The same mixture on the plain FP64 path.
        _steps("settling128_fp64", "settling", 128, 128, 128, 20, "fp64", FIXED, 1),
        # Fluid alone in a periodic box: the flow stages and the two projections without bodies.
        _steps("fluid128_fp32", "fluid", 128, 128, 128, 0, "fp32", FIXED, 2),
        # The large end of the serving mix driven from the host: u is uploaded from page-locked
        # memory, stepped and read back on every step (a coupled code, live monitoring).
        _steps("swimmers192_hostio_fp32", "swimmers", 192, 192, 192, 4, "fp32", FIXED, 1, "host"),
        # The benchmark's scene: 256^3, 8 active swimmers.
        _steps("swimmers256_fp32", "swimmers", 256, 256, 256, 8, "fp32", FIXED, 4),
        # Many small simulations at once (parameter sweeps): cavities of 32 to 128 cells a side.
        {"name": "batch12_cavities_fp32", "kind": "batch", "sims": 12, "largest": 128, "steps": 2},
        # A short burst of jobs through the server: admission, graph capture, steps, retirement.
        {"name": "serve5_fp32", "kind": "serve", "jobs": 5, "largest": 112, "steps": 24},
        # A caller that cannot allocate while it runs extrapolates one body's map on its own buffers.
        {"name": "extrapolate96", "kind": "extrap", "n": 96, "layers": 4, "radius": 0.25},
    ]


def _size(rng, lo, hi):
    """A side between lo and hi, a multiple of 8, spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, 8 * round(v / 8)))


def draw(rng):
    kind = rng.choice(["steps"] * 7 + ["batch", "serve", "extrap"])
    if kind == "batch":
        return {"kind": "batch", "sims": rng.randint(2, 12), "largest": rng.choice([48, 64, 96, 128]),
                "steps": rng.randint(1, 3)}
    if kind == "serve":
        return {"kind": "serve", "jobs": rng.randint(2, 5), "largest": rng.choice([64, 80, 96, 112]),
                "steps": rng.randint(8, 24)}
    if kind == "extrap":
        return {"kind": "extrap", "n": rng.randint(28, 128), "layers": rng.randint(1, 5),
                "radius": round(rng.uniform(0.18, 0.3), 3)}
    scene = rng.choice(["cavity", "settling", "swimmers", "swimmers", "fluid", "ragged"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    solver = rng.choice([FIXED, FIXED, ADAPTIVE])
    top = 96 if precision == "fp64" else (128 if solver == ADAPTIVE else 224)
    if scene == "ragged":
        n = [_size(rng, 32, min(top, 160)) for _ in range(3)]
        bodies = 1
    else:
        n = [_size(rng, 32 if scene != "settling" else 48, top)] * 3
        most = {"cavity": 1, "fluid": 0, "settling": 3 if n[0] < 64 else (6 if n[0] < 96 else 16), "swimmers": 8}[scene]
        bodies = rng.randint(min(1, most), most)
    io = rng.choice(["device", "device", "host"]) if precision == "fp32" else "device"
    return _steps(None, scene, n[0], n[1], n[2], bodies, precision, solver, rng.randint(1, 3), io)


# ------------------------------------------------------------------------------- inputs
def _ints(seed, count):
    return [int(v) for v in np.random.Generator(np.random.PCG64(seed)).integers(1, 2**31 - 1, count)]


def _scene(case, seed):
    n, k = case["nx"], case["scene"]
    scene_seed, gen = _ints(seed, 2)
    rng = np.random.Generator(np.random.PCG64(gen))
    if k == "settling":
        sc = scenes.settling(n=n, nbodies=case["bodies"], seed=scene_seed)
    elif k == "swimmers":
        sc = scenes.swimmers(n=n, nbodies=case["bodies"], seed=scene_seed)
    elif k == "cavity":
        sc = scenes.cavity_sphere(n)
        sc["dt"] = 0.2 / n if n <= 48 else 0.0  # 0.2 h is beyond the viscous limit on finer grids
        sc["solids"][0]["center"] = tuple(0.5 + rng.uniform(-0.1, 0.1, 3))
    elif k == "fluid":
        sc = scenes._box(n, periodic=True)
    else:  # ragged: unequal sides between no-slip walls, a lid and one ellipsoid
        m = (case["nx"], case["ny"], case["nz"])
        sc = scenes._box(max(m), periodic=False, lid=1.0)
        hi = tuple(v / max(m) for v in m)
        s = min(hi)
        axes = np.array([0.2, 0.15, 0.17]) * s
        sc.update(n=m, hi=hi)
        sc["solids"] = [scenes.solid(scenes.ELLIPSOID, [0.5 * v for v in hi], axes, scenes.random_rotation(rng),
                                     rho_s=1.3, G=0.4, mu_a=0.01)]
    sc["precision"] = case["precision"]
    if case["solver"] == FIXED:
        sc.update(CYCLES, options=dict(SCHEDULE, graph=1))
    elif case["precision"] == "fp32":
        sc["mg_rtol"] = 1e-9
    return sc


def _velocity(sc, seed, amplitude=0.3, dtype=torch.float32):
    """A smooth solenoidal velocity, zero at walls: the curl of a few random Fourier modes (times a
    bump that vanishes at the walls), by centred differences over half a cell."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n, lo, hi = sc["n"], sc.get("lo", (0, 0, 0)), sc.get("hi", (1, 1, 1))
    h = (hi[0] - lo[0]) / n[0]
    per = sc["bc"][0] == scenes.PERIODIC
    modes = [(rng.integers(-2, 3, 3), rng.normal(size=3), rng.uniform(0, 2 * np.pi)) for _ in range(6)]
    ax = [(torch.arange(n[d], device="cuda", dtype=torch.float64) + 0.5) * h for d in range(3)]

    def potential(shift):
        x, y, z = (ax[d] + shift[d] for d in range(3))
        x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
        out = [0.0, 0.0, 0.0]
        for k, a, ph in modes:
            w = torch.sin(2 * np.pi * (float(k[0]) * x / (hi[0] - lo[0]) + float(k[1]) * y / (hi[1] - lo[1]) +
                                       float(k[2]) * z / (hi[2] - lo[2])) + ph)
            for c in range(3):
                out[c] = out[c] + float(a[c]) * w
        if not per:
            bump = 1.0
            for d, v in enumerate((x, y, z)):
                t = v / (hi[d] - lo[d])
                bump = bump * (4 * t * (1 - t)) ** 2
            out = [v * bump for v in out]
        return out

    def diff(c, d):
        s = [0.0, 0.0, 0.0]
        s[d] = 0.5 * h
        p = potential(s)[c]
        s[d] = -0.5 * h
        return (p - potential(s)[c]) / h

    u = torch.stack([diff(2, 1) - diff(1, 2), diff(0, 2) - diff(2, 0), diff(1, 0) - diff(0, 1)])
    return (u * (amplitude / u.abs().max())).reshape(-1).to(dtype).contiguous()


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _write_u(g, u):
    if u.dtype == torch.float32:
        g.write_float_ptr(rmt.RMT_F_U, u.data_ptr(), u.numel() * 4, 1)
    else:
        g.write_ptr(rmt.RMT_F_U, u.data_ptr(), u.numel() * 8, 1)


def _buffers(sc):
    """Device buffers for a grid's whole state, in its storage precision."""
    dt = torch.float32 if sc["precision"] == "fp32" else torch.float64
    n = sc["n"]
    cells = n[0] * n[1] * n[2]
    nodes = cells if sc["bc"][0] == scenes.PERIODIC else (n[0] + 1) * (n[1] + 1) * (n[2] + 1)
    new = lambda k: torch.empty(k, dtype=dt, device="cuda")  # noqa: E731
    out = {"u": new(3 * cells), "p": new(nodes), "rho": new(cells)}
    if sc["solids"]:
        out["xi"] = new(3 * cells * len(sc["solids"])).reshape(len(sc["solids"]), 3 * cells)
    return out


def _read(g, field, t, solid=0):
    if t.dtype == torch.float32:
        g.read_float_ptr(field, t.data_ptr(), t.numel() * 4, 1, solid)
    else:
        g.read_device(field, t.data_ptr(), t.numel() * 8, solid)


def _read_state(g, buf, skip=()):
    for key, field in (("u", rmt.RMT_F_U), ("p", rmt.RMT_F_P), ("rho", rmt.RMT_F_RHO)):
        if key not in skip:
            _read(g, field, buf[key])
    for m in range(len(buf.get("xi", ()))):
        _read(g, rmt.RMT_F_XI, buf["xi"][m], m)
    return buf


def _cavity(n, bodies, rng):
    """One lid-driven cavity with 1 to 3 soft spheres in separate quarters of the box."""
    sc = scenes._box(n, periodic=False, lid=1.0)
    sc.update(precision="fp32")
    spots = [(0.3, 0.3, 0.35), (0.7, 0.3, 0.6), (0.3, 0.7, 0.6)]
    for c in spots[:bodies]:
        r = rng.uniform(0.1, 0.17)
        sc["solids"].append(scenes.solid(scenes.SPHERE, c, (r,) * 3, rho_s=rng.uniform(0.5, 1.5),
                                         G=rng.uniform(0.05, 1.0), mu_a=0.01))
    return sc


def _batch_sizes(case):
    """The sides of the batch's grids: the sizes of the benchmark's batch up to the case's largest."""
    sizes = [n for n in (32, 48, 64, 96, 128) if n <= case["largest"]]
    return [sizes[-1 - k % len(sizes)] for k in range(case["sims"])]


def _serve_sizes(case):
    sizes = [n for n in (48, 64, 80, 96, 112) if n <= case["largest"]]
    return [sizes[-1 - k % len(sizes)] for k in range(case["jobs"])]


# ------------------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    if kind == "steps":
        sc = _scene(case, seed)
        g = rmt.Grid(sc, stream=_stream())
        g.step(2)  # a running simulation: both step graphs are there
        dt = torch.float32 if case["precision"] == "fp32" else torch.float64
        u = _velocity(sc, _ints(seed, 3)[2], dtype=dt)
        _write_u(g, u)
        st = {"case": case, "grid": g, "buf": _buffers(sc)}
        if case["io"] == "host":
            st["host_in"] = u.cpu().pin_memory()
            st["host_out"] = torch.empty_like(st["host_in"]).pin_memory()
        return st
    if kind == "batch":
        rng = np.random.Generator(np.random.PCG64(seed))
        grids, bufs = [], []
        batch = rmt.Batch(stream=_stream())
        for k, n in enumerate(_batch_sizes(case)):
            sc = dict(_cavity(n, 1 + k % 3, rng), **CYCLES, options=dict(SCHEDULE))
            g = rmt.Grid(sc, stream=_stream())
            _write_u(g, _velocity(sc, int(rng.integers(1, 2**31 - 1))))
            batch.add(g)
            grids.append(g)
            bufs.append(_buffers(sc))
        batch.step(2)
        batch.sync()
        return {"case": case, "batch": batch, "grids": grids, "bufs": bufs}
    if kind == "serve":
        jobs = []
        for k, (n, s) in enumerate(zip(_serve_sizes(case), _ints(seed, case["jobs"]))):
            make = scenes.settling if k % 2 else scenes.swimmers
            sc = make(n=n, nbodies=1 + k % 3, seed=s, precision="fp32")
            jobs.append((dict(sc, **CYCLES), case["steps"] - 4 * (k % 2)))
        server = rmt.Server(80 * 10**9, stream=_stream(), options=SCHEDULE)
        return {"case": case, "server": server, "jobs": jobs, "bufs": [_buffers(sc) for sc, _ in jobs]}
    sc, body, xi = _extrap_inputs(case, seed)
    n3 = xi.shape[1]
    return {"case": case, "desc": rmt.make_grid_desc(sc), "body": rmt.make_solid_desc(body), "xi": xi,
            "out": {"xi": torch.empty_like(xi), "phi": torch.empty(n3, dtype=torch.float64, device="cuda"),
                    "layer": torch.empty(n3, dtype=torch.int8, device="cuda")}}


def _extrap_inputs(case, seed):
    """A walled unit box, one ellipsoid and a smooth map of every cell: the identity plus a few
    low-frequency displacements of a few per cent of the body's size."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n, r = case["n"], case["radius"]
    sc = scenes._box(n, periodic=False)
    sc["band_layers"] = case["layers"]
    body = scenes.solid(scenes.ELLIPSOID, 0.5 + rng.uniform(-0.05, 0.05, 3), r * rng.uniform(0.6, 1.0, 3),
                        scenes.random_rotation(rng))
    x = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
    Z, Y, X = torch.meshgrid(x, x, x, indexing="ij")
    comp = []
    for base in (X, Y, Z):
        d = 0.0
        for _ in range(4):
            k = rng.integers(-2, 3, 3)
            d = d + float(rng.normal()) * torch.sin(2 * np.pi * (float(k[0]) * X + float(k[1]) * Y + float(k[2]) * Z) +
                                                    rng.uniform(0, 2 * np.pi))
        comp.append((base + 0.01 * r * d).reshape(-1))
    return sc, body, torch.stack(comp).contiguous()


# ------------------------------------------------------------------------------- run
def run(state):
    kind = state["case"]["kind"]
    if kind == "steps":
        g, steps, buf = state["grid"], state["case"]["steps"], state["buf"]
        if state["case"]["io"] == "device":
            g.step(steps)
            return _read_state(g, buf)
        a, b = state["host_in"], state["host_out"]
        for _ in range(steps):
            g.write_float_ptr(rmt.RMT_F_U, a.data_ptr(), a.numel() * 4, 0)
            g.step(1)
            g.read_float_ptr(rmt.RMT_F_U, b.data_ptr(), b.numel() * 4, 0)
        return dict(_read_state(g, buf, skip=("u",)), u=b)
    if kind == "batch":
        state["batch"].step(state["case"]["steps"])
        state["batch"].sync()
        return [_read_state(g, b) for g, b in zip(state["grids"], state["bufs"])]
    if kind == "serve":
        srv = state["server"]
        ids = [srv.submit(sc, steps) for sc, steps in state["jobs"]]
        while srv.poll() != (0, 0):
            pass
        for j, buf in zip(ids, state["bufs"]):
            if srv.job(j)["state"] != rmt.RMT_JOB_DONE:
                raise RuntimeError("a job failed: %r" % (srv.job(j),))
            _read_state(srv.grid(j), buf)
            srv.release(j)
        return state["bufs"]
    out = state["out"]
    rc = rmt.load().rmt_extrapolate_noalloc(C.byref(state["desc"]), C.byref(state["body"]), state["xi"].data_ptr(),
                                            out["xi"].data_ptr(), out["phi"].data_ptr(), out["layer"].data_ptr(),
                                            _stream())
    if rc != rmt.RMT_OK:
        raise RuntimeError("rmt_extrapolate_noalloc: status %d" % rc)
    return out


# ------------------------------------------------------------------------------- work
# Operations per cell and step: the slope limiter, face states, stress and update arithmetic; and
# per unknown of one multigrid sweep or transfer of the 7-point and the 27-point operator.
STAGE_FLOPS, MAC_PASS_FLOPS, FE_PASS_FLOPS = 900, 30, 60


def _step_work(cells, bodies, word, steps, host=False):
    """State in and out once per pass (u, p, rho, each body's map over the whole grid as it is
    read), whatever the number of steps; the operations of the fixed schedule's passes."""
    state = (5 + 5 + 3 * bodies) * word * cells
    if host:
        state += steps * 2 * 3 * word * cells
    passes = 8 / 7 * (CYCLES["mg_fixed_cycles"] * 6 * MAC_PASS_FLOPS + CYCLES["mg_fixed_cycles_fe"] * 5 * FE_PASS_FLOPS)
    return state, steps * cells * (STAGE_FLOPS + passes)


def work(case):
    kind = case["kind"]
    if kind == "steps":
        cells = case["nx"] * case["ny"] * case["nz"]
        b, f = _step_work(cells, case["bodies"], 4 if case["precision"] == "fp32" else 8, case["steps"],
                          case["io"] == "host")
    elif kind == "batch":
        b, f = np.sum([_step_work(n**3, 1 + k % 3, 4, case["steps"]) for k, n in enumerate(_batch_sizes(case))], axis=0)
    elif kind == "serve":
        b, f = np.sum([_step_work(n**3, 1 + k % 3, 4, case["steps"] - 4 * (k % 2))
                       for k, n in enumerate(_serve_sizes(case))], axis=0)
    else:
        cells = case["n"] ** 3
        band = 4 * math.pi * (0.8 * case["radius"] * case["n"]) ** 2 * case["layers"]
        b, f = (3 + 3 + 1) * 8 * cells + cells, 30 * cells + band * 125 * 2 * 50
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------------------- exact
def exact(case, seed):
    if case["kind"] == "extrap":
        return _exact_extrap(case, seed)
    if case["kind"] == "steps" and case["scene"] == "fluid" and case["io"] == "device":
        return _exact_fluid(case, seed)
    return None  # bodies, walls: no closed form of the projections


def _limited_slope(q, dim, ih):
    """Fourth-order monotonicity-limited slope along a periodic axis."""
    at = lambda s: torch.roll(q, -s, dim)  # noqa: E731
    zero = torch.zeros((), dtype=q.dtype, device=q.device)

    def centred(a, b, c):
        return 0.5 * (c - a), torch.where((c - b) * (b - a) > 0, 2 * torch.minimum((c - b).abs(), (b - a).abs()), zero)

    def second(a, b, c):
        d, lim = centred(a, b, c)
        return torch.copysign(torch.minimum(d.abs(), lim), d)

    m2, m1, p1, p2 = at(-2), at(-1), at(1), at(2)
    d, lim = centred(m1, q, p1)
    d4 = 4.0 / 3.0 * d - (second(q, p1, p2) + second(m2, m1, q)) / 6.0
    return torch.copysign(torch.minimum(d4.abs(), lim), d) * ih


def _exact_fluid(case, seed):
    """The timestep of a periodic box without bodies, unit density: Godunov advection, and both
    projections by Fourier transforms of their constant-coefficient stencils."""
    sc = _scene(case, seed)
    n, mu, rho = case["nx"], sc["mu"], sc["rho_f"]
    h = 1.0 / n
    ih = float(n)
    dt = min(0.2 * h, 0.8 * rho * h * h / (6.0 * mu))
    tol = 1e-12 * h / dt
    dim = (2, 1, 0)  # tensor axis of x, y, z
    dtype = torch.float32 if case["precision"] == "fp32" else torch.float64
    u = _velocity(sc, _ints(seed, 3)[2], dtype=dtype).double().reshape(3, n, n, n)
    p = torch.zeros(n, n, n, dtype=torch.float64, device="cuda")  # at rest until u is written
    up = lambda a, d: torch.roll(a, -1, dim[d])  # noqa: E731  value at index + 1
    dn = lambda a, d: torch.roll(a, 1, dim[d])  # noqa: E731

    def symbol(f):
        c = torch.cos(2 * np.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n)
        s = f(c[None, None, :], c[None, :, None], c[:, None, None]).clone()
        s[0, 0, 0] = 1.0
        return s

    def invert(b, s):
        r = torch.fft.fftn(b) / s
        r[0, 0, 0] = 0.0
        return torch.fft.ifftn(r).real

    mac = symbol(lambda x, y, z: (6 - 2 * x - 2 * y - 2 * z) * (ih * ih / rho))
    fe = symbol(lambda x, y, z: (32 - 8 * x * y * z - 8 * (x * y + x * z + y * z)) * (h / 12.0 / rho))

    def cell_gradient(q):
        g = [torch.zeros_like(q) for _ in range(3)]
        for b in range(8):
            v = q
            for d in range(3):
                v = up(v, d) if b >> d & 1 else v
            for d in range(3):
                g[d] = g[d] + (v if b >> d & 1 else -v)
        return [v * (0.25 * ih) for v in g]

    def godunov(lo, hi):
        z = torch.zeros_like(lo)
        return torch.where((lo > tol) & (lo + hi > tol), lo, torch.where((hi < -tol) & (lo + hi < -tol), hi, z))

    def upwind(lo, hi, v):
        return torch.where(v > tol, lo, torch.where(v < -tol, hi, 0.5 * (lo + hi)))

    def states(base, d):
        """Left and right states at the face below each cell along d."""
        lo = [dn(base[a] + (0.5 * h - 0.5 * dt * u[d]) * slope[d][a], d) for a in range(3)]
        hi = [base[a] - (0.5 * h + 0.5 * dt * u[d]) * slope[d][a] for a in range(3)]
        return lo, hi

    for _ in range(case["steps"]):
        gp = cell_gradient(p)
        visc = [mu * ih * ih * (sum(up(u[a], d) + dn(u[a], d) for d in range(3)) - 6 * u[a]) for a in range(3)]
        slope = [[_limited_slope(u[a], dim[d], ih) for a in range(3)] for d in range(3)]
        term = []
        for e in range(3):
            lo, hi = states(u, e)
            v = godunov(lo[e], hi[e])
            bar = [upwind(lo[a], hi[a], v) for a in range(3)]
            term.append([0.5 * (v + up(v, e)) * (up(bar[a], e) - bar[a]) * ih for a in range(3)])
        face = []
        for d in range(3):
            base = [u[a] + 0.5 * dt / rho * (visc[a] - gp[a]) - 0.5 * dt * sum(term[e][a] for e in range(3) if e != d)
                    for a in range(3)]
            lo, hi = states(base, d)
            v = godunov(lo[d], hi[d])
            face.append([v if a == d else upwind(lo[a], hi[a], v) for a in range(3)])
        div = sum((up(face[d][d], d) - face[d][d]) * ih for d in range(3))
        q = invert(-div * (2.0 / dt), mac)
        um = [face[d][d] - 0.5 * dt * ih / rho * (q - dn(q, d)) for d in range(3)]
        star = []
        for a in range(3):
            adv = 0.0
            for d in range(3):
                f = um[d] if a == d else face[d][a]
                adv = adv + 0.5 * (um[d] + up(um[d], d)) * (up(f, d) - f) * ih
            star.append(u[a] - dt * adv + dt / rho * (visc[a] - gp[a]))
        # weak divergence of the increment at every node (the low corner of its cell)
        b = 0.0
        for c in range(8):
            for d in range(3):
                v = star[d] - u[d]
                for e in range(3):
                    v = v if c >> e & 1 else dn(v, e)
                b = b + (-v if c >> d & 1 else v)
        psi = invert(b * (h * h / 4.0 / dt), fe)
        g = cell_gradient(psi)
        u = torch.stack([star[a] - dt / rho * g[a] for a in range(3)])
        p = p + psi
    return {"u": u.reshape(-1), "p": p.reshape(-1), "rho": torch.full((n**3,), rho, dtype=torch.float64, device="cuda")}


def _exact_extrap(case, seed):
    """Layer 0 by the level set, layers by face neighbours, and one weighted least-squares fit per
    band cell over the 5^3 box (layers 1 and 2 again with the normal's weight)."""
    sc, body, xi = _extrap_inputs(case, seed)
    n = case["n"]
    dev, f8 = xi.device, torch.float64
    cen, axes = (torch.tensor(np.asarray(body[k]), dtype=f8, device=dev) for k in ("center", "semi_axes"))
    R = torch.tensor(np.asarray(body["rot"]), dtype=f8, device=dev)

    def level_set(X):  # [m, 3]
        y = (X - cen) @ R / axes
        g = y.norm(dim=1)
        w = (y / axes).norm(dim=1)
        return torch.where(g < 1e-12, -axes.min(), (g - 1) * g / w)

    out = xi.t().clone()
    layer = torch.where(level_set(out) < 0, 0, -1).reshape(n, n, n)
    for l in range(1, case["layers"] + 1):
        hit = torch.zeros_like(layer, dtype=torch.bool)
        prev = layer == l - 1
        for d in range(3):
            size = n - 1
            hit.narrow(d, 1, size).logical_or_(prev.narrow(d, 0, size))
            hit.narrow(d, 0, size).logical_or_(prev.narrow(d, 1, size))
        layer = torch.where(hit & (layer == -1), l, layer)
    flat = layer.reshape(-1)
    r = torch.arange(-2, 3, device=dev)
    dk, dj, di = (v.reshape(-1) for v in torch.meshgrid(r, r, r, indexing="ij"))
    off = torch.stack([di, dj, dk], 1).to(f8)
    v4 = torch.cat([torch.ones(125, 1, dtype=f8, device=dev), off], 1)
    kernel = 2.0 ** -(off.abs().sum(1))
    length = off.norm(dim=1).clamp_min(1e-300)
    for l in range(1, case["layers"] + 1):
        cells = torch.nonzero(flat == l).reshape(-1)
        for c in torch.split(cells, 16384):
            i, j, k = c % n, c // n % n, c // (n * n)
            I, J, K = i[:, None] + di, j[:, None] + dj, k[:, None] + dk
            inside = (I >= 0) & (I < n) & (J >= 0) & (J < n) & (K >= 0) & (K < n)
            idx = torch.where(inside, I + n * (J + n * K), 0)
            ok = inside & (flat[idx] >= 0) & (flat[idx] < l)
            data = torch.where(ok[..., None], out[idx], 0.0)

            def fit(w):
                A = torch.einsum("mc,ca,cb->mab", w, v4, v4)
                return torch.linalg.solve(A, torch.einsum("mc,ca,mcd->mad", w, v4, data))

            s = fit(ok * kernel)
            if l <= 2:
                g = ((s[:, 0] - cen) @ R / (axes * axes)) @ R.t()
                nrm = torch.einsum("mqd,md->mq", s[:, 1:], g)
                nrm = nrm / nrm.norm(dim=1, keepdim=True)
                s = fit(ok * kernel * (-(nrm @ off.t()) / length).clamp_min(0.0))
            out[c] = s[:, 0]
    nan = float("nan")
    band = flat >= 0
    phi = torch.where(band, level_set(out), nan)
    return {"xi": torch.where(band[:, None], out, nan).t().contiguous(), "phi": phi, "layer": flat.to(torch.int8)}
