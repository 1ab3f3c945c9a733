"""The work that users of the flux-limited diffusion solver have it do, as timed cases.

Every case goes through the package's public entry points.  The media are fBm sphere clouds (vacuum
outside a sphere, extinction up to ~100 inside), the ones the library's own benchmark solves, made
here on the GPU from the seed.  `exact` repeats the sweeps, the FP64 fixed point and the light bake in
64-bit torch, without the library.

Kinds of case:

  sweeps    a solve with a fixed budget of iterations (a preview, or a step of a progressive solve):
            fld_solve with tol 0, cold from the paper's initial state or warm from a given state
  tick      the same iterations through fld_iterate, with no residual checks
  fp64      a double-precision solve of a point source to a tolerance (the reference configuration)
  solve     a mixed-precision solve to a tolerance with Anderson mixing
  batch     many small clouds, each lit by its own light, solved together
  frame     a rendered frame: bake, quarter-resolution solve, primary ray march
  bake      the single-scatter source of a point light or an oblique directional light
"""
import math

import numpy as np
import torch

import paper_1403_8105_gb300 as fld

# Floating-point operations of one voxel update with two local rounds (differences, face sums, gradient,
# two evaluations of Knudsen number, limiter and update, blend), and of one trilinear sample of a march.
UPDATE_FLOPS = 90
SAMPLE_FLOPS = 30


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # An editor's preview tick: a few iterations of a small grid, where launches and latency count.
        dict(name="tick_32", kind="tick", nx=32, ny=32, nz=32, precision="fp32", limiter="lp", bf16=False,
             start="cold", iterations=16),
        # The reference configuration: a point source in a homogeneous 32^3 cube, FP64 throughout, to 1e-10.
        dict(name="point_32_fp64", kind="fp64", nx=32, ny=32, nz=32, tol=1e-10),
        # A rendered frame of a 200^3 cloud, phi solved at 50^3 to 1e-4, 1024^2 image (the paper's "Nebulae").
        dict(name="frame_200", kind="frame", nx=200, ny=200, nz=200, factor=4, width=1024, height=1024, tol=1e-4),
        # A progressive solve of a ragged region, continued from the state of the frame before, phi as a hi/lo pair.
        dict(name="ragged_pair", kind="sweeps", nx=131, ny=97, nz=115, precision="pair", limiter="kershaw",
             bf16=False, start="warm", iterations=128),
        # The bulk sweeps of the 128^3 benchmark cloud (fields resident in L2).
        dict(name="sweeps_128", kind="sweeps", nx=128, ny=128, nz=128, precision="fp32", limiter="lp", bf16=False,
             start="warm", iterations=256),
        # Its correction sweeps (float-float sums), where a mixed solve spends half of its time.
        dict(name="correct_128", kind="tick", nx=128, ny=128, nz=128, precision="mixed", limiter="lp", bf16=False,
             start="warm", iterations=64),
        # A 256^3 volume with a bfloat16 medium and another limiter: the fields stream from HBM.
        dict(name="bf16_256", kind="sweeps", nx=256, ny=256, nz=256, precision="fp32", limiter="larsen", bf16=True,
             start="cold", iterations=64),
        # The same size as a hi/lo pair, the family with the most iterations of a plain mixed solve.
        dict(name="pair_256", kind="sweeps", nx=256, ny=256, nz=256, precision="pair", limiter="lp", bf16=False,
             start="warm", iterations=32),
        # A heavy request of the serving mix.
        dict(name="heavy_512", kind="sweeps", nx=512, ny=512, nz=512, precision="fp32", limiter="lp", bf16=False,
             start="cold", iterations=16),
        # The benchmark cloud solved to 1e-6, the stop test in FP64.
        dict(name="solve_128", kind="solve", nx=128, ny=128, nz=128, tol=1e-6, albedo=0.95, max_iters=20000),
        # The batched mix: small clouds of uneven size, point and directional lights, solved together to 1e-6.
        dict(name="batch_16", kind="batch", count=16, edges="32,48,64", tol=1e-6, max_iters=6000),
        # The light bake of a 160^3 cloud lit by a point light above it.
        dict(name="bake_point_160", kind="bake", nx=160, ny=160, nz=160, light="point"),
    ]


def _edge(rng, lo, hi):
    """A length between lo and hi, even over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extents(rng, lo, hi):
    """A cube or a ragged box of about that edge."""
    n = _edge(rng, lo, hi)
    if rng.random() < 0.4:
        return n, n, n
    return tuple(max(lo, min(hi, int(round(n * rng.uniform(0.75, 1.25))))) for _ in range(3))


def draw(rng):
    kind = rng.choice(["sweeps", "sweeps", "sweeps", "tick", "tick", "fp64", "solve", "batch", "frame", "bake"])
    if kind in ("sweeps", "tick"):
        nx, ny, nz = _extents(rng, 24, 288)
        precision = rng.choice(["fp32", "pair"] if kind == "sweeps" else ["fp32", "pair", "mixed"])
        budget = 1.5e9 if precision == "fp32" else 6e8          # voxel updates, at most
        start = rng.choice(["cold", "warm"])
        # a cold start fills the vacuum from 1e-20: more of its first iterations say little about D there
        most = 32 if start == "cold" else 256
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision,
                    limiter=rng.choice(["lp", "lp", "lp", "kershaw", "larsen", "sum"]),
                    bf16=precision != "mixed" and rng.random() < 0.25, start=start,
                    iterations=max(4, min(_edge(rng, 8, most), int(budget / (nx * ny * nz)))))
    if kind == "fp64":
        n = _edge(rng, 16, 32)
        return dict(kind=kind, nx=n, ny=n, nz=rng.randint(16, 32), tol=rng.choice([1e-8, 1e-10]))
    if kind == "solve":
        nx, ny, nz = _extents(rng, 24, 104)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, tol=rng.choice([1e-4, 1e-5, 1e-6]),
                    albedo=round(rng.uniform(0.8, 0.97), 3), max_iters=rng.randrange(4000, 12001, 64))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 16), edges=rng.choice(["32,48,64", "24,37,53", "40,61", "32,96"]),
                    tol=rng.choice([1e-4, 1e-5, 1e-6]), max_iters=rng.randrange(2000, 4001, 64))
    if kind == "frame":
        nx, ny, nz = _extents(rng, 96, 220)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, factor=4, width=rng.randint(320, 1280),
                    height=rng.randint(240, 1024), tol=1e-4)
    nx, ny, nz = _extents(rng, 32, 224)
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, light=rng.choice(["point", "oblique", "down"]))


# ---------------------------------------------------------------------------
# Inputs, made on the GPU from the seed
# ---------------------------------------------------------------------------
DEV = "cuda"


def _lattice_weights(n, h, freq):
    """n x (cells + 1) matrix of the quintic blend of lattice values at the voxel centres of one axis."""
    u = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) * h * freq
    i = u.floor().long()
    t = u - i
    w = t * t * t * (t * (t * 6 - 15) + 10)
    m = torch.zeros(n, int(i.max()) + 2, dtype=torch.float64, device=DEV)
    m.scatter_(1, i[:, None], (1 - w)[:, None])
    m.scatter_(1, i[:, None] + 1, w[:, None])
    return m


def _fbm(nx, ny, nz, h, gen, octaves=5, freq=4.0):
    """fBm of lattice value noise in [0, 1], shape (nz, ny, nx)."""
    out, amp, total = None, 1.0, 0.0
    for _ in range(octaves):
        wx, wy, wz = (_lattice_weights(n, h, freq) for n in (nx, ny, nz))
        lat = torch.rand(wz.shape[1], wy.shape[1], wx.shape[1], dtype=torch.float64, generator=gen).to(DEV)
        v = torch.einsum("zc,cyx->zyx", wz, torch.einsum("yb,cbx->cyx", wy, torch.einsum("xa,cba->cbx", wx, lat)))
        out = amp * v if out is None else out.add_(v, alpha=amp)
        total += amp
        amp, freq = 0.5 * amp, 2 * freq
    return out / total


def _centres(n, h):
    return (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) * h


def _cloud(nx, ny, nz, gen, albedo=None):
    """(sigma_t, albedo, h) of an fBm sphere cloud on a box whose longest side is 1."""
    h = 1.0 / max(nx, ny, nz)
    sig = 200.0 * (_fbm(nx, ny, nz, h, gen) - 0.35).clamp_(min=0.0) ** 1.5
    r2 = ((_centres(nz, h)[:, None, None] - 0.5 * nz * h) ** 2 + (_centres(ny, h)[None, :, None] - 0.5 * ny * h) ** 2
          + (_centres(nx, h)[None, None, :] - 0.5 * nx * h) ** 2)
    sig = torch.where(r2 > (0.45 * min(nx, ny, nz) * h) ** 2, 0.0, sig).float().contiguous()
    if albedo is None:
        albedo = 0.8 + 0.19 * float(torch.rand((), generator=gen))
    return sig, torch.full_like(sig, albedo), h


def _down_light(sig, alb, h):
    """Single-scatter source of a unit light along -z: sigma_s times the transmittance from above (float32)."""
    s = sig.double()
    above = torch.flip(torch.cumsum(torch.flip(s, (0,)), 0), (0,)) - 0.5 * s
    return (alb.double() * s * torch.exp(-h * above)).float().contiguous()


def _warm_state(sig, j, h):
    """A smooth positive state (phi, D), padded FP64: blurred emission over the extinction, D near 1/(3 sigma)."""
    x = torch.nn.functional.avg_pool3d(j.double()[None, None], 5, 1, 2)
    for _ in range(2):
        x = torch.nn.functional.avg_pool3d(x, 5, 1, 2)
    x = x[0, 0] / (sig.double() + 1.0) + 1e-3 * float(j.double().square().mean().sqrt()) * h
    d = 1.0 / (3.0 * (sig.double() + 1.0))
    return (torch.nn.functional.pad(x, (1,) * 6).contiguous(), torch.nn.functional.pad(d, (1,) * 6).contiguous())


def _gen(case, seed):
    g = torch.Generator()
    g.manual_seed(1000003 * int(seed) + 17)
    return g


def _light(gen, nx, ny, nz, h, kind):
    """A point light above the box or an oblique direction, by kind."""
    u = torch.rand(3, dtype=torch.float64, generator=gen).tolist()
    if kind == "point":
        pos = (nx * h * (0.1 + 0.8 * u[0]), ny * h * (0.1 + 0.8 * u[1]), nz * h * (1.05 + 0.45 * u[2]))
        ctr = (0.5 * nx * h, 0.5 * ny * h, 0.5 * nz * h)
        return "point", pos, 4.0 * math.pi * sum((a - b) ** 2 for a, b in zip(pos, ctr))
    if kind == "down":
        return "directional", (0.0, 0.0, -1.0), 0.5 + u[0]
    th, ph = 0.35 * math.pi * (0.1 + 0.9 * u[0]), 2 * math.pi * u[1]
    return "directional", (math.sin(th) * math.cos(ph), math.sin(th) * math.sin(ph), -math.cos(th)), 1.0


def _bake(g, light):
    kind, where, power = light
    if kind == "point":
        g.bake_point(where, power)
    else:
        g.bake_directional(where, power)


def _fields(case, seed):
    """(sigma_t, albedo, source, h, start state or None) of a sweeps or tick case."""
    gen = _gen(case, seed)
    sig, alb, h = _cloud(case["nx"], case["ny"], case["nz"], gen)
    j = _down_light(sig, alb, h)
    return sig, alb, j, h, _warm_state(sig, j, h) if case["start"] == "warm" else None


def _point(case, seed):
    """sigma_t, albedo, source and h of a point source near the middle of a homogeneous box."""
    gen = _gen(case, seed)
    u = torch.rand(3, dtype=torch.float64, generator=gen).tolist()
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    h = 1.0 / max(nx, ny, nz)
    sig = torch.full((nz, ny, nx), 10.0 * (0.9 + 0.2 * u[0]), device=DEV)
    alb = torch.full_like(sig, 0.9 * (0.95 + 0.1 * u[1]))
    j = torch.zeros_like(sig)
    j[nz // 2, ny // 2, nx // 2 + (1 if u[2] > 0.5 else 0)] = 1.0 / h ** 3
    return sig, alb, j, h


def _state_out(nx, ny, nz):
    return [torch.empty((nz + 2, ny + 2, nx + 2), dtype=torch.float64, device=DEV) for _ in range(2)]


def prepare(case, seed):
    kind, nx, ny, nz = case["kind"], case.get("nx"), case.get("ny"), case.get("nz")
    s = {"case": dict(case)}
    if kind in ("sweeps", "tick"):
        sig, alb, j, h, start = _fields(case, seed)
        g = fld.Grid(nx, ny, nz, h)
        g.set_medium(sig, alb)
        g.set_source(j)
        common = dict(precision=case["precision"], limiter=case["limiter"], medium_bf16=int(case["bf16"]),
                      warm_start=int(case["start"] == "warm"))
        if kind == "sweeps":
            # tol 0: the budget decides; the cold start's default warm-up relaxes with omega = 1, and a
            # continued solve is given the modest factor that a few iterations can use
            s["p"] = fld.params(tol=0.0, max_iters=case["iterations"],
                                omega=1.0 if case["start"] == "cold" else 1.5, **common)
        else:
            s["p"] = fld.params(omega=1.2, **common)
        s.update(g=g, start=start, out=_state_out(nx, ny, nz))
    elif kind == "fp64":
        sig, alb, j, h = _point(case, seed)
        g = fld.Grid(nx, ny, nz, h)
        g.set_medium(sig, alb)
        g.set_source(j)
        s.update(g=g, out=_state_out(nx, ny, nz),
                 p=fld.params(precision="fp64", limiter="lp", tol=case["tol"], check_every=32, max_iters=20000))
    elif kind == "solve":
        gen = _gen(case, seed)
        sig, alb, h = _cloud(nx, ny, nz, gen, case["albedo"])
        g = fld.Grid(nx, ny, nz, h)
        g.set_medium(sig, alb)
        s.update(g=g, out=_state_out(nx, ny, nz),
                 p=fld.params(precision="mixed", limiter="lp", tol=case["tol"], anderson=8, check_every=64,
                              max_iters=case["max_iters"]))
    elif kind == "batch":
        gen = _gen(case, seed)
        edges = [int(x) for x in case["edges"].split(",")]
        s.update(grids=[], media=[], lights=[], outs=[],
                 p=fld.params(precision="mixed", limiter="lp", tol=case["tol"], anderson=8, check_every=64,
                              max_iters=case["max_iters"]))
        for b in range(case["count"]):
            n = edges[b % len(edges)]
            sig, alb, h = _cloud(n, n, n, gen)
            s["grids"].append(fld.Grid(n, n, n, h))
            s["media"].append((sig, alb))
            s["lights"].append(_light(gen, n, n, n, h, "point" if b % 2 else "oblique"))
            s["outs"].append(_state_out(n, n, n)[0])
    elif kind == "frame":
        gen = _gen(case, seed)
        sig, alb, h = _cloud(nx, ny, nz, gen, 0.9)
        f = case["factor"]
        box = (nx * h, ny * h, nz * h)
        ctr = tuple(0.5 * b for b in box)
        s.update(sig=sig, alb=alb, light=_light(gen, nx, ny, nz, h, "oblique"), g=fld.Grid(nx, ny, nz, h),
                 coarse=fld.Grid(-(-nx // f), -(-ny // f), -(-nz // f), f * h),
                 cam=fld.camera(eye=(ctr[0] + 0.35 * box[1], ctr[1] + 0.45 * box[1], ctr[2] - 2.1 * box[1]),
                                target=ctr, width=case["width"], height=case["height"], background=0.05),
                 p=fld.params(precision="mixed", limiter="lp", tol=case["tol"], check_every=64, max_iters=20000),
                 image=torch.empty((case["height"], case["width"]), dtype=torch.float32, device=DEV))
    elif kind == "bake":
        gen = _gen(case, seed)
        sig, alb, h = _cloud(nx, ny, nz, gen)
        g = fld.Grid(nx, ny, nz, h)
        g.set_medium(sig, alb)
        s.update(g=g, light=_light(gen, nx, ny, nz, h, case["light"]), out=torch.empty_like(sig))
    else:
        raise ValueError(kind)
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _read(s):
    """The state (phi, D): FP64, or the single-precision values that FP32 sweeps hold."""
    phi, D = s["out"]
    fld.fld_get_state(s["g"].handle, phi, D)
    if s["case"].get("precision") == "fp32":
        return phi.float(), D.float()
    return phi, D


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("sweeps", "tick"):
        if s["start"] is not None:
            s["g"].set_state(*s["start"])
        if kind == "sweeps":
            s["g"].solve(s["p"])
        else:
            s["g"].iterate(s["p"], case["iterations"])
        return _read(s)
    if kind == "fp64":
        s["g"].solve(s["p"])
        return _read(s)
    if kind == "solve":
        s["g"].bake_directional((0.0, 0.0, -1.0), 1.0)
        s["g"].solve(s["p"])
        # converged to tol, the fluence goes to a renderer in single precision
        return [x.float() for x in _read(s)]
    if kind == "batch":
        for g, (sig, alb), light in zip(s["grids"], s["media"], s["lights"]):
            g.set_medium(sig, alb)
            _bake(g, light)
        fld.fld_solve_batch(s["grids"], s["p"])
        for g, out in zip(s["grids"], s["outs"]):
            fld.fld_get_state(g.handle, out)
        return [out.float() for out in s["outs"]]
    if kind == "frame":
        s["g"].set_medium(s["sig"], s["alb"])
        _bake(s["g"], s["light"])
        s["g"].downsample_to(s["coarse"], case["factor"])
        s["coarse"].solve(s["p"])
        fld.fld_render(s["g"].handle, s["coarse"].handle, s["cam"], s["image"])
        return s["image"]
    _bake(s["g"], s["light"])
    fld.fld_get_source(s["g"].handle, s["out"])
    return s["out"]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "batch":
        edges = [int(x) for x in case["edges"].split(",")]
        n = sum(edges[b % len(edges)] ** 3 for b in range(case["count"]))
        return {"bytes": 12.0 * n, "flops": float(UPDATE_FLOPS * n)}        # medium in, phi out; one sweep at least
    n = case["nx"] * case["ny"] * case["nz"]
    state = 8.0 if case.get("precision") == "fp32" else 16.0                # phi and D, single or double
    if kind in ("sweeps", "tick"):
        warm = 16.0 if case["start"] == "warm" else 0.0
        return {"bytes": (12.0 + state + warm) * n, "flops": float(UPDATE_FLOPS) * case["iterations"] * n}
    if kind == "fp64":
        return {"bytes": 28.0 * n, "flops": float(UPDATE_FLOPS * n)}
    if kind == "solve":
        return {"bytes": 16.0 * n, "flops": float(UPDATE_FLOPS * n)}
    if kind == "frame":
        px = case["width"] * case["height"]
        return {"bytes": 8.0 * n + 4.0 * px,
                "flops": float(UPDATE_FLOPS * n / case["factor"] ** 3 + SAMPLE_FLOPS * (n * 0.5 * case["nz"] + px))}
    steps = 1.0 if case["light"] == "down" else float(case["nz"])          # half-voxel steps, half the column on average
    return {"bytes": 12.0 * n, "flops": SAMPLE_FLOPS * steps * n}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _limiter(name, R):
    if name == "sum":
        return 1 / (3 + R)
    if name == "kershaw":
        return 2 / (3 + torch.hypot(torch.full_like(R, 3.0), 2 * R))
    if name == "larsen":
        return 1 / torch.hypot(torch.full_like(R, 3.0), R)
    r = R.clamp(min=0.2)
    e = torch.exp(-2 * r)
    big = ((1 - 1 / r) + 2 * e / (1 - e)) / r
    x = R.clamp(max=0.2) ** 2
    small = 1 / 3 + x * (-1 / 45 + x * (2 / 945 + x * (-1 / 4725 + x * (2 / 93555 + x * (-1382 / 638512875
                                                                                         + x * 4 / 18243225)))))
    return torch.where(R < 0.2, small, big)


class _Sweeps:
    """Red-black iterations (red: i + j + k even) of the discretised equation on padded FP64 arrays."""

    def __init__(self, sig, alb, j, h, limiter, bf16=False):
        seps = 1e-3 / (max(sig.shape) * h)
        if bf16:   # the medium is defined as rounded to bfloat16 from its single-precision values
            s = sig.clamp(min=float(np.float32(seps)))
            a = ((1 - alb) * s).bfloat16().double()
            self.s = s.bfloat16().double()
        else:
            self.s = sig.double().clamp(min=seps)
            a = (1 - alb.double()) * self.s
        self.a, self.j = a * h * h, j.double() * h * h
        jbar = float(j.double().square().mean().sqrt())
        self.floor = 1e-20 * jbar
        self.h, self.limiter = h, limiter
        nz, ny, nx = sig.shape
        k, jj, i = (torch.arange(n, device=DEV) for n in (nz, ny, nx))
        self.red = (k[:, None, None] + jj[None, :, None] + i[None, None, :]) % 2 == 0
        self.phi = torch.full((nz + 2, ny + 2, nx + 2), 1e-20 * jbar * h, dtype=torch.float64, device=DEV)
        self.D = torch.full_like(self.phi, 1e-20 * h)

    def set(self, phi, D):
        self.phi, self.D = phi.clone(), D.clone()

    def half(self, mask, omega):
        p, c = self.phi, slice(1, -1)
        p0 = p[c, c, c]
        shifts = [(c, c, slice(0, -2)), (c, c, slice(2, None)), (c, slice(0, -2), c), (c, slice(2, None), c),
                  (slice(0, -2), c, c), (slice(2, None), c, c)]
        g = [(p[shifts[2 * a + 1]] - p[shifts[2 * a]]) / (2 * self.h) for a in range(3)]
        grad = (g[0] * g[0] + g[1] * g[1] + g[2] * g[2]).sqrt_().clamp_(min=self.floor)
        del g
        A, B, C = torch.zeros_like(p0), torch.zeros_like(p0), torch.zeros_like(p0)
        for w in shifts:
            d, Ds = p[w] - p0, self.D[w]
            A += d
            B += Ds * d
            C += Ds
        base, den = self.j - self.a * p0 + 0.5 * B, self.a + 0.5 * C
        delta = torch.zeros_like(p0)
        for _ in range(2):
            R = grad / (self.s * (p0 + delta)).clamp_(min=self.floor)
            Dp = _limiter(self.limiter, R) / self.s
            delta = (base + 0.5 * Dp * A) / (den + 3 * Dp)
        self.D[c, c, c] = torch.where(mask, Dp, self.D[c, c, c])
        self.phi[c, c, c] = torch.where(mask, p0 + omega * delta, p0)

    def run(self, iterations, omega):
        for _ in range(iterations):
            self.half(self.red, omega)
            self.half(~self.red, omega)


def _exact_bake(case, seed):
    gen = _gen(case, seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    sig, alb, h = _cloud(nx, ny, nz, gen)
    kind, where, power = _light(gen, nx, ny, nz, h, case["light"])
    s = sig.double()
    if case["light"] == "down":
        # half-voxel steps from the centre: the quarter points blend two centres 3:1 and 1:3
        up = torch.cat([s[1:], torch.zeros_like(s[:1])])
        tau = torch.flip(torch.cumsum(torch.flip(0.5 * h * (s + up), (0,)), 0), (0,))
        return power * alb.double() * s * torch.exp(-tau)
    x = torch.stack(torch.meshgrid(_centres(nz, h), _centres(ny, h), _centres(nx, h), indexing="ij")[::-1], -1).view(-1, 3)
    if kind == "point":
        d = torch.tensor(where, dtype=torch.float64, device=DEV) - x
        r = d.norm(dim=1, keepdim=True)
        w = d / r
    else:
        v = torch.tensor(where, dtype=torch.float64, device=DEV)
        w = (-v / v.norm()).expand_as(x)
        r = None
    ext = torch.tensor([nx * h, ny * h, nz * h], dtype=torch.float64, device=DEV)
    to = torch.where(w > 0, (ext - x) / w, torch.where(w < 0, -x / w, math.inf))
    length = to.min(dim=1).values
    if r is not None:
        length = torch.minimum(length, r[:, 0])
    step = 0.5 * h
    n = torch.tensor([nx, ny, nz], device=DEV)
    tau = torch.zeros_like(length)
    flat = s.reshape(-1)
    q = power * alb.double().reshape(-1) * flat
    live = torch.nonzero(q > 0)[:, 0]                    # a voxel without scattering emits nothing
    m = 0
    while live.numel():
        rest = length[live] - m * step
        live, rest = live[rest > 0], rest[rest > 0]
        if not live.numel():
            break
        part = rest.clamp(max=step)
        u = (x[live] + (m * step + 0.5 * part)[:, None] * w[live]) / h - 0.5
        u = torch.minimum(u.clamp(min=0.0), (n - 1).double())
        i0 = torch.minimum(u.floor().long(), (n - 2).clamp(min=0))
        f = u - i0
        i1 = torch.minimum(i0 + 1, n - 1)
        v = torch.zeros_like(part)
        for cz, wz in ((i0[:, 2], 1 - f[:, 2]), (i1[:, 2], f[:, 2])):
            for cy, wy in ((i0[:, 1], 1 - f[:, 1]), (i1[:, 1], f[:, 1])):
                b = (cz * ny + cy) * nx
                v += wz * wy * ((1 - f[:, 0]) * flat[b + i0[:, 0]] + f[:, 0] * flat[b + i1[:, 0]])
        tau[live] += v * part
        m += 1
    q = q * torch.exp(-tau)
    if r is not None:
        q = q / (4 * math.pi * r[:, 0].clamp(min=0.5 * h) ** 2)
    return q.view(nz, ny, nx)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sweeps", "tick"):
        sig, alb, j, h, start = _fields(case, seed)
        sw = _Sweeps(sig, alb, j, h, case["limiter"], case["bf16"])
        if start is not None:
            sw.set(*start)
        sw.run(case["iterations"], (1.0 if start is None else 1.5) if kind == "sweeps" else 1.2)
        return sw.phi, sw.D
    if kind == "fp64":
        sig, alb, j, h = _point(case, seed)
        sw = _Sweeps(sig, alb, j, h, "lp")
        sw.run(600, 1.8)
        return sw.phi, sw.D
    if kind == "bake":
        return _exact_bake(case, seed)
    return None      # stopped at a tolerance: how far from the fixed point it ends is the tolerance's, not the arithmetic's
