"""The calls whose speed is measured, one dict of plain sizes each.

A case goes through the public entry points only, as a program that maps
simulations would: it holds a potential (drawn here as a Gaussian random field,
the stand-in for an N-body potential), a grid, a bundle of rays and a step
schedule, and asks for maps, gradients or records. ``exact`` gives the same
outputs in 64 bits from plain torch: the finite differences on the whole grid,
every ray cut at every cell face, three-point Gauss quadrature per piece (the
integrands are polynomials of degree five at most, so it is exact).

Kinds:
  kappa     trace_kappa: the convergence map of a periodic box (or a bounded one)
  shear     trace_shear: convergence and shear in one walk
  method_a  trace_method_a: convergence from grad(Phi) and the surface terms
  tiles     trace_tiles: a bundle through a stack of separate boxes, no wrap
  grad      TraceKappa forward and backward: maps and dL/dPhi
  batch     Batch: many lightcones of uneven sizes, traced together
  amr       AmrMesh records and Tracer.amr_steps over an adaptive mesh
  records   rr_tidal_tensor: the records of a whole grid
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1601_02012_gb300 as rr

HUBBLE = 2997.92458                    # c / H0 in Mpc/h
POISSON = 1.5 * 0.3 / HUBBLE ** 2      # 1.5 Omega_m (H0/c)^2, Omega_m = 0.3
F64 = torch.float64


def listed():
    return [
        # the smallest call: a first look at one snapshot, where launches and host work count
        {"name": "kappa_64", "kind": "kappa", "n0": 64, "n1": 64, "n2": 64, "cell": 4.0, "nx": 128, "ny": 128,
         "fov": 2.0, "depth": 1.0, "steps": 1, "trilinear": True, "periodic": True},
        # an ordinary map of a box whose sides and rays fit no tile: odd sizes, rows that are no multiple of 16 bytes
        {"name": "kappa_ragged", "kind": "kappa", "n0": 201, "n1": 187, "n2": 230, "cell": 2.0, "nx": 701, "ny": 503,
         "fov": 7.0, "depth": 0.97, "steps": 12, "trilinear": True, "periodic": True},
        # the production map: 512^3 cells, 2048^2 rays over 10 x 10 degrees, 40 steps of a simulation
        {"name": "kappa_512", "kind": "kappa", "n0": 512, "n1": 512, "n2": 512, "cell": 2.0, "nx": 2048, "ny": 2048,
         "fov": 10.0, "depth": 0.9765625, "steps": 40, "trilinear": True, "periodic": True},
        # the cell-constant form, which maps of one field at many resolutions use
        {"name": "ngp_256", "kind": "kappa", "n0": 256, "n1": 256, "n2": 256, "cell": 2.0, "nx": 1024, "ny": 1024,
         "fov": 10.0, "depth": 0.9765625, "steps": 20, "trilinear": False, "periodic": True},
        # convergence and shear of an ordinary box
        {"name": "shear_256", "kind": "shear", "n0": 256, "n1": 256, "n2": 256, "cell": 2.0, "nx": 1024, "ny": 1024,
         "fov": 10.0, "depth": 0.9765625, "steps": 20, "trilinear": True, "periodic": True},
        # Method A, by which production maps are made too
        {"name": "method_a_256", "kind": "method_a", "n0": 256, "n1": 256, "n2": 256, "cell": 2.0, "nx": 1024,
         "ny": 1024, "fov": 10.0, "depth": 0.9765625, "steps": 20, "trilinear": True, "periodic": True},
        # a lightcone through three boxes put end to end
        {"name": "tiles_3x128", "kind": "tiles", "n0": 128, "n1": 128, "n2": 128, "cell": 2.0, "nx": 512, "ny": 512,
         "fov": 8.0, "depth": 0.98, "steps": 12, "boxes": 3, "trilinear": True, "periodic": False},
        # a gradient step on a small box: what a fit of initial conditions repeats thousands of times
        {"name": "grad_64", "kind": "grad", "n0": 64, "n1": 64, "n2": 64, "cell": 4.0, "nx": 96, "ny": 96,
         "fov": 10.0, "depth": 1.0, "steps": 2, "trilinear": True, "periodic": True},
        # the gradient of a large map
        {"name": "grad_256", "kind": "grad", "n0": 256, "n1": 256, "n2": 256, "cell": 2.0, "nx": 1024, "ny": 1024,
         "fov": 5.0, "depth": 1.0, "steps": 1, "trilinear": True, "periodic": True},
        # many realisations at once
        {"name": "batch_16", "kind": "batch", "cones": 16, "n_low": 64, "n_high": 256, "ray_low": 256,
         "ray_high": 1024, "steps": 1, "trilinear": True, "periodic": True},
        # an adaptive mesh: 128^3 and up to four levels below, records of each step and the walk
        {"name": "amr_128", "kind": "amr", "n0": 128, "cell": 2.0, "lmax": 4, "nx": 1024, "ny": 1024, "fov": 5.0,
         "depth": 0.9765625, "steps": 8, "trilinear": True, "periodic": True},
        # the records of a whole grid, as a program computes them that keeps them for many bundles
        {"name": "records_512", "kind": "records", "n0": 512, "n1": 512, "n2": 512, "cell": 2.0, "trilinear": True},
    ]


def draw(rng):
    def span(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["kappa", "kappa", "kappa", "shear", "method_a", "tiles", "grad", "batch", "amr", "records"])
    c = {"kind": kind, "trilinear": True, "periodic": True, "steps": span(1, 40),
         "cell": round(rng.uniform(1.0, 5.0), 3), "fov": round(rng.uniform(2.0, 10.0), 3),
         "depth": round(rng.uniform(0.5, 1.0), 4)}
    if kind == "batch":
        lo, ray = span(32, 128), span(64, 400)
        return {"kind": kind, "cones": rng.randint(2, 24), "n_low": lo, "n_high": lo + span(8, 128), "ray_low": ray,
                "ray_high": ray + span(16, 500), "steps": 1, "trilinear": True, "periodic": True}
    if kind == "amr":
        c.update(n0=span(24, 128), lmax=rng.randint(1, 4), nx=span(64, 1024), ny=span(64, 1024),
                 steps=rng.randint(1, 8))
        return c
    if kind == "records":
        return {"kind": kind, "n0": span(32, 480), "n1": span(32, 480), "n2": span(32, 480), "cell": c["cell"],
                "trilinear": rng.random() < 0.8}
    big, rays = {"kappa": (400, 1800), "shear": (256, 1024), "method_a": (256, 1024), "tiles": (160, 700),
                 "grad": (256, 1024)}[kind]
    side = span(40, big)
    for a in ("n0", "n1", "n2"):
        c[a] = min(big, max(32, side + rng.randint(-7, 7)))
    c["nx"], c["ny"] = span(64, rays), span(64, rays)
    if kind == "kappa":
        c["trilinear"], c["periodic"] = rng.random() < 0.75, rng.random() < 0.8
    if kind == "grad":
        c["steps"] = rng.randint(1, 4)
    if kind == "tiles":
        c.update(periodic=False, boxes=rng.randint(2, 4), steps=rng.randint(2, 16))
    return c


# ---- inputs --------------------------------------------------------------------------------------------------------

def _generator(seed, *more):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + sum(int(m) * 7919 ** i for i, m in enumerate(more, 1)))
    return g


def _k2(n, h, zero=1.0):
    k = [2 * math.pi * torch.fft.fftfreq(n[0], d=h, device="cuda", dtype=F64),
         2 * math.pi * torch.fft.fftfreq(n[1], d=h, device="cuda", dtype=F64),
         2 * math.pi * torch.fft.rfftfreq(n[2], d=h, device="cuda", dtype=F64)]
    k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    k2[0, 0, 0] = zero
    return k2


def _potential(n, h, gen):
    """Gaussian random Phi/c^2 with P propto k^-3 below the Nyquist wavenumber, rms density contrast 1."""
    k2 = _k2(n, h)
    wk = torch.fft.rfftn(torch.randn(n, generator=gen, device="cuda", dtype=F64))
    wk *= torch.where(k2 <= (math.pi / h) ** 2, k2 ** -0.75, torch.zeros_like(k2))
    wk[0, 0, 0] = 0
    delta = torch.fft.irfftn(k2 * wk, s=n)
    phi = torch.fft.irfftn(wk, s=n)
    return (phi * (POISSON / delta.square().mean().sqrt())).to(torch.float32).contiguous()


def _schedule(chi_s, nsteps):
    """Equal steps in the scale factor of flat LCDM, the potential rescaled by D(a)/a; one step: none."""
    if nsteps == 1:
        return [SimpleNamespace(chi_a=chi_s, chi_b=0.0, scale=1.0, a=1.0)]
    a = np.linspace(0.02, 1.0, 20001)
    e = np.sqrt(0.3 / a ** 3 + 0.7)

    def integral(y):
        return np.concatenate([[0.0], np.cumsum(0.5 * (y[1:] + y[:-1]) * np.diff(a))])

    chi = integral(HUBBLE / (a ** 2 * e))
    chi = chi[-1] - chi
    grow = e * (integral(1.0 / (a * e) ** 3) + 0.4 * a[0] ** 2.5 / 0.3 ** 1.5)
    grow /= grow[-1]
    edges = np.linspace(np.interp(chi_s, chi[::-1], a[::-1]), 1.0, nsteps + 1)
    cuts = [chi_s] + [float(np.interp(x, a, chi)) for x in edges[1:-1]] + [0.0]
    return [SimpleNamespace(chi_a=cuts[i], chi_b=cuts[i + 1], a=float(edges[i]),
                            scale=float(np.interp(edges[i], a, grow) / edges[i])) for i in range(nsteps)]


def _setup(c):
    """Grid, bundle and steps: the observer at the centre of the z = 0 face, looking along z."""
    n = (c["n0"], c.get("n1", c["n0"]), c.get("n2", c["n0"]))
    h = c["cell"]
    grid = SimpleNamespace(n=n, box=n[0] * h, omega_m=0.3, h=h)
    if c["kind"] == "records":
        return grid, None, None
    chi_s = c["depth"] * n[2] * h * c.get("boxes", 1)
    fov = math.radians(c["fov"])
    bundle = SimpleNamespace(nx=c["nx"], ny=c["ny"], fov_x=fov, fov_y=fov, obs=(n[0] * h / 2, n[1] * h / 2, 0.0),
                             chi_s=chi_s, interp=1 if c["trilinear"] else 0, periodic=c["periodic"])
    return grid, bundle, _schedule(chi_s, c["steps"])


def _cones(c):
    """The lightcones of a batch: sides and ray counts spread evenly over the ranges, one step size each."""
    out, m = [], max(1, c["cones"] - 1)
    for i in range(c["cones"]):
        f = (i * 7 % c["cones"]) / m
        n = int(round(c["n_low"] + (c["n_high"] - c["n_low"]) * i / m))
        rays = int(round(c["ray_low"] * (c["ray_high"] / c["ray_low"]) ** f))
        out.append(_setup({"kind": "kappa", "n0": n, "cell": 1.5 + 2.0 * f, "nx": rays, "ny": rays,
                           "fov": 1.0 + 9.0 * (i / m), "depth": 1.0, "steps": c["steps"], "trilinear": c["trilinear"],
                           "periodic": c["periodic"]}))
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(kind=kind)
    if kind == "batch":
        s.cones = _cones(case)
        s.phi = [_potential(g.n, g.h, _generator(seed, i)) for i, (g, _, _) in enumerate(s.cones)]
        s.rec = [rr.record_buffer(g) for g, _, _ in s.cones]
        s.batch = rr.Batch([b for _, b, _ in s.cones])
        return s
    s.grid, s.bundle, s.steps = _setup(case)
    if kind == "amr":
        octs, phi = _mesh(case, seed)
        s.mesh = rr.AmrMesh(case["n0"], case["lmax"], s.grid.box, [o.cpu().numpy() for o in octs])
        s.phi = torch.cat([p.reshape(-1) for p in phi]).to(torch.float32)
        s.rec = [s.mesh.record_buffer() for _ in range(min(4, len(s.steps)))]
        s.tracer = rr.Tracer(s.bundle)
    elif kind == "tiles":
        s.tiles = [(_potential(s.grid.n, s.grid.h, _generator(seed, i)), s.grid,
                    (s.bundle.obs[0], s.bundle.obs[1], -i * s.grid.n[2] * s.grid.h)) for i in range(case["boxes"])]
    else:
        s.phi = _potential(s.grid.n, s.grid.h, _generator(seed))
    if kind == "records":
        s.rec = rr.record_buffer(s.grid)
        s.where = rr.RR_AT_VERTICES if case["trilinear"] else rr.RR_AT_CENTRES
    if kind == "grad":
        s.phi.requires_grad_(True)
        s.out = _cotangents(s.bundle, seed)
    return s


def _cotangents(b, seed):
    g = _generator(seed, 5)
    return [torch.randn((b.ny, b.nx), generator=g, device="cuda", dtype=F64) for _ in range(2)]


def run(s):
    if s.kind == "kappa":
        return rr.trace_kappa(s.phi, s.grid, s.bundle, s.steps)
    if s.kind == "shear":
        return rr.trace_shear(s.phi, s.grid, s.bundle, s.steps)
    if s.kind == "method_a":
        return rr.trace_method_a(s.phi, s.grid, s.bundle, s.steps)
    if s.kind == "tiles":
        return rr.trace_tiles(s.tiles, s.bundle, s.steps)
    if s.kind == "grad":
        k, kb = rr.TraceKappa.apply(s.phi, s.grid, s.bundle, s.steps)
        return k, kb, torch.autograd.grad((k, kb), s.phi, s.out)[0]
    if s.kind == "records":
        rr.rr_tidal_tensor(rr.grid_desc(s.grid), s.phi, None, s.rec, s.where)
        return s.rec
    if s.kind == "batch":
        s.batch.reset()
        for (g, b, _), phi, rec in zip(s.cones, s.phi, s.rec):
            rr.rr_tidal_tensor(rr.grid_desc(g), phi, None, rec, s.batch.where)
        for k in range(len(s.cones[0][2])):
            for i, ((g, b, steps), rec) in enumerate(zip(s.cones, s.rec)):
                st = steps[k]
                s.batch.stage(i, g, rec, st.chi_a, st.chi_b, st.scale, st.a)
            s.batch.upload()
            s.batch.trace()
        maps = [torch.empty((2, b.ny, b.nx), dtype=F64, device="cuda") for _, b, _ in s.cones]
        s.batch.finalize([m[0] for m in maps], [m[1] for m in maps])
        code, segments = s.batch.sync()
        return maps, code, segments
    # amr: the records of up to four steps, then those steps in one call
    s.tracer.reset()
    for i in range(0, len(s.steps), len(s.rec)):
        group = s.steps[i:i + len(s.rec)]
        for st, rec in zip(group, s.rec):
            s.mesh.tidal(s.phi, rec, bbox=s.mesh.footprint(s.tracer, st.chi_a, st.chi_b))
        s.tracer.amr_steps(s.mesh, s.rec[:len(group)], group)
    k, kb = s.tracer.finalize()
    return k, kb, s.tracer.segments()


def work(case):
    """Inputs once and outputs once; per cell segment the method's FP32 operations (a multiply-add counts two):
    about 240 trilinear, 40 cell-constant, the shear a second pair of channels, the gradient twice the forward."""
    kind = case["kind"]
    if kind == "batch":
        parts = [_work_one(dict(case, kind="kappa"), g, b) for g, b, _ in _cones(case)]
    elif kind == "amr":
        grid, b, _ = _setup(case)
        p = _work_one(case, grid, b)
        # a lognormal density refines one cell in a hundred or so: counted as the coarse grid and a quarter more
        parts = [{"bytes": 1.25 * p["bytes"], "flops": 1.25 * p["flops"]}]
    else:
        parts = [_work_one(case, *_setup(case)[:2])]
    return {k: float(sum(p[k] for p in parts)) for k in ("bytes", "flops")}


def _work_one(c, g, b):
    cells = g.n[0] * g.n[1] * g.n[2] * c.get("boxes", 1)
    if c["kind"] == "records":
        return {"bytes": 36.0 * cells, "flops": 40.0 * cells}
    rays = b.nx * b.ny
    # the cells the cone passes through are what has to be read
    cone = min(1.0, (b.chi_s * 2 * math.sin(b.fov_x / 2)) ** 2 * b.chi_s / 3 / (g.h ** 3 * cells) + 0.02)
    segments = rays * (b.chi_s / g.h * (1 + b.fov_x / 2) + c["steps"])
    per = 240.0 if c["trilinear"] else 40.0
    per *= {"shear": 1.6, "grad": 3.0}.get(c["kind"], 1.0)
    maps = {"shear": 4, "grad": 4}.get(c["kind"], 2)
    bytes_ = 4.0 * cells * cone + 8.0 * maps * rays + (4.0 * cells if c["kind"] == "grad" else 0.0)
    return {"bytes": bytes_, "flops": per * segments}


# ---- the same in 64 bits, without this repository's code ---------------------------------------------------------------

def _channels(phi, h, gradient=False):
    """{H_xx, H_yy, H_zz, H_xy, H_xz, H_yz, delta} (or {d_x, d_y, d_z Phi, delta}) at cell centres, channel last."""
    def at(*s):
        return torch.roll(phi, [-x for x in s], (0, 1, 2))

    unit = ((1, 0, 0), (0, 1, 0), (0, 0, 1))
    diag = [(at(*u) + at(*(-x for x in u)) - 2 * phi) / h ** 2 for u in unit]
    delta = (diag[0] + diag[1] + diag[2]) / POISSON
    if gradient:
        return torch.stack([(at(*u) - at(*(-x for x in u))) / (2 * h) for u in unit] + [delta], -1)
    out = torch.empty(tuple(phi.shape) + (7,), dtype=F64, device=phi.device)
    for i in range(3):
        out[..., i] = diag[i]
    out[..., 6] = delta
    del diag, delta
    for i, (p, q) in enumerate(((0, 1), (0, 2), (1, 2))):
        s, d = [0, 0, 0], [0, 0, 0]
        s[p], s[q], d[p], d[q] = 1, 1, 1, -1
        out[..., 3 + i] = (at(*s) + at(*(-x for x in s)) - at(*d) - at(*(-x for x in d))) / (4 * h * h)
    return out


def _vertices(f):
    """Vertex (i, j, k) is the mean of the eight cells around the lower corner of cell (i, j, k)."""
    for a in range(3):
        f = (f + torch.roll(f, 1, a)) / 2
    return f


def _directions(b):
    def angles(n, fov):
        return (2 * torch.arange(n, device="cuda", dtype=F64) - (n - 1)) * (fov / (2 * (n - 1))) if n > 1 else \
            torch.zeros(1, device="cuda", dtype=F64)

    ty, tx = torch.meshgrid(angles(b.ny, b.fov_y), angles(b.nx, b.fov_x), indexing="ij")
    th = torch.hypot(tx, ty)
    s = torch.where(th > 0, torch.sin(th) / th.clamp_min(1e-300), torch.ones_like(th))
    return torch.stack([s * tx, s * ty, torch.cos(th)], -1).reshape(-1, 3)


def _weights(n, kind):
    """[rays, channels of a record, integrals]: what a ray takes from a record."""
    x, y, z = n.unbind(-1)
    zero = torch.zeros_like(x)
    if kind == "method_a":
        return torch.stack([torch.stack([x, y, z, zero], -1), torch.stack([zero, zero, zero, zero + 1], -1)], -1)
    w = [torch.stack([y * y + z * z, x * x + z * z, x * x + y * y, -2 * x * y, -2 * x * z, -2 * y * z, zero], -1),
         torch.stack([zero] * 6 + [zero + 1], -1)]
    if kind == "shear":
        st = torch.hypot(x, y)
        cp = torch.where(st > 0, x / st.clamp_min(1e-300), zero + 1)
        sp = torch.where(st > 0, y / st.clamp_min(1e-300), zero)
        p, t = (-sp, cp, zero), (z * cp, z * sp, -st)
        pairs = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
        w.append(torch.stack([(p[i] * p[j] - t[i] * t[j]) * (1 if i == j else 2) for i, j in pairs] + [zero], -1))
        w.append(torch.stack([2 * p[i] * t[j] if i == j else 2 * (p[i] * t[j] + p[j] * t[i]) for i, j in pairs]
                             + [zero], -1))
    return torch.stack(w, -1)


def _project(rows, w):
    """[rays, points, channels] by [rays, channels, integrals]; summed in place of a product of tiny matrices."""
    return torch.stack([sum(rows[..., k] * w[:, None, k, d] for k in range(w.shape[1])) if d != 1 else rows[..., -1]
                        for d in range(w.shape[2])], -1)


GAUSS = ((-math.sqrt(0.6), 5 / 9), (0.0, 8 / 9), (math.sqrt(0.6), 5 / 9))
BITS = [(i & 1, i >> 1 & 1, i >> 2 & 1) for i in range(8)]


def _kernels(kind, chi, chi_s):
    g = chi * (1 - chi / chi_s)
    return [1 - 2 * chi / chi_s if kind == "method_a" else g, g, g, g]


def _interpolate(q, u, trilinear):
    """q: [..., 8 corners, integrals] at u in [0, 1]^3 of the cell; or [..., 1, integrals]."""
    if not trilinear:
        return q[..., 0, :]
    w = torch.stack([math.prod(u[..., a] if bit else 1 - u[..., a] for a, bit in enumerate(bits)) for bits in BITS], -1)
    return (q * w[..., None]).sum(-2)


def _pieces(n, obs, st, h, size, periodic):
    """The chi edges [rays, pieces + 1] at which rays cross cell faces between chi_b and chi_a, ascending."""
    lo = torch.full_like(n[:, 0], st.chi_b)
    hi = torch.full_like(lo, st.chi_a)
    if not periodic:
        for a in range(3):
            c = torch.stack([-obs[a] / n[:, a], (size[a] * h - obs[a]) / n[:, a]])
            c = torch.nan_to_num(c, nan=0.0, posinf=1e30, neginf=-1e30)
            inside = 0.0 <= obs[a] <= size[a] * h
            still = n[:, a] == 0
            lo = torch.where(still, lo if inside else hi, torch.maximum(lo, c.amin(0)))
            hi = torch.where(still, hi, torch.minimum(hi, c.amax(0)))
        hi = torch.maximum(hi, lo)
    cuts = [lo[:, None], hi[:, None]]
    for a in range(3):
        x0, x1 = obs[a] + lo * n[:, a], obs[a] + hi * n[:, a]
        k0 = torch.ceil(torch.minimum(x0, x1) / h)
        m = int((torch.floor(torch.maximum(x0, x1) / h) - k0).max().item()) + 1
        if m > 0:
            k = k0[:, None] + torch.arange(m, device="cuda", dtype=F64)
            chi = torch.nan_to_num((k * h - obs[a]) / n[:, a:a + 1], nan=0.0, posinf=0.0, neginf=0.0)
            cuts.append(torch.minimum(torch.maximum(chi, lo[:, None]), hi[:, None]))
    return torch.sort(torch.cat(cuts, 1), 1).values


def _trace(f, c, grid, b, steps, n, obs=None, most=8_000_000):
    """The integrals [rays, 2 or 4] of the rays n through the records f [cells, channels] over the steps."""
    obs = b.obs if obs is None else obs
    size = torch.tensor(grid.n, device="cuda")
    w = _weights(n, c["kind"])
    tri = c["trilinear"]
    bits = torch.tensor(BITS if tri else BITS[:1], device="cuda")
    origin = torch.tensor(obs, device="cuda", dtype=F64)
    total = torch.zeros((n.shape[0], w.shape[-1]), device="cuda", dtype=F64)
    for st in steps:
        reach = (st.chi_a - st.chi_b) / grid.h * (1 + b.fov_x) + 6
        at = max(1, int(most / reach))
        parts = []
        for r in range(0, n.shape[0], at):
            nr, wr = n[r:r + at], w[r:r + at]
            edge = _pieces(nr, obs, st, grid.h, grid.n, b.periodic)
            mid, half = (edge[:, 1:] + edge[:, :-1]) / 2, (edge[:, 1:] - edge[:, :-1]) / 2
            cell = torch.floor((origin + mid[..., None] * nr[:, None]) / grid.h)
            at8 = torch.remainder(cell.to(torch.int64)[..., None, :] + bits, size)
            idx = (at8[..., 0] * grid.n[1] + at8[..., 1]) * grid.n[2] + at8[..., 2]
            rows = f[idx.reshape(-1)].reshape(nr.shape[0], -1, f.shape[-1])
            q = _project(rows, wr).reshape(idx.shape + (w.shape[-1],))
            acc = 0.0
            for x, weight in GAUSS:
                chi = mid + x * half
                u = (origin + chi[..., None] * nr[:, None]) / grid.h - cell
                k = torch.stack(_kernels(c["kind"], chi, b.chi_s)[:w.shape[-1]], -1)
                acc = acc + (weight * half)[..., None] * k * _interpolate(q, u, tri)
            acc = acc.sum(1)
            if c["kind"] == "method_a":   # the surface terms at the two ends of the step
                for side, sign in ((0, 1.0), (-1, -1.0)):
                    chi = edge[:, side]
                    u = (origin + chi[:, None] * nr) / grid.h - cell[:, side]
                    g = chi * (1 - chi / b.chi_s) * (edge[:, -1] > edge[:, 0])
                    ends = torch.zeros_like(acc)
                    ends[:, 0] = sign * g * _interpolate(q[:, side], u, tri)[:, 0]
                    acc = acc + ends
            parts.append(acc)
        born = torch.full((w.shape[-1],), st.scale, device="cuda", dtype=F64)
        born[1] = st.scale * POISSON / st.a
        total = total + torch.cat(parts) * born
    return total


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        maps = []
        for i, (g, b, steps) in enumerate(_cones(case)):
            f = _vertices(_channels(_potential(g.n, g.h, _generator(seed, i)).to(F64), g.h)).reshape(-1, 7)
            maps.append(_trace(f, dict(case, kind="kappa"), g, b, steps, _directions(b)).T.reshape(2, b.ny, b.nx))
        return maps, None, None
    grid, b, steps = _setup(case)
    if kind == "amr":
        k = _trace_mesh(case, seed, grid, b, steps)
        return k[0], k[1], None
    if kind == "records":
        f = _channels(_potential(grid.n, grid.h, _generator(seed)).to(F64), grid.h)
        f = _vertices(f) if case["trilinear"] else f
        return torch.nn.functional.pad(f.reshape(-1, 7), (0, 1))
    n = _directions(b)
    if kind == "grad":
        phi = _potential(grid.n, grid.h, _generator(seed)).to(F64).requires_grad_(True)
        records = _vertices(_channels(phi, grid.h)).reshape(-1, 7)
        f = records.detach().requires_grad_(True)
        g = torch.stack([x.reshape(-1) for x in _cotangents(b, seed)], -1)
        maps, at = [], max(1, 2_000_000 // int(b.chi_s / grid.h * 1.2 + 6))
        for r in range(0, n.shape[0], at):
            m = _trace(f, case, grid, b, steps, n[r:r + at])
            (m * g[r:r + at]).sum().backward()
            maps.append(m.detach())
        records.backward(f.grad)
        m = torch.cat(maps).T.reshape(2, b.ny, b.nx)
        return m[0], m[1], phi.grad
    if kind == "tiles":
        m = 0.0
        for i in range(case["boxes"]):
            f = _vertices(_channels(_potential(grid.n, grid.h, _generator(seed, i)).to(F64), grid.h)).reshape(-1, 7)
            m = m + _trace(f, case, grid, b, steps, n, (b.obs[0], b.obs[1], -i * grid.n[2] * grid.h))
    else:
        f = _channels(_potential(grid.n, grid.h, _generator(seed)).to(F64), grid.h, kind == "method_a")
        f = _vertices(f) if case["trilinear"] else f
        m = _trace(f.reshape(-1, f.shape[-1]), case, grid, b, steps, n)
        if kind == "method_a":
            m[:, 0] += m[:, 1]
    return tuple(x.reshape(b.ny, b.nx) for x in m.T) + (None,)


# ---- adaptive meshes ---------------------------------------------------------------------------------------------------

def _key(x, side):
    return (x[..., 0] * side + x[..., 1]) * side + x[..., 2]


def _unkey(k, side):
    return torch.stack([k // (side * side), k // side % side, k % side], -1)


def _kids(octs):
    return 2 * octs[:, None, :] + torch.tensor(BITS, device="cuda")


class _Levels:
    """Finds cells of the levels 0 .. lmax by their integer coordinates."""

    def __init__(self, n, octs):
        self.n, self.octs, self.keys, self.order = n, octs, [None], [None]
        for level in range(1, len(octs)):
            k, o = torch.sort(_key(_kids(octs[level]).reshape(-1, 3), n << level))
            self.keys.append(k)
            self.order.append(o)

    def find(self, level, x):
        """Number within the level of the cells at x (periodic), -1 where there is none."""
        side = self.n << level
        k = _key(torch.remainder(x, side), side)
        if level == 0:
            return k
        if self.keys[level].numel() == 0:
            return torch.full_like(k, -1)
        p = torch.searchsorted(self.keys[level], k).clamp_max(self.keys[level].numel() - 1)
        return torch.where(self.keys[level][p] == k, self.order[level][p], -1)

    def leaf(self, q):
        """Level and number of the deepest cell that holds the finest cells q."""
        top = len(self.octs) - 1
        lev, num = torch.zeros_like(q[..., 0]), self.find(0, q >> top)
        for level in range(1, top + 1):
            k = self.find(level, q >> (top - level))
            lev, num = torch.where(k >= 0, level, lev), torch.where(k >= 0, k, num)
        return lev, num


def _normal(level, x, seed):
    """A standard normal for each cell, by its level, coordinates and the seed."""
    def mix(v):
        v = (v ^ (v >> 31 & 0x1FFFFFFFF)) * 0x3C79AC492BA7B653
        return (v ^ (v >> 27 & 0x1FFFFFFFFF)) * 0x1C69B3F74AC4AE35

    k = mix(mix(mix(mix(torch.full_like(x[..., 0], seed * 16 + level)) + x[..., 0]) + x[..., 1]) + x[..., 2])
    u = (((k >> 11) & 0x1FFFFFFFFFFFFF).to(F64) + 0.5) / 2.0 ** 53
    v = (((mix(k + 12345) >> 11) & 0x1FFFFFFFFFFFFF).to(F64) + 0.5) / 2.0 ** 53
    return torch.sqrt(-2 * torch.log(u)) * torch.cos(2 * math.pi * v)


def _children(level, octs, rho, seed):
    f = torch.exp(0.5 * _normal(level, _kids(octs), seed))
    return rho[:, None] * f / f.mean(1, keepdim=True)


def _coarser(level, x):
    """The eight cells of the level above around the centres of cells x, and their trilinear weights."""
    lo, fr = torch.div(x - 1, 2, rounding_mode="floor"), torch.where(x % 2 == 0, 0.75, 0.25).to(F64)
    for bits in BITS:
        w = math.prod(fr[:, a] if bits[a] else 1 - fr[:, a] for a in range(3))
        yield lo + torch.tensor(bits, device="cuda"), w


def _mesh(case, seed):
    """(octs, phi) per level: a lognormal density refines cells of more than 8 mean masses, two neighbouring leaves
    differ by a level at most; Phi by FFT on level 0, below it prolonged and relaxed on the seven-point equation."""
    n, top, h = case["n0"], case["lmax"], case["cell"]
    k2 = _k2((n, n, n), h)
    wk = torch.fft.rfftn(torch.randn((n, n, n), generator=_generator(seed), device="cuda", dtype=F64)) / k2.sqrt()
    wk[0, 0, 0] = 0
    g = torch.fft.irfftn(wk, s=(n, n, n))
    rho0 = torch.exp(g * (1.5 / g.std()) - 1.125)
    flags, cells, rho = [], torch.nonzero(rho0 > 8.0), rho0[rho0 > 8.0]
    for level in range(top):
        flags.append(cells)
        if level + 1 < top:
            kids = _children(level + 1, cells, rho, seed).reshape(-1)
            keep = kids / 8.0 ** (level + 1) > 8.0
            cells, rho = _kids(cells).reshape(-1, 3)[keep], kids[keep]
    near = torch.tensor([(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)], device="cuda")
    for level in range(top - 1, 0, -1):
        side = n << (level - 1)
        more = torch.remainder((flags[level] // 2)[:, None] + near, side).reshape(-1, 3)
        flags[level - 1] = _unkey(torch.unique(torch.cat([_key(flags[level - 1], side), _key(more, side)])), side)
    flags = [_unkey(torch.unique(_key(f, n << level)), n << level) for level, f in enumerate(flags)]
    octs = [torch.zeros((0, 3), dtype=torch.int64, device="cuda")] + flags
    levels = _Levels(n, octs)

    def laplacian(m):
        return 2 - 2 * torch.cos(2 * math.pi * m)

    f = [torch.fft.fftfreq(n, device="cuda", dtype=F64)] * 2 + [torch.fft.rfftfreq(n, device="cuda", dtype=F64)]
    lam = (laplacian(f[0])[:, None, None] + laplacian(f[1])[None, :, None] + laplacian(f[2])[None, None]) / h ** 2
    lam[0, 0, 0] = 1.0
    dk = torch.fft.rfftn(rho0 / rho0.mean() - 1) / lam
    dk[0, 0, 0] = 0
    phi, rho = [-POISSON * torch.fft.irfftn(dk, s=(n, n, n))], rho0.reshape(-1)
    for level in range(1, top + 1):
        x = _kids(octs[level]).reshape(-1, 3)
        rho = _children(level, octs[level], rho[levels.find(level - 1, octs[level])], seed).reshape(-1)
        v = sum(w * phi[-1].reshape(-1)[levels.find(level - 1, y)] for y, w in _coarser(level, x))
        nb = torch.stack([levels.find(level, x + s * torch.eye(3, dtype=torch.int64, device="cuda")[a])
                          for a in range(3) for s in (-1, 1)], 1)
        inner = (nb >= 0).all(1)
        source = (h / 2 ** level) ** 2 * POISSON * (rho / rho0.mean() - 1)
        for _ in range(8):
            v = torch.where(inner, (v[nb.clamp_min(0)].sum(1) - source) / 6, v)
        phi.append(v)
    return octs, phi


def _mesh_records(case, octs, phi):
    """The corner values [leaves per level, 8, 7] of every cell that is a leaf, by the rules of the paper's Secs. 2.7
    and 3.3: same-level stencils or the coarser level interpolated; vertex weights by mass at refinement boundaries."""
    n, top, h = case["n0"], case["lmax"], case["cell"]
    levels = _Levels(n, octs)
    tidal = [_channels(phi[0].to(torch.float32).to(F64), h).reshape(-1, 7)]
    unit = torch.eye(3, dtype=torch.int64, device="cuda")
    for level in range(1, top + 1):
        x, hl = _kids(octs[level]).reshape(-1, 3), h / 2 ** level
        p = phi[level].to(torch.float32).to(F64)
        out, whole = torch.zeros((len(x), 7), device="cuda", dtype=F64), torch.ones(len(x), device="cuda", dtype=bool)

        def at(d):
            nonlocal whole
            k = levels.find(level, x + d)
            whole = whole & (k >= 0)
            return p[k.clamp_min(0)]

        for i in range(3):
            out[:, i] = (at(unit[i]) + at(-unit[i]) - 2 * p) / hl ** 2
        for i, (a, c) in enumerate(((0, 1), (0, 2), (1, 2))):
            out[:, 3 + i] = (at(unit[a] + unit[c]) + at(-unit[a] - unit[c]) - at(unit[a] - unit[c])
                             - at(unit[c] - unit[a])) / (4 * hl * hl)
        coarse = sum(w[:, None] * tidal[-1][levels.find(level - 1, y)] for y, w in _coarser(level, x))
        out = torch.where(whole[:, None], out, coarse)
        out[:, 6] = out[:, :3].sum(1) / POISSON
        tidal.append(out)
    base = torch.tensor([0] + list(np.cumsum([len(t) for t in tidal])), device="cuda")
    tidal = torch.cat(tidal)
    bits = torch.tensor(BITS, device="cuda")

    def around(v):
        lev, num = levels.leaf(torch.remainder(v[:, None] + bits - 1, n << top))
        return lev, base[lev] + num

    def corner(v):
        """Values of lattice vertices that are corners of every leaf around them."""
        lev, num = around(v)
        w = torch.full(lev.shape, 0.125, device="cuda", dtype=F64)
        mixed = torch.nonzero(lev.amin(1) != lev.amax(1))[:, 0]
        if len(mixed):
            lm, fine = lev[mixed], lev[mixed].amax(1, keepdim=True)
            size = torch.pow(2, top - fine)
            low = torch.div(v[mixed][:, None] + bits - 1, size[..., None], rounding_mode="floor") * size[..., None]
            touch = torch.zeros(lm.shape, device="cuda", dtype=F64)
            for d in BITS:   # the corners of a fine leaf that touch a coarser one
                c = low + torch.tensor(d, device="cuda") * size[..., None]
                lv, _ = around(c.reshape(-1, 3))
                touch += (lv.amin(1).reshape(lm.shape) < fine).to(F64)
            share = torch.where(lm < fine, 1.0, touch / 8)
            w[mixed] = share / share.sum(1, keepdim=True)
        return torch.einsum("vk,vkc->vc", w, tidal[num])

    out = []
    for level in range(top + 1):
        x = _kids(octs[level]).reshape(-1, 3) if level else _unkey(torch.arange(n ** 3, device="cuda"), n)
        is_leaf = levels.find(level + 1, 2 * x) < 0 if level < top else torch.ones(len(x), device="cuda", dtype=bool)
        size = 1 << (top - level)
        v = torch.remainder((x[is_leaf][:, None] + bits) * size, n << top).reshape(-1, 3)
        key, back = torch.unique(_key(v, n << top), return_inverse=True)
        v = _unkey(key, n << top)
        lev, _ = around(v)
        step = torch.pow(2, top - lev.amin(1, keepdim=True))
        odd = v % step != 0           # off the lattice of the coarsest leaf around: the mean of its edge's or face's ends
        value = torch.zeros((len(v), 7), device="cuda", dtype=F64)
        plain = torch.nonzero(~odd.any(1))[:, 0]
        value[plain] = corner(v[plain])
        hang = torch.nonzero(odd.any(1))[:, 0]
        for d in BITS:
            s = torch.where(odd[hang], (2 * torch.tensor(d, device="cuda") - 1) * step[hang] // 2, 0)
            value[hang] += corner(torch.remainder(v[hang] + s, n << top)) / 8
        rec = torch.zeros((len(x), 8, 7), device="cuda", dtype=F64)
        rec[is_leaf] = value[back].reshape(-1, 8, 7)
        out.append(rec)
    return levels, base, torch.cat(out)


def _trace_mesh(case, seed, grid, b, steps):
    octs, phi = _mesh(case, seed)
    levels, base, rec = _mesh_records(case, octs, phi)
    top, fine = case["lmax"], grid.h / 2 ** case["lmax"]
    n, obs = _directions(b), torch.tensor(b.obs, device="cuda", dtype=F64)
    total, one = torch.zeros((2, len(n)), device="cuda", dtype=F64), torch.ones((), device="cuda", dtype=F64)
    for st in steps:
        ray = torch.arange(len(n), device="cuda")
        chi = torch.full((len(n),), st.chi_a, device="cuda", dtype=F64)
        while len(ray):
            d = n[ray]
            q = torch.floor((obs + (chi - 1e-8 * fine)[:, None] * d) / fine).to(torch.int64)
            lev, num = levels.leaf(torch.remainder(q, case["n0"] << top))
            size = torch.pow(2, top - lev)[:, None]
            low, side = torch.div(q, size, rounding_mode="floor") * size * (one * fine), size * (one * fine)
            out = (torch.where(d > 0, low, low + side) - obs) / d
            out = torch.where(d == 0, -1.0, out).amax(1)
            # a face that rounding has not left behind yet does not hold the ray up
            out = torch.minimum(out, chi - 1e-8 * fine).clamp_min(st.chi_b)
            w = _weights(d, "kappa")
            value = _project(rec[base[lev] + num], w)
            mid, half, acc = (chi + out) / 2, (chi - out) / 2, 0.0
            for x, weight in GAUSS:
                c = mid + x * half
                u = (obs + c[:, None] * d - low) / side
                acc = acc + (weight * half * c * (1 - c / b.chi_s))[:, None] * _interpolate(value, u, True)
            total[0, ray] += st.scale * acc[:, 0]
            total[1, ray] += st.scale * POISSON / st.a * acc[:, 1]
            more = out > st.chi_b
            ray, chi = ray[more], out[more]
    return total.reshape(2, b.ny, b.nx)
