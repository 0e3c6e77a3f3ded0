"""The work that users of this framework have it do, as measurable cases.

A case is a dict of plain values; ``prepare`` makes what a program has in hand
before the call (a context holding seeded particles, device or pinned host
buffers), ``run`` is one pass through the public entry points, ``exact`` the
same numbers in plain 64-bit torch where a pass has such values.

Kinds of cases:

* ``cells``    independent relaxation cells: steps, then the moments on the
               device or on the host, optionally with every particle;
* ``host``     cells whose particles live in pinned host buffers: one call
               takes them up, steps them and brings moments and state back;
* ``channel``  force-driven Poiseuille flow with its time averages;
* ``gradient`` the channel's derivative forms: profiles and their gradient;
* ``plane``    hypersonic flow past a cylinder, on a uniform or a three-level
               grid, with or without time averages;
* ``pool``     moments of a device-resident state, without any allocation.

Sizes are those of the workloads in ``paper_2508_05642_gb300/inputs.py``, of
the tests and of the benchmark.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2508_05642_gb300 import inputs as I
from paper_2508_05642_gb300 import usp

KB = 1.380649e-23
FORMS = {"f64": usp.USP_FP64, "f32": usp.USP_FP32,
         "f64_tangent": usp.USP_FP64_TANGENT, "f32_tangent": usp.USP_FP32_TANGENT}


def listed():
    return [
        # The smallest call: the step-and-look loop of a relaxation study (one
        # cell of 20,000 particles, plain FP64, moments on the host after each
        # step); launches and latency are all it is made of.
        dict(name="one_cell_f64", kind="cells", cells=1, nmin=20000, nmax=20000, form="f64",
             method="usp", steps=1, particles=False, host_moments=True),
        # The same cell in the FP32 form, advanced 25 steps and read back whole
        # (a stored snapshot of a run).
        dict(name="one_cell_f32", kind="cells", cells=1, nmin=20000, nmax=20000, form="f32",
             method="usp", steps=25, particles=True, host_moments=True),
        # The batched relaxation at its full size: 4096 instances, 154 million
        # particles, twenty steps replayed from a graph, moments left on the
        # device.  The state stays in the context, as between a program's calls.
        dict(name="batched_f32", kind="cells", cells=4096, nmin=1000, nmax=200000, form="f32",
             method="usp", steps=20, particles=False, host_moments=False),
        # The batch in plain FP64, the form that accuracy studies run, at a
        # tenth of the particles.
        dict(name="batched_f64", kind="cells", cells=4096, nmin=100, nmax=20000, form="f64",
             method="usp", steps=4, particles=False, host_moments=False),
        # The first-order method that the second-order one is compared with.
        dict(name="batched_fpm_f32", kind="cells", cells=4096, nmin=250, nmax=50000, form="f32",
             method="fpm", steps=5, particles=False, host_moments=False),
        # A coupling code that keeps its particles in host memory: up, one
        # step, moments and state down.
        dict(name="host_f32", kind="host", cells=1024, nmin=1000, nmax=200000, form="f32", steps=1),
        # Poiseuille flow: the sampling part of a run, 64 cells of 200 particles.
        dict(name="channel_f32", kind="channel", ny=64, ppc=200, form="f32", method="usp",
             steps=100),
        # Gradient of the averaged profiles, the default (FP64) derivative form.
        dict(name="gradient_f64", kind="gradient", ny=64, ppc=200, form="f64_tangent", steps=50),
        # Mach-10 cylinder on the 600 x 400 grid, 6.9 million particles: the
        # transient part of a run (no averages yet).
        dict(name="cylinder_f32", kind="plane", grid="uniform", nx=600, ny=400, ppc=30.0,
             form="f32", method="usp", warm=32, steps=8, sample=False, particles=False),
        # The three-level grid of the cylinder case (422,730 cells, 8.5 million
        # particles) while its averages and surface tallies are taken: half of
        # such a run's steps.
        dict(name="refined_sampled_f32", kind="plane", grid="paper", nx=640, ny=480, ppc=30.0,
             form="f32", method="usp", warm=32, steps=16, sample=True, particles=False),
        # A smaller cylinder grid in plain FP64, read back particle by particle
        # (verification runs).
        dict(name="cylinder_f64", kind="plane", grid="uniform", nx=240, ny=160, ppc=20.0,
             form="f64", method="usp", warm=0, steps=4, sample=False, particles=True),
        # Moments of particles that a host framework holds in its own device pool.
        dict(name="pool_moments_f64", kind="pool", cells=4096, nmin=100, nmax=20000),
    ]


def _log_uniform(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["cells", "cells", "cells", "host", "channel", "gradient", "plane", "plane",
                       "pool"])
    if kind in ("cells", "host", "pool"):
        form = rng.choice(["f32", "f64"])
        method = rng.choice(["usp", "usp", "fpm"])
        cells = _log_uniform(rng, 1, 4096 if kind != "pool" else 8192)
        # the mean count of a log-uniform draw in [lo, 20 lo] is about 6.3 lo
        most = {"cells": 6.0e7 if form == "f32" else 8.0e6, "host": 3.0e7, "pool": 1.5e7}[kind]
        lo = _log_uniform(rng, 50, max(60, min(2.0e5, most / (6.3 * cells))))
        hi = int(lo * rng.uniform(1.0, 20.0))
        if kind == "pool":
            return dict(kind=kind, cells=cells, nmin=lo, nmax=hi)
        if kind == "host":
            return dict(kind=kind, cells=cells, nmin=lo, nmax=hi, form=form,
                        steps=rng.randint(1, 3))
        few = 6.3 * cells * lo < 3.0e5
        return dict(kind=kind, cells=cells, nmin=lo, nmax=hi, form=form, method=method,
                    steps=rng.randint(1, 20 if form == "f32" else 4),
                    particles=few and rng.random() < 0.5, host_moments=rng.random() < 0.5)
    if kind == "channel":
        form = rng.choice(["f32", "f32", "f64"])
        return dict(kind=kind, ny=_log_uniform(rng, 5, 600), ppc=_log_uniform(rng, 10, 400),
                    form=form, method=rng.choice(["usp", "usp", "fpm"]),
                    steps=rng.randint(4, 60) if form == "f32" else rng.randint(4, 24))
    if kind == "gradient":
        return dict(kind=kind, ny=_log_uniform(rng, 8, 200), ppc=_log_uniform(rng, 20, 300),
                    form=rng.choice(["f64_tangent", "f32_tangent"]), steps=rng.randint(4, 40))
    form = rng.choice(["f32", "f32", "f64"])
    nx = _log_uniform(rng, 60, 600 if form == "f32" else 200)
    return dict(kind=kind, grid=rng.choice(["uniform", "refined"]), nx=nx,
                ny=max(40, int(nx * rng.uniform(0.6, 0.75))), ppc=round(rng.uniform(4.0, 32.0), 2),
                form=form, method=rng.choice(["usp", "usp", "usp", "fpm"]),
                warm=rng.randint(0, 24) if form == "f32" else 0, steps=rng.randint(1, 8),
                sample=rng.random() < 0.5, particles=False)


# ---------------------------------------------------------------------------
# seeded inputs, made on the GPU
# ---------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)
    return g


def _equilibrium(g, n, single, U, Ttr, Trot, Tvib, theta):
    """n particles of the species' mass: Maxwellian velocities, exponential
    rotational energy, geometric levels; the temperatures are numbers or one
    per particle.  ``single``: values that FP32 holds exactly."""
    R = KB / I.N2_MASS
    at = lambda v: v if torch.is_tensor(v) else torch.full((), float(v), device="cuda",
                                                           dtype=torch.float64)
    out = []
    s = torch.sqrt(R * at(Ttr)).float()
    for k in range(3):
        c = torch.randn(n, generator=g, device="cuda") * s + float(U[k])
        out.append(c)
    u = torch.rand(n, generator=g, device="cuda").clamp_(min=1e-7)
    out.append(-torch.log(u) * (R * at(Trot)).float())
    if not single:     # the low-order bits of a state that FP64 arithmetic made
        out = [c.double() * (1.0 + 2.0 ** -24 * torch.rand(n, generator=g, device="cuda",
                                                          dtype=torch.float64)) for c in out]
    else:
        out = [c.double() for c in out]
    u = torch.rand(n, generator=g, device="cuda").clamp_(min=1e-7)
    lev = torch.floor(-torch.log(u) * (at(Tvib) / theta).float()).to(torch.int32)
    return out + [lev]


def _cells(case, seed):
    """Offsets, number densities, temperatures and (on the device) particles of
    the batched relaxation's ranges; one cell takes the single-cell state."""
    sp = I.n2_vhs_relaxation_species()
    m = case["cells"]
    if m == 1:
        counts = np.array([case["nmin"]], dtype=np.int64)
        T = np.array([[10000.0, 300.0, 300.0]])
    else:
        # counts and temperatures spread evenly over their ranges (so that the
        # work does not depend on the seed), in an order of the seed's own
        r = np.random.default_rng([int(seed), 0xCE11])
        q = (np.arange(m) + 0.5) / m
        counts = np.floor(np.exp(np.log(case["nmin"]) +
                                 q * (np.log(case["nmax"]) - np.log(case["nmin"])))).astype(np.int64)
        counts = np.maximum(r.permutation(counts), 2)
        # the last cell fills the batch's storage (cells start on multiples of
        # four particles) up to a multiple of 64, whatever the odd sizes before
        counts[-1] += -int(np.sum((counts + 3) // 4 * 4)) % 64
        T = np.stack([r.permutation(a + q * (b - a)) for a, b in
                      ((2000.0, 20000.0), (300.0, 3000.0), (300.0, 3000.0))], axis=1)
    off = np.zeros(m + 1, dtype=np.int64)
    off[1:] = np.cumsum(counts)
    n = int(off[-1])
    dc, dT = torch.from_numpy(counts).cuda(), torch.from_numpy(T).cuda()
    per = lambda k: dT[0, k] if m == 1 else torch.repeat_interleave(dT[:, k], dc, output_size=n)
    p = _equilibrium(_gen(seed, 1), n, case.get("form", "f64") == "f32", (0.0, 0.0, 0.0), per(0), per(1),
                     per(2), sp["theta_v"])
    nd = np.full(m, 1e23)
    dt = np.array([0.5 * usp.usp_tau_c(sp, nd[i], T[i, 0]) for i in range(m)])
    return sp, off, nd, dt, p


def _pinned(tensors):
    out = []
    for t in tensors:
        h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
        h.copy_(t, non_blocking=True)
        out.append(h)
    torch.cuda.synchronize()
    return out


@functools.lru_cache(maxsize=1)
def _stream():
    """The program's own stream, on which all of its contexts work."""
    return torch.cuda.Stream()


def _method(case):
    return usp.USP_METHOD_FPM if case.get("method") == "fpm" else usp.USP_METHOD_USP_FPM


@functools.lru_cache(maxsize=8)
def _plane_grid(grid, nx, ny):
    """Domain, cells and fluid fractions of a cylinder case (no randomness)."""
    if grid == "paper":
        d = dict(x0=-0.4, x1=0.4, y0=0.0, y1=0.6, r=0.1524, n_inf=2.124e21, U_inf=2883.0,
                 levels=3, r2=0.24, r3=0.155)
    else:
        d = dict(x0=-0.35, x1=0.40, y0=0.0, y1=0.50, r=0.1, n_inf=1.2012e21, U_inf=2883.3,
                 levels=3 if grid == "refined" else 0, r2=0.22, r3=0.14)
    box = (nx, ny, d["x0"], d["x1"], d["y0"], d["y1"], 0.0, 0.0, d["r"])
    if d["levels"]:
        lv, li, lj = leaves = I.refined_leaves(*box, d["levels"], d["r2"], d["r3"])
        af = I.refined_cut_fractions(*box, leaves)
    else:
        c = np.arange(nx * ny)
        lv, li, lj = np.ones(nx * ny, dtype=np.int32), c % nx, c // nx
        af = I.cut_cell_fractions(*box)
    return d, lv, li, lj, af


def _plane(case, seed):
    """The impulsive start of the cylinder flow: the freestream everywhere
    outside the body, ppc particles per free level-1 cell."""
    nx, ny, ppc = case["nx"], case["ny"], case["ppc"]
    d, lv, li, lj, af = _plane_grid(case["grid"], nx, ny)
    sp = I.n2_vhs_cylinder_species()
    dx, dy = (d["x1"] - d["x0"]) / nx, (d["y1"] - d["y0"]) / ny
    g = _gen(seed, 2)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    sc = cu(1.0 / (1 << (lv - 1)).astype(np.float64))
    rand = lambda n: torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    counts = torch.floor(ppc * cu(af) * sc * sc + rand(len(lv))).long()
    leaf = torch.repeat_interleave(torch.arange(len(lv), device="cuda"), counts)
    n = int(leaf.numel())
    h, k = dx * sc[leaf], dy * sc[leaf]
    xl, yl = d["x0"] + cu(li)[leaf] * h, d["y0"] + cu(lj)[leaf] * k
    x, y = xl + rand(n) * h, yl + rand(n) * k
    bad = torch.nonzero(x * x + y * y <= d["r"] ** 2).reshape(-1)
    while bad.numel():                    # redraw inside the cut cells' fluid part
        x[bad] = xl[bad] + rand(bad.numel()) * h[bad]
        y[bad] = yl[bad] + rand(bad.numel()) * k[bad]
        bad = bad[x[bad] ** 2 + y[bad] ** 2 <= d["r"] ** 2]
    T_inf = 200.0
    p = _equilibrium(g, n, case["form"] == "f32", (d["U_inf"], 0.0, 0.0), T_inf, T_inf, T_inf,
                     sp["theta_v"])
    plane = dict(nx=nx, ny=ny, x0=d["x0"], x1=d["x1"], y0=d["y0"], y1=d["y1"], cyl_xc=0.0,
                 cyl_yc=0.0, cyl_r=d["r"], T_wall=500.0, n_inf=d["n_inf"], T_inf=T_inf,
                 U_inf=d["U_inf"], bc=(I.BC_OPEN, I.BC_OPEN, I.BC_SPECULAR, I.BC_OPEN),
                 inflow=(1, 0, 0, 1), F_num=d["n_inf"] * dx * dy / ppc, depth=1.0, reconstruct=1,
                 amr_levels=d["levels"], amr_r2=d["r2"] if d["levels"] else 0.0,
                 amr_r3=d["r3"] if d["levels"] else 0.0)
    dt = 1.6e-7 if case["grid"] == "paper" else 0.5 * usp.usp_tau_c(sp, d["n_inf"], T_inf)
    return sp, plane, dt, af, [x, y] + p


def _channel(case, seed):
    w = I.channel_poiseuille(seed=int(seed) & 0x7FFFFFFF, ny=case["ny"], ppc=case["ppc"])
    return w, w.dt_over_tau_c * usp.usp_tau_c(w.species, w.n, w.channel["T_wall"])


# ---------------------------------------------------------------------------
# a pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    key = 1 + int(seed) % 1000003                # the run's own random numbers
    on = dict(seed=key, method=_method(case), stream=_stream().cuda_stream)
    if kind == "pool":
        sp, off, nd, dt, p = _cells(case, seed)
        return dict(case=case, sp=sp, off=torch.from_numpy(off).cuda(), p=p,
                    out=torch.empty(usp.USP_NMOM, case["cells"], dtype=torch.float64,
                                    device="cuda"))
    if kind in ("cells", "host"):
        sp, off, nd, dt, p = _cells(case, seed)
        h = _pinned(p)
        ctx = usp.usp_init_homogeneous(sp, off, nd, dt, *[a.numpy() for a in h],
                                       precision=FORMS[case["form"]], **on)
        st = dict(case=case, ctx=ctx)
        if kind == "host":
            real = torch.float32 if case["form"] == "f32" else torch.float64
            st["h_in"] = [a.numpy() for a in _pinned([q.to(real) for q in p[:4]] + [p[4]])]
            st["h_out"] = [torch.empty(q.shape, dtype=real, pin_memory=True).numpy()
                           for q in p[:4]] + \
                          [torch.empty(p[4].shape, dtype=torch.int32, pin_memory=True).numpy()]
            st["mom"] = torch.empty(usp.USP_NMOM, case["cells"], dtype=torch.float64,
                                    pin_memory=True).numpy()
        elif not case["host_moments"]:
            st["mom"] = torch.empty(usp.USP_NMOM, case["cells"], dtype=torch.float64,
                                    device="cuda")
        return st
    if kind in ("channel", "gradient"):
        w, dt = _channel(case, seed)
        p = w.particles
        ctx = usp.usp_init_channel(w.species, w.channel, dt, w.y, p.cx, p.cy, p.cz, p.erot, p.lev,
                                   precision=FORMS[case["form"]], **on)
        usp.usp_channel_sample(ctx, True)
        st = dict(case=case, ctx=ctx)
        if kind == "gradient":
            st["dL"] = torch.randn(usp.USP_NPROF, case["ny"], dtype=torch.float64, device="cuda",
                                   generator=_gen(seed, 3))
        return st
    sp, plane, dt, af, p = _plane(case, seed)
    h = [a.numpy() for a in _pinned(p)]
    room = int(2 * case["ppc"] * np.sum(af)) + 4096
    ctx = usp.usp_init_plane(sp, plane, dt, af, *h, room, precision=FORMS[case["form"]], **on)
    if case["warm"]:
        usp.usp_step(ctx, case["warm"])          # a run that is under way
    if case["sample"]:
        usp.usp_sample(ctx, True)
    st = dict(case=case, ctx=ctx)
    if not case["sample"] and not case["particles"]:
        st["mom"] = torch.empty(usp.USP_NMOM, ctx.n_cells, dtype=torch.float64, device="cuda")
    usp.usp_sync(ctx)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "pool":
        p = st["p"]
        usp.usp_moments_noalloc(st["sp"], case["cells"], st["off"].data_ptr(),
                                *[a.data_ptr() for a in p], st["out"].data_ptr(),
                                stream=_stream().cuda_stream)
        return {"moments": st["out"]}
    ctx = st["ctx"]
    if kind == "host":
        usp.usp_step_host(ctx, *st["h_in"], case["steps"], st["mom"], out=st["h_out"])
        return {"moments": st["mom"], "state": st["h_out"]}
    usp.usp_step(ctx, case["steps"])
    if kind == "cells":
        out = {}
        if case["host_moments"]:
            out["moments"] = usp.usp_moments(ctx)
        else:
            usp.usp_moments(ctx, st["mom"].data_ptr(), out_is_device=True)
            out["moments"] = st["mom"]
        if case["particles"]:
            out["state"] = usp.usp_get_particles(ctx)
        return out
    if kind == "channel":
        return {"sums": usp.usp_channel_read(ctx, reset=True),
                "state": usp.usp_channel_get_particles(ctx)}
    if kind == "gradient":
        return {"profiles": usp.usp_profiles(ctx),
                "gradient": usp.usp_backward(ctx, st["dL"].data_ptr()),
                "state": usp.usp_channel_get_particles(ctx)}
    if case["sample"]:
        return {"sums": usp.usp_sample_read(ctx, reset=True)}
    if case["particles"]:
        # the live particles at the front of arrays as long as the storage
        return {"moments": usp.usp_moments(ctx),
                "state": [a.base for a in usp.usp_plane_get_particles(ctx)]}
    usp.usp_moments(ctx, st["mom"].data_ptr(), out_is_device=True)
    return {"moments": st["mom"]}


def work(case):
    """Per step the state read once and written once (a step's rescale and the
    next step's coefficients need every particle of the cell first), the moments'
    read of the state, the results once.  FLOPs: about 120 per particle and step."""
    kind = case["kind"]
    es = 4 if case.get("form", "f64").startswith("f32") else 8
    if kind in ("cells", "host", "pool"):
        m, lo, hi = case["cells"], case["nmin"], case["nmax"]
        n = m * lo if m == 1 or hi == lo else m * (hi - lo) / math.log(hi / lo)
        one, mom = 4 * es + 4, 8.0 * usp.USP_NMOM * m
        if kind == "pool":
            return {"bytes": n * 36 + mom, "flops": 40.0 * n}
        k = case["steps"]
        b = n * one * (2 * k + 1) + mom
        if kind == "host":
            b += 2 * n * one                     # the copies over the link touch HBM once each
        elif case["particles"]:
            b += n * (one + 36)
        return {"bytes": b, "flops": 120.0 * n * k}
    if kind in ("channel", "gradient"):
        n, k = case["ny"] * case["ppc"], case["steps"]
        f = 4 if kind == "gradient" else 1
        one = 5 * es * f + 8
        return {"bytes": n * one * 2.0 * k + n * 48.0, "flops": 150.0 * n * k * f}
    d, lv, li, lj, af = _plane_grid(case["grid"], case["nx"], case["ny"])
    n = float(case["ppc"] * np.sum(af / 4.0 ** (lv - 1)))
    one, k = 6 * es + 8, case["steps"]
    b = n * one * (2 * k + (1 if not case["sample"] else k)) + len(lv) * 8.0 * 22
    return {"bytes": b + (n * 56 if case["particles"] else 0.0), "flops": 250.0 * n * k}


# ---------------------------------------------------------------------------
# the same values in 64 bits: the relaxation cells' steps and the moments
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _mul32(a, b):
    """(high, low) 32-bit words of a constant times a tensor of 32-bit words."""
    lo, hi = b & 0xFFFF, b >> 16
    t = a * lo + (((a * hi) & 0xFFFF) << 16)
    return ((a * hi) >> 16) + (t >> 32), t & _M32


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 words as int64 tensors; c0..c3 ints or tensors."""
    z = torch.zeros_like(c0)
    c = [c0, z + c1, z + c2, z + c3]
    k0, k1 = key & _M32, (key >> 32) & _M32
    for _ in range(10):
        h0, l0 = _mul32(0xD2511F53, c[0])
        h1, l1 = _mul32(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c


def _sum(v, cid, m):
    return v.sum().reshape(1) if m == 1 else \
        torch.zeros(m, dtype=torch.float64, device=v.device).index_add_(0, cid, v)


def _moments(sp, m, cid, cnt, c, e, lev):
    R, th = KB / sp["m"], sp["theta_v"]
    inv = 1.0 / cnt
    l = lev.double()
    U = [_sum(v, cid, m) * inv for v in c]
    eb, er = _sum(l, cid, m) * inv, _sum(e, cid, m) * inv
    C = [v - u[cid] for v, u in zip(c, U)]
    Pi = [_sum(C[a] * C[b], cid, m) * inv for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
    q = 0.5 * (C[0] ** 2 + C[1] ** 2 + C[2] ** 2)
    Tv = torch.where(eb > 0, th / torch.log1p(1.0 / eb), 0.0 * eb)
    flux = [_sum(w * v, cid, m) * inv * f for w, f in ((q, 1.0), (e, 1.0), (l, R * th)) for v in C]
    return torch.stack([cnt] + U + [(Pi[0] + Pi[1] + Pi[2]) / (3 * R), er / R, Tv] + Pi + flux)


def _invert(u, P, ratio, n=None):
    """Sequential inversion: the least k with u below the cumulative sum, the
    pmf stepped by ratio(k, at); n (or None): the largest value per draw."""
    k = torch.zeros_like(u, dtype=torch.int64)
    at = torch.nonzero(u >= P).reshape(-1)
    u, P, cdf, j = u[at], P[at], P[at].clone(), 0
    while at.numel():
        if n is not None:
            keep = n[at] > j
            at, u, P, cdf = at[keep], u[keep], P[keep], cdf[keep]
        P = P * ratio(j, at)
        j += 1
        k[at] = j
        new = cdf + P
        go = (u >= new) & (new != cdf)
        at, u, P, cdf = at[go], u[go], P[go], new[go]
    return k


def _coeffs(sp, n, dt, Ttr, Trot, Tvib, Pi, fpm):
    """alpha, L (sqrt(1 - alpha^2) times the Cholesky factor), a_rot, the jump
    parameters and the energy targets of every cell; None where the positivity
    fix of the method would apply."""
    R, th = KB / sp["m"], sp["theta_v"]
    ca, w = sp["c_alpha"], sp["omega"]
    ev = lambda T: torch.where(T > 0, R * th / torch.expm1(th / T.clamp(min=1e-3)), 0.0 * T)
    mu = (5 * (ca + 1) * (ca + 2) * math.sqrt(sp["m"] * KB * sp["T_ref"] / math.pi) /
          (4 * ca * (5 - 2 * w) * (7 - 2 * w) * sp["d_ref"] ** 2)) * (Ttr / sp["T_ref"]) ** w
    mu_p = mu / (n * KB * Ttr)
    tc = ca * (5 - 2 * w) * (7 - 2 * w) / (5 * (ca + 1) * (ca + 2)) * mu_p
    tr, tv = sp["Z_rot"] * tc, sp["Z_vib"] * tc
    x = th / Tvib.clamp(min=1e-3)
    xi = torch.where(Tvib > 0, x / torch.expm1(x), 0.0 * x)
    Pr = (14 + 2 * xi) / (19 + 2 * xi)
    RT, evn = R * Ttr, ev(Tvib)
    if fpm:
        nu = 1 - 3 / (2 * Pr)
        tau = 2 * mu_p * (1 - nu)
        al = torch.exp(-dt / tau)
        gr, gv = tau / (2 * tr), tau / (2 * tv)
        etr = 1.5 * RT + gr * (R * Trot - RT) + gv * (evn - ev(Ttr))
        erot, evib = R * Trot + gr * (RT - R * Trot), evn + gv * (ev(Ttr) - evn)
        RTr, a2 = etr / 1.5, al * al
        eb = evib / (R * th)
        jump = (2 * dt * eb / tau, 2 * dt * (1 + eb) / tau)
        tgt = (erot + (R * Trot - erot) * a2, evib + (evn - evib) * a2)
        if bool(((etr < 0) | (erot < 0) | (evib < 0)).any()):
            return None
    else:
        A, B = (2 * mu_p - Pr * dt) / (2 * mu_p + Pr * dt), (2 * mu_p - dt) / (2 * mu_p + dt)
        al = torch.sign(A) * A.abs() ** (1.0 / 3.0)
        a2 = al * al
        nu = (B - a2) / (1 - a2)
        g1, g2 = dt / (dt + 2 * tr), dt / (dt + 2 * tv)
        cv = lambda T: R * ((0.5 * th / T) / torch.sinh(0.5 * th / T)) ** 2
        y = cv(Ttr)
        for _ in range(40):
            Tc = Ttr + (g1 * R * (Trot - Ttr) + g2 * y * (Tvib - Ttr)) / (1.5 * R + g1 * R + g2 * y)
            near = (Tc - Tvib).abs() <= 1e-9 * torch.maximum(Tc.abs(), Tvib.abs())
            y = torch.where(near, cv(Tvib.clamp(min=1.0)),
                            (ev(Tc) - evn) / torch.where(near, torch.ones_like(Tc), Tc - Tvib))
        den = 1.5 * R + g1 * R + g2 * y
        ktr, ktv = 2 * g1 * 1.5 * R * R / den, 2 * g2 * 1.5 * R * y / den
        krv = 2 * g1 * g2 * R * y / den
        tgt = (R * Trot + ktr * (Ttr - Trot) - krv * (Trot - Tvib),
               evn + ktv * (Ttr - Tvib) + krv * (Trot - Tvib))
        o = 1 - a2
        RTr = RT - (ktr * (Ttr - Trot) + ktv * (Ttr - Tvib)) / (1.5 * o)
        erot = R * Trot + (ktr * (Ttr - Trot) - krv * (Trot - Tvib)) / o
        evib = evn + (ktv * (Ttr - Tvib) + krv * (Trot - Tvib)) / o
        if bool(((RTr < 0) | (erot < 0) | (evib < 0) | (tgt[0] < 0) | (tgt[1] < 0)).any()):
            return None
        eb = evib / (R * th)
        jump = (1 / (1 + eb * o), (1 + eb) * o)
    M = torch.zeros(len(Ttr), 3, 3, dtype=torch.float64, device=Ttr.device)
    for q, (a, b) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
        M[:, a, b] = M[:, b, a] = nu * (Pi[q] - (RT if a == b else 0.0)) + (RTr if a == b else 0.0)
    L, bad = torch.linalg.cholesky_ex(M)
    if bool(bad.any()):
        return None
    return al, torch.sqrt(1 - a2)[:, None, None] * L, erot * (1 - a2) / 2, jump, tgt


def _gillespie(lev, up, dn, pid, step, key):
    lev, t = lev.clone(), torch.zeros_like(up)
    at, ev = torch.arange(lev.numel(), device=lev.device), 0
    u32 = lambda x: (x.double() + 0.5) * 2.0 ** -32
    w = None
    while at.numel():
        if ev % 2 == 0:
            w = torch.stack(_philox(pid[at], step, 8, ev // 2, key))
        a, b = (0, 1) if ev % 2 == 0 else (2, 3)
        lu, ld = up[at] * (lev[at] + 1).double(), dn[at] * lev[at].double()
        rate = lu + ld
        t[at] = t[at] - torch.log(u32(w[a])) / rate
        go = (rate > 0) & (t[at] <= 1)
        step_up = u32(w[b]) < lu / rate
        lev[at[go & step_up]] += 1
        lev[at[go & ~step_up]] -= 1
        at, w, ev = at[go], w[:, go], ev + 1
    return lev


def _correct(lev, off, cnt, Id, step, key):
    """The +-1 corrections of Sec. 4.C, draw after draw, every cell at once."""
    cell = torch.nonzero(Id != 0).reshape(-1)
    rem, j = Id[cell].clone(), 0
    words = None
    while cell.numel():
        if j % 4 == 0:
            words = torch.stack(_philox(cell, step, 0x80000001, j // 4, key))
        at = off[cell] + ((words[j % 4] * cnt[cell]) >> 32)
        ok = (rem > 0) | (lev[at] > 0)
        s = torch.sign(rem) * ok
        lev[at] += s
        rem -= s
        j += 1
        go = (rem != 0) & (j < 64 * cnt[cell])
        if not bool(go.all()):
            cell, rem, words = cell[go], rem[go], words[:, go]


def _relax(sp, off, nd, dt, p, steps, key, fpm):
    """``steps`` steps of every cell: (velocities, energies, levels), or None."""
    m = len(nd)
    dev = p[0].device
    o = torch.from_numpy(off).to(dev)
    cnt = o[1:] - o[:-1]
    N = cnt.double()
    cid = torch.repeat_interleave(torch.arange(m, device=dev), cnt)
    pid = torch.arange(int(off[-1]), device=dev)
    n, dt = torch.from_numpy(nd).to(dev), torch.from_numpy(dt).to(dev)
    c, e, lev = [q.double() for q in p[:3]], p[3].double(), p[4].long()
    R, th = KB / sp["m"], sp["theta_v"]
    for step in range(steps):
        U = [_sum(v, cid, m) / N for v in c]
        C = [v - u[cid] for v, u in zip(c, U)]
        Pi = [_sum(C[a] * C[b], cid, m) / N for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
        er, eb = _sum(e, cid, m) / N, _sum(lev.double(), cid, m) / N
        Ttr = (Pi[0] + Pi[1] + Pi[2]) / (3 * R)
        k = _coeffs(sp, n, dt, Ttr, er / R, torch.where(eb > 0, th / torch.log1p(1 / eb), 0 * eb), Pi,
                    fpm)
        if k is None:
            return None
        al, L, ar, jump, tgt = k
        w = _philox(pid, step, 0, 0, key)
        u23 = lambda x: (2 * (x >> 9) + 1).double() * 2.0 ** -24
        ang = lambda x, y: (2 * (((x & 511) << 9) | (y & 511)) + 1).double() * 2.0 ** -19
        g = []
        for a, b, d in ((0, 0, 1), (1, 2, 3)):
            r, f = torch.sqrt(-2 * torch.log(u23(w[a]))), 2 * math.pi * ang(w[b], w[d])
            g += [r * torch.cos(f), r * torch.sin(f)]
        ca = al[cid]
        C = [ca * C[i] + sum(L[:, i, q][cid] * g[q] for q in range(i + 1)) for i in range(3)]
        arc = ar[cid]
        e = arc + (torch.sqrt(e) * ca + torch.sqrt(arc) * g[3]) ** 2
        j0, j1 = jump[0][cid], jump[1][cid]
        if fpm:
            lev = _gillespie(lev, j0, j1, pid, step, key)
        else:
            r = (lev + 1).double()
            up = _invert(u23(w[2]), j0 ** r, lambda q, at: (q + r[at]) / (q + 1) * (1 - j0[at]))
            flip = j1 > 0.5
            pb = torch.where(flip, 1 - j1, j1).clamp(min=0.0)
            dn = _invert(u23(w[3]), (1 - pb) ** lev.double(),
                         lambda q, at: (lev[at] - q).double() / (q + 1) * (pb[at] / (1 - pb[at])),
                         lev)
            dn = torch.where(j1 >= 1, lev, torch.where(flip, lev - dn, dn))
            lev = lev + up - dn
        del w, g, j0, j1, arc, ca
        # conservation of Sec. 4.C
        wd = _philox(torch.arange(m, device=dev), step, 0x80000000, 0, key)[0]
        Id = torch.floor(N * tgt[1] / (R * th) - _sum(lev.double(), cid, m) +
                         (wd.double() + 0.5) * 2.0 ** -32).long()
        _correct(lev, o, cnt, Id, step, key)
        e = e * (tgt[0] / (_sum(e, cid, m) / N))[cid]
        mean = [_sum(v, cid, m) / N for v in C]
        C = [v - u[cid] for v, u in zip(C, mean)]
        et = 0.5 * sum(_sum(v * v, cid, m) / N for v in C)
        rad = (1.5 * R * Ttr + er + R * th * eb - tgt[0] -
               R * th * _sum(lev.double(), cid, m) / N) / et
        if bool((rad <= 0).any()):
            return None
        s = torch.sqrt(rad)[cid]
        c = [u[cid] + s * v for u, v in zip(U, C)]
    return c, e, lev, cid, N


def exact(case, seed):
    """64-bit values of a pass over relaxation cells or of the pool's moments.
    The flows (channel, gradient, plane) have none: within a pass a particle's
    cell, wall event or branch turns on the last bit of its coordinates, so two
    correct roundings are two realisations of the flow."""
    kind = case["kind"]
    if kind not in ("cells", "host", "pool"):
        return None
    m, lo, hi = case["cells"], case["nmin"], case["nmax"]
    n = m * lo if m == 1 or hi == lo else m * (hi - lo) / math.log(hi / lo)
    if n * case.get("steps", 1) > 2.0e8:          # beyond 20 seconds
        return None
    sp, off, nd, dt, p = _cells(case, seed)
    if kind == "pool":
        o = torch.from_numpy(off).cuda()
        cnt = o[1:] - o[:-1]
        cid = torch.repeat_interleave(torch.arange(m, device="cuda"), cnt)
        return {"moments": _moments(sp, m, cid, cnt.double(), p[:3], p[3], p[4])}
    r = _relax(sp, off, nd, dt, p, case["steps"], 1 + int(seed) % 1000003,
               case.get("method") == "fpm")
    if r is None:
        return None
    c, e, lev, cid, N = r
    out = {"moments": _moments(sp, m, cid, N, c, e, lev)}
    if kind == "host" or case["particles"]:
        out["state"] = c + [e, None]
    return out
