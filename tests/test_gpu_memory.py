"""FP64 contexts in a memory pool of limited size: the tables of draws and jumps are
taken only where they fit beside everything else, and every call works without
them, with the same results."""
import numpy as np
import pytest

from paper_2508_05642_gb300 import inputs as I
from paper_2508_05642_gb300 import usp

pytestmark = pytest.mark.gpu

DRAWS = (1 << 23) * 8 + (1 << 18) * 16


class _Pool:
    """Device memory of at most ``limit`` bytes; records the requests."""

    def __init__(self, limit=1 << 62):
        import torch
        self.limit, self.used, self.live, self.log = limit, 0, {}, []
        dev = torch.cuda.current_device()

        @usp.ALLOC_FN
        def _alloc(nbytes, user):
            if self.used + nbytes > self.limit:
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), dev)
            self.used += nbytes
            self.live[p] = nbytes
            self.log.append(nbytes)
            return p

        @usp.FREE_FN
        def _free(ptr, user):
            nbytes = self.live.pop(ptr)
            self.used -= nbytes
            self.log.append(-nbytes)
            torch.cuda.caching_allocator_delete(ptr)

        self.fns = (_alloc, _free, None)

    def peak(self, without):
        """The most in use at a time, requests of the sizes ``without`` left out."""
        rest = [b for b in self.log if abs(b) not in without]
        return int(np.max(np.cumsum(rest)))


def _cells(n, ncell):
    spd = I.n2_vhs_relaxation_species()
    off = np.linspace(0, n, ncell + 1).astype(np.int64)
    p = I.equilibrium_particles(np.random.default_rng(n), n, spd["m"], spd["theta_v"],
                                T_tr=15000.0, T_rot=800.0, T_vib=4000.0)
    dt = np.full(ncell, 0.5 * usp.usp_tau_c(spd, 1e23, 15000.0))
    rows, guides = 4 * ncell * 32 * 48, ncell * 32 * 256

    def run(fns):
        ctx = usp.usp_init_homogeneous(spd, off, np.full(ncell, 1e23), dt, p.cx, p.cy, p.cz,
                                       p.erot, p.lev, precision=usp.USP_FP64, seed=3,
                                       allocator=fns)
        usp.usp_step(ctx, 2)
        got = usp.usp_get_particles(ctx)
        buf = [np.empty(n) for _ in range(4)] + [np.empty(n, dtype=np.int32)]
        mom = np.zeros((usp.USP_NMOM, ncell))
        usp.usp_step_host(ctx, p.cx, p.cy, p.cz, p.erot, p.lev, 1, mom, out=buf)
        ctx.destroy()
        return list(got) + buf

    return run, {DRAWS, rows, guides}


def _flow(kind):
    if kind == "channel":
        w = I.channel_poiseuille(ny=32, ppc=2100)
        dt = w.dt_over_tau_c * usp.usp_tau_c(w.species, w.n, w.channel["T_wall"])
    else:
        w = I.cylinder_flow(nx=60, ny=40, ppc=30.0)
        dt = w.dt_over_tau_c * usp.usp_tau_c(w.species, w.plane["n_inf"], w.plane["T_inf"])
    p = w.particles
    assert p.n > 65536

    def run(fns):
        if kind == "channel":
            ctx = usp.usp_init_channel(w.species, w.channel, dt, w.y, p.cx, p.cy, p.cz, p.erot,
                                       p.lev, precision=usp.USP_FP64, seed=3, allocator=fns)
        else:
            ctx = usp.usp_init_plane(w.species, w.plane, dt, w.area_frac, w.x, w.y, p.cx, p.cy,
                                     p.cz, p.erot, p.lev, w.capacity, precision=usp.USP_FP64,
                                     seed=3, allocator=fns)
        usp.usp_step(ctx, 2)
        got = usp.usp_channel_get_particles(ctx) if kind == "channel" else \
            usp.usp_plane_get_particles(ctx)
        usp.usp_moments(ctx)
        ctx.destroy()
        return list(got)

    return run, {DRAWS}


@pytest.mark.parametrize("kind", ["few cells", "cells", "tuned", "channel", "plane"])
def test_tables_are_done_without(kind):
    run, optional = {"few cells": lambda: _cells(70000, 100), "cells": lambda: _cells(150000, 200),
                     "tuned": lambda: _cells((1 << 20) + 4096, 1500)}.get(kind, lambda: _flow(kind))()
    pool = _Pool()
    ref = run(pool.fns)
    assert not pool.live and any(b in optional for b in pool.log)
    least, most = pool.peak(optional), pool.peak(())
    assert least < most
    for limit in (least, least + (most - least) // 2, most):
        p = _Pool(limit)
        got = run(p.fns)
        assert not p.live
        taken = {b for b in p.log if b in optional}
        assert taken == (optional & set(pool.log) if limit == most else taken)
        assert limit > least or not taken
        for a, b in zip(got, ref):
            if a.dtype.kind != "f":
                assert np.array_equal(a, b)
            else:       # the sums of two runs differ in their order
                assert np.max(np.abs(a - b)) <= 1e-11 * np.max(np.abs(b))
