"""GPU tests of the size-dependent paths of the library at the sizes where they
change: one-pass moments, the tables of the FP64 draws and jumps, the channel's
one-pass sort, the per-cell passes of few cells in one kernel, the host-buffer
step's copies, the plane's sums over the sorted state and FP32 estimates of
Gillespie's method.  Each is compared with the oracle or with plain sums.

Tolerances: a sum of n FP64 terms in any order is within n 2^-53 of the sum of
the terms' magnitudes (n below 10^6 here: 1.2e-10 of it, 1e-12 for the cells of
at most 5,000); values that pass through a step's arithmetic take the
bars of the parity tests (1e-9 of the scale after a few steps)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2508_05642_gb300 import inputs as I
from paper_2508_05642_gb300 import usp

pytestmark = pytest.mark.gpu


def _moments(sp, off, c, e, lev):
    """USP_NMOM fields by plain two-pass sums, and each field's sum of
    magnitudes over n (the scale of its rounding)."""
    R = 1.380649e-23 / sp["m"]
    m = np.zeros((usp.USP_NMOM, len(off) - 1))
    s = np.zeros_like(m)
    for i in range(len(off) - 1):
        b, f = off[i], off[i + 1]
        n = f - b
        if n == 0:
            continue
        v, er, l = c[:, b:f], e[b:f], lev[b:f].astype(float)
        U = v.mean(axis=1)
        C = v - U[:, None]
        q = 0.5 * (C * C).sum(axis=0)
        rows = {1: v[0], 2: v[1], 3: v[2], 5: er / R}
        for k, (a, d) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            rows[7 + k] = C[a] * C[d]
        for k in range(3):
            rows[13 + k], rows[16 + k], rows[19 + k] = q * C[k], C[k] * er, C[k] * l * R * sp["theta_v"]
        m[0, i] = n
        s[0, i] = n
        for k, t in rows.items():
            m[k, i], s[k, i] = t.mean(), np.abs(t).mean() + np.sqrt((t * t).mean())
        m[4, i] = m[7:10, i].sum() / (3 * R)
        s[4, i] = m[4, i]
        eb = l.mean()
        m[6, i] = sp["theta_v"] / np.log1p(1 / eb) if eb > 0 else 0.0
        s[6, i] = m[6, i]
    return m, s


def _near(got, ref, bar):
    bad = np.argwhere(~(np.abs(got - ref) <= bar))
    assert len(bad) == 0, [(tuple(int(v) for v in i), float(got[tuple(i)]), float(ref[tuple(i)]),
                            float(bar[tuple(i)])) for i in bad[:8]] + [len(bad)]


SIZES = [0, 1, 2, 3, 31, 32, 33, 63, 64, 65, 127, 511, 512, 513, 1025, 4999, 0]


@pytest.mark.parametrize("ncell", [1, 17, 300, 1100])
def test_one_pass_moments_at_odd_cell_sizes(ncell):
    torch = pytest.importorskip("torch")
    sp = I.n2_vhs_relaxation_species()
    rng = np.random.default_rng(ncell)
    sizes = [5000] if ncell == 1 else (SIZES * (ncell // len(SIZES) + 1))[:ncell]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    c = 2900.0 * np.array([[1.0], [-0.2], [0.0]]) + 250.0 * rng.standard_normal((3, n))
    e = rng.exponential(6e4, n)
    lev = rng.poisson(0.3, n).astype(np.int32)
    ref, scale = _moments(sp, off, c, e, lev)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    dc, de, dl, do = [d(a) for a in c], d(e), d(lev), d(off)
    out = torch.full((usp.USP_NMOM, ncell), np.nan, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    usp.usp_moments_noalloc(sp, ncell, do.data_ptr(), *[a.data_ptr() for a in dc], de.data_ptr(),
                            dl.data_ptr(), out.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    # third moments about a shifted reference lose a little: 16 times the bar
    bar = 1e-12 * scale * 16 + 1e-300
    _near(out.cpu().numpy(), ref, bar)
    ctx = usp.usp_init_homogeneous(sp, off, np.full(ncell, 1e23), np.full(ncell, 1e-10), *c, e,
                                   lev, precision=usp.USP_FP64)
    _near(usp.usp_moments(ctx), ref, bar)
    ctx.destroy()


@pytest.mark.parametrize("sizes,T_vib", [
    ([70000], 20000.0),                 # tabled draws and jumps, levels past the table's rows
    ([65536], 1500.0),
    ([65535], 9000.0),                  # one short of the draw tables
    ([511] * 3, 3000.0),                # too small for jump tables
    ([2, 40000, 600, 31000], 12000.0),
    ([300] * 160, 4000.0),              # more cells than the one-kernel passes take
    ([2000] * 156, 20000.0),            # levels corrected by hundreds of decrements
])
def test_fp64_forms_by_size_match_oracle(sizes, T_vib):
    spd = I.n2_vhs_relaxation_species()
    sp = O.species(**spd)
    rng = np.random.default_rng(len(sizes) + sizes[0])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    p = I.equilibrium_particles(rng, int(off[-1]), spd["m"], spd["theta_v"], T_tr=15000.0,
                                T_rot=800.0, T_vib=T_vib)
    nd = np.full(len(sizes), 1e23)
    dto = np.full(len(sizes), 0.5 * O.tau_c(sp, 1e23, 15000.0))
    st = O.State.from_arrays(p.cx, p.cy, p.cz, p.erot, p.lev)
    O.homog_step(sp, 0, 11, 0, 4, off, nd, dto, st)
    ctx = usp.usp_init_homogeneous(spd, off, nd, dto, p.cx, p.cy, p.cz, p.erot, p.lev,
                                   precision=usp.USP_FP64, seed=11)
    usp.usp_step(ctx, 3)
    buf = usp.usp_save(ctx)             # the FP64 tables are not in a checkpoint
    usp.usp_step(ctx, 1)
    one = usp.usp_get_particles(ctx)
    usp.usp_load(ctx, buf)
    usp.usp_step(ctx, 1)
    for got in (one, usp.usp_get_particles(ctx)):
        assert np.array_equal(got[4], st.lev)
        for a, b in zip(got[:4], (st.cx, st.cy, st.cz, st.erot)):
            assert np.max(np.abs(a - b)) <= 1e-9 * np.max(np.abs(b))
    fl, _ = usp.usp_status(ctx)
    assert fl & usp.ERROR_FLAGS == 0
    ctx.destroy()


@pytest.mark.parametrize("ny,ppc", [(1, 70), (3, 1), (256, 20), (257, 20), (64, 512), (65, 505)])
@pytest.mark.parametrize("precision", [usp.USP_FP64, usp.USP_FP32])
def test_channel_sorts_match_oracle(ny, ppc, precision):
    """The one-pass sort ends at 256 cells and at 32,768 particles."""
    w = I.channel_poiseuille(ny=ny, ppc=ppc, steps=0)
    sp, ch = O.species(**w.species), O.channel(**w.channel)
    form = 1 if precision == usp.USP_FP32 else 0
    p = w.particles.astype_f32_exact() if form else w.particles
    y = w.y.astype(np.float32).astype(np.float64) if form else w.y
    dt = w.dt_over_tau_c * O.tau_c(sp, w.n, w.channel["T_wall"])
    st = O.ChannelState.from_arrays(y, p.cx, p.cy, p.cz, p.erot, p.lev)
    ctx = usp.usp_init_channel(w.species, w.channel, dt, y, p.cx, p.cy, p.cz, p.erot, p.lev,
                               precision=precision, seed=w.seed)
    steps = 1 if form else 5            # FP32 positions part from the oracle's at cell faces
    acc = np.zeros(ny * O.NACC + 2)
    usp.usp_channel_sample(ctx, True)
    O.channel_step(sp, form, w.seed, 0, steps, ch, dt, st, acc)
    usp.usp_step(ctx, steps)
    gy, gx, gv, gz, ge, gl, gp = usp.usp_channel_get_particles(ctx)
    if form == 0:
        assert np.array_equal(gp, st.pid) and np.array_equal(gl, st.lev)
        assert np.max(np.abs(gx - st.cx)) < 1e-8 * 300.0
        np.testing.assert_allclose(usp.usp_channel_read(ctx), acc, rtol=1e-9, atol=1e-6)
    else:
        assert np.mean(gp == st.pid) > 0.999
        a = usp.usp_channel_read(ctx)
        assert a[0:ny * O.NACC:O.NACC].sum() == len(gp)
    assert usp.usp_status(ctx)[0] & usp.ERROR_FLAGS == 0
    ctx.destroy()


@pytest.mark.parametrize("kind", ["pinned", "pageable", "in place", "crossed"])
def test_host_step_returns_the_stepped_state(kind):
    """The state comes down while later cells go up only where the buffers
    allow it; every arrangement gives the same state."""
    torch = pytest.importorskip("torch")
    w = I.batched_instances(seed=5, n_inst=40, nmin=1, nmax=9000, steps=0)
    p = w.particles.astype_f32_exact()
    n = p.n
    dt = np.array([0.5 * usp.usp_tau_c(w.species, w.ndens[i], w.T_nominal[i, 0])
                   for i in range(w.n_cells)])
    ctx = usp.usp_init_homogeneous(w.species, w.offsets, w.ndens, dt, p.cx, p.cy, p.cz, p.erot,
                                   p.lev, precision=usp.USP_FP32, seed=3)
    mk = (lambda m, t: torch.empty(m, dtype=t, pin_memory=True).numpy()) if kind != "pageable" \
        else (lambda m, t: torch.empty(m, dtype=t).numpy())
    src = [mk(n, torch.float32) for _ in range(4)] + [mk(n, torch.int32)]
    for a, b in zip(src, (p.cx, p.cy, p.cz, p.erot, p.lev)):
        a[:] = b
    mom = np.zeros((usp.USP_NMOM, w.n_cells))
    if kind == "in place":
        out = src
    elif kind == "crossed":
        # the outputs overlap the inputs, shifted: they may come down only
        # after every cell is up
        big = mk(2 * n + 64, torch.float32)
        src[0], out0 = big[:n], big[33:n + 33]
        src[0][:] = p.cx
        out = [out0] + [mk(n, torch.float32) for _ in range(3)] + [mk(n, torch.int32)]
    else:
        out = [mk(n, torch.float32) for _ in range(4)] + [mk(n, torch.int32)]
    usp.usp_step_host(ctx, *src, 2, mom, out=out)
    got = [a.copy() for a in out]
    ref = usp.usp_get_particles(ctx)        # the state the call left on the device
    for a, b in zip(got[:4], ref[:4]):
        assert np.array_equal(a, b.astype(np.float32))
    assert np.array_equal(got[4], ref[4])
    # and it is the state that the device path steps to
    ctx2 = usp.usp_init_homogeneous(w.species, w.offsets, w.ndens, dt, p.cx, p.cy, p.cz, p.erot,
                                    p.lev, precision=usp.USP_FP32, seed=3)
    usp.usp_step(ctx2, 2)
    two = usp.usp_get_particles(ctx2)
    assert np.mean(two[4] != ref[4]) < 1e-3
    assert np.max(np.abs(two[0] - ref[0])) < 1e-4 * np.max(np.abs(ref[0]))
    ctx.destroy()
    ctx2.destroy()


@pytest.mark.parametrize("precision", [usp.USP_FP64, usp.USP_FP32])
@pytest.mark.parametrize("refined", [False, True])
def test_plane_sums_are_the_particles(precision, refined):
    """Moments and time averages over the sorted state against sums of the
    particles that the context returns (cells with no, one and many
    particles)."""
    kw = dict(amr_levels=3, amr_r2=0.24, amr_r3=0.16) if refined else {}
    w = I.cylinder_flow(nx=32, ny=24, ppc=5.0, **kw)
    p = w.particles
    dt = w.dt_over_tau_c * usp.usp_tau_c(w.species, w.plane["n_inf"], w.plane["T_inf"])
    ctx = usp.usp_init_plane(w.species, w.plane, dt, w.area_frac, w.x, w.y, p.cx, p.cy, p.cz,
                             p.erot, p.lev, w.capacity, precision=precision, seed=4)
    before = usp.usp_moments(ctx)           # a state that no step has sorted
    usp.usp_step(ctx, 5)
    usp.usp_sample(ctx, True)
    usp.usp_step(ctx, 1)
    x, y, cx, cy, cz, er, lev, pid = usp.usp_plane_get_particles(ctx)
    mom = usp.usp_moments(ctx)
    acc = usp.usp_sample_read(ctx)
    nc = ctx.n_cells
    assert before[0].sum() == len(w.x) and mom[0].sum() == len(x)
    assert (mom[0] == 0).any() and (mom[0] == 1).any()
    off = np.concatenate([[0], np.cumsum(mom[0].astype(np.int64))])
    c = np.stack([cx, cy, cz])
    ref, scale = _moments(w.species, off, c, er, lev)
    _near(mom, ref, 16e-12 * scale + 1e-300)
    a = acc[:nc * 12].reshape(nc, 12)
    seg = lambda t: np.add.reduceat(np.append(t, 0.0), off[:-1]) * (mom[0] > 0)
    terms = [np.ones(len(x)), cx, cy, cz, cx * cx, cy * cy, cz * cz, cx * cy, cx * cz, cy * cz, er,
             lev.astype(float)]
    for k, t in enumerate(terms):
        _near(a[:, k], seg(t), 1e-12 * seg(np.abs(t)) + 1e-9 * (k > 0))
    assert acc[nc * 12] == 1.0
    ctx.destroy()


@pytest.mark.parametrize("precision", [usp.USP_FP64, usp.USP_FP32])
@pytest.mark.parametrize("T", [300.0, 4000.0, 20000.0])
def test_gillespie_levels_match_oracle(precision, T):
    """The levels of the first-order method, from cold cells (rates near
    zero) to ones where a particle makes many transitions a step."""
    spd = I.n2_vhs_relaxation_species()
    sp = O.species(**spd)
    n = 60000
    rng = np.random.default_rng(int(T))
    p = I.equilibrium_particles(rng, n, spd["m"], spd["theta_v"], T_tr=T, T_rot=T, T_vib=0.7 * T)
    form = 1 if precision == usp.USP_FP32 else 0
    p = p.astype_f32_exact() if form else p
    off, nd = np.array([0, n], dtype=np.int64), np.array([1e23])
    dt = np.array([1.5 * O.tau_c(sp, 1e23, T)])
    st = O.State.from_arrays(p.cx, p.cy, p.cz, p.erot, p.lev)
    O.homog_step_fpm(sp, form, 7, 0, 1, off, nd, dt, st)
    ctx = usp.usp_init_homogeneous(spd, off, nd, dt, p.cx, p.cy, p.cz, p.erot, p.lev,
                                   precision=precision, seed=7, method=usp.USP_METHOD_FPM)
    usp.usp_step(ctx, 1)
    lev = usp.usp_get_particles(ctx)[4]
    # FP32 rates differ from the oracle's in the last bit: a few decisions turn
    assert np.sum(lev != st.lev) <= (0 if form == 0 else 20)
    ctx.destroy()


@pytest.mark.parametrize("precision", [usp.USP_FP64, usp.USP_FP32])
@pytest.mark.parametrize("nx", [181, 182])          # 32,761 and 33,124 cells
def test_plane_sums_on_both_sides_of_the_warp_per_cell_rule(precision, nx):
    w = I.cylinder_flow(nx=nx, ny=nx, ppc=3.0)
    p = w.particles
    dt = w.dt_over_tau_c * usp.usp_tau_c(w.species, w.plane["n_inf"], w.plane["T_inf"])
    ctx = usp.usp_init_plane(w.species, w.plane, dt, w.area_frac, w.x, w.y, p.cx, p.cy, p.cz,
                             p.erot, p.lev, w.capacity, precision=precision, seed=4)
    assert (ctx.n_cells <= 32768) == (nx == 181)
    usp.usp_sample(ctx, True)
    usp.usp_step(ctx, 2)
    cx, cy, cz, er, lev = usp.usp_plane_get_particles(ctx)[2:7]
    mom = usp.usp_moments(ctx)
    off = np.concatenate([[0], np.cumsum(mom[0].astype(np.int64))])
    pick = np.linspace(0, ctx.n_cells - 1, 900).astype(int)
    ref, scale = [], []
    c = np.stack([cx, cy, cz])
    for i in pick:
        k = slice(off[i], off[i + 1])
        r, s = _moments(w.species, np.array([0, off[i + 1] - off[i]]), c[:, k], er[k], lev[k])
        ref.append(r[:, 0])
        scale.append(s[:, 0])
    _near(mom[:, pick], np.array(ref).T, 16e-12 * np.array(scale).T + 1e-300)
    ctx.destroy()


@pytest.mark.parametrize("precision", [usp.USP_FP64, usp.USP_FP32])
@pytest.mark.parametrize("ncell", [40, 400])        # one compute kernel a run, or three
def test_host_step_reads_every_input_before_it_writes_an_overlapping_output(precision, ncell):
    """Pinned outputs half a state away from the inputs they overlap, within one
    field and across two: what a first run of cells sends down lies where the later
    runs still come from."""
    torch = pytest.importorskip("torch")
    spd = I.n2_vhs_relaxation_species()
    sizes = np.random.default_rng(ncell).integers(1, 2 * (3_000_000 // ncell), ncell)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    p = I.equilibrium_particles(np.random.default_rng(1), n, spd["m"], spd["theta_v"],
                                T_tr=15000.0, T_rot=800.0, T_vib=2500.0)
    p = p.astype_f32_exact()
    nd = np.full(ncell, 1e23)
    dt = np.full(ncell, 0.5 * usp.usp_tau_c(spd, 1e23, 15000.0))
    new = lambda: usp.usp_init_homogeneous(spd, off, nd, dt, p.cx, p.cy, p.cz, p.erot, p.lev,
                                           precision=precision, seed=3)
    ft = torch.float32 if precision == usp.USP_FP32 else torch.float64
    mk = lambda m, t: torch.empty(m, dtype=t, pin_memory=True).numpy()
    ctx = new()
    usp.usp_step(ctx, 1)
    ref = usp.usp_get_particles(ctx)
    ctx.destroy()
    h = n // 2
    # x comes down into x half a state on; y into the half of z's input
    bx, bz = mk(n + h, ft), mk(n + h, ft)
    src = [bx[:n], mk(n, ft), bz[:n], mk(n, ft), mk(n, torch.int32)]
    out = [bx[h:], bz[h:], mk(n, ft), mk(n, ft), mk(n, torch.int32)]
    for a, b in zip(src, (p.cx, p.cy, p.cz, p.erot, p.lev)):
        a[:] = b
    mom = np.zeros((usp.USP_NMOM, ncell))
    ctx = new()
    usp.usp_step_host(ctx, *src, 1, mom, out=out)
    # the sums are atomic, so that two runs part by roundings
    assert np.mean(out[4] != ref[4]) < 1e-5
    for a, b in zip(out[:4], ref[:4]):
        assert np.max(np.abs(a - b)) < 1e-4 * np.max(np.abs(b))
    ctx.destroy()


@pytest.mark.parametrize("nx", [24, 184])           # a warp and four lanes per cell
def test_plane_fields_of_cells_whose_first_particle_is_far_out(nx):
    """The energy of an FP64 cell is kept to the rounding of its fields, which
    central sums give whatever the particles' order: about the first particle, 20
    thermal speeds out, they lose a factor of 200 (400 particles: variance 2, squares
    400 in units of the thermal speed).  Central sums of 400 terms are good to some
    3e-16 (random roundings), the others to some 3e-14; the bar lies between."""
    w = I.cylinder_flow(nx=nx, ny=nx, ppc=1.0, cylinder=False)
    pl = dict(w.plane, bc=(I.BC_SPECULAR,) * 4, inflow=(0,) * 4)
    sp = w.species
    R = 1.380649e-23 / sp["m"]
    rng = np.random.default_rng(nx)
    ci, cj = (a.ravel() for a in np.meshgrid(np.arange(1, 23, 3), np.arange(1, 23, 3)))
    N, m = 400, len(ci)
    h = ((pl["x1"] - pl["x0"]) / nx, (pl["y1"] - pl["y0"]) / nx)
    x = np.repeat(pl["x0"] + (ci + 0.5) * h[0], N)
    y = np.repeat(pl["y0"] + (cj + 0.5) * h[1], N)
    s = np.sqrt(R * 200.0)
    c = s * rng.standard_normal((3, m * N))
    c[:, ::N] += 20.0 * s * rng.standard_normal((3, m)) / np.sqrt(3.0)
    er, lev = rng.exponential(R * 200.0, m * N), np.zeros(m * N, dtype=np.int32)
    ctx = usp.usp_init_plane(sp, pl, 1e-12, w.area_frac, x, y, *c, er, lev, 2 * m * N,
                             precision=usp.USP_FP64, seed=2)
    usp.usp_step(ctx, 1)
    g = usp.usp_plane_get_particles(ctx)
    W = np.longdouble
    energy = lambda c, e, l: (0.5 * (W(c) ** 2).sum(axis=0) + W(e) +
                              W(l) * W(R) * W(sp["theta_v"])).reshape(m, N).sum(axis=1)
    before, after = energy(c, er, lev), energy(np.stack(g[2:5]), g[5], g[6])
    assert np.array_equal(np.sort(g[7].reshape(m, N), axis=1),
                          np.arange(m * N).reshape(m, N))        # every particle in its cell
    err = np.abs(after / before - 1)
    assert np.sqrt(np.mean(err.astype(float) ** 2)) < 3e-15, float(err.max())
    ctx.destroy()


@pytest.mark.parametrize("precision,nx", [(usp.USP_FP64, 8), (usp.USP_FP64, 184), (usp.USP_FP32, 8)])
def test_plane_averages_of_levels_beyond_31_bits(precision, nx):
    """A cell of 64 particles at rest (no temperature, so no collision) whose levels add up
    to 34 bits, and to more than 31 in every lane's share."""
    w = I.cylinder_flow(nx=nx, ny=nx, ppc=1.0, cylinder=False)
    pl = dict(w.plane, bc=(I.BC_SPECULAR,) * 4, inflow=(0,) * 4)
    n = 64
    at = lambda a, b: np.full(n, a + (b - a) * 2.5 / nx)      # cell (2, 2)
    z = np.zeros(n)
    lev = np.full(n, (1 << 30) + 12345, dtype=np.int32)
    ctx = usp.usp_init_plane(w.species, pl, 1e-9, w.area_frac, at(pl["x0"], pl["x1"]),
                             at(pl["y0"], pl["y1"]), z, z, z, np.full(n, 1e4), lev, 2 * n,
                             precision=precision, seed=2)
    usp.usp_sample(ctx, True)
    usp.usp_step(ctx, 1)
    acc = usp.usp_sample_read(ctx)[:nx * nx * 12].reshape(-1, 12)
    assert np.array_equal(usp.usp_plane_get_particles(ctx)[6], lev)
    assert acc[2 * nx + 2, 0] == n and acc[2 * nx + 2, 11] == lev.sum(dtype=np.int64)
    assert acc[:, 11].sum() == lev.sum(dtype=np.int64)
    ctx.destroy()


@pytest.mark.parametrize("precision", [usp.USP_FP64, usp.USP_FP32])
@pytest.mark.parametrize("steps_tau", [7.0, 9.0, 20.0, 25.0, 200.0])
def test_gillespie_levels_of_hot_cells_match_oracle(precision, steps_tau):
    """Cells on both sides of the mean transitions a step (21 and 27, 59 and 74) from
    which the exact loop is run at once, and far above.  A rounding of a rate or a
    logarithm moves a particle's time by 1e-7 of it, which turns a last transition
    for some 1e-7 times their number of the particles: a few of 60,000."""
    spd = I.n2_vhs_relaxation_species()
    sp = O.species(**spd)
    n, T = 60000, 8000.0
    p = I.equilibrium_particles(np.random.default_rng(9), n, spd["m"], spd["theta_v"], T_tr=T,
                                T_rot=T, T_vib=0.9 * T).astype_f32_exact()
    form = 1 if precision == usp.USP_FP32 else 0
    off, nd = np.array([0, n], dtype=np.int64), np.array([1e23])
    dt = np.array([steps_tau * O.tau_c(sp, 1e23, T)])
    st = O.State.from_arrays(p.cx, p.cy, p.cz, p.erot, p.lev)
    O.homog_step_fpm(sp, form, 7, 0, 1, off, nd, dt, st)
    ctx = usp.usp_init_homogeneous(spd, off, nd, dt, p.cx, p.cy, p.cz, p.erot, p.lev,
                                   precision=precision, seed=7, method=usp.USP_METHOD_FPM)
    usp.usp_step(ctx, 1)
    lev = usp.usp_get_particles(ctx)[4]
    assert np.sum(lev != st.lev) <= (0 if form == 0 else 20)
    ctx.destroy()


def test_plane_moments_between_a_capture_and_its_first_replay():
    """Steps captured into a caller's graph have not sorted the state yet: moments in
    between are those of the state as it is, and after the replay those of the steps."""
    torch = pytest.importorskip("torch")
    w = I.cylinder_flow(nx=32, ny=24, ppc=5.0)
    p = w.particles
    dt = w.dt_over_tau_c * usp.usp_tau_c(w.species, w.plane["n_inf"], w.plane["T_inf"])
    s = torch.cuda.Stream()
    new = lambda **kw: usp.usp_init_plane(w.species, w.plane, dt, w.area_frac, w.x, w.y, p.cx,
                                          p.cy, p.cz, p.erot, p.lev, w.capacity,
                                          precision=usp.USP_FP64, seed=4, **kw)
    ctx = new(stream=s.cuda_stream, use_graph=False)
    before = usp.usp_moments(ctx)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        usp.usp_step(ctx, 2)            # an even number: the state's buffers alternate
    close = lambda a, b: np.max(np.abs(a - b) / (np.max(np.abs(b), axis=1, keepdims=True) + 1e-300))
    assert close(usp.usp_moments(ctx), before) < 1e-9      # sums by atomics
    with torch.cuda.stream(s):
        g.replay()
    torch.cuda.synchronize()
    after = usp.usp_moments(ctx)
    ref = new()
    usp.usp_step(ref, 2)
    assert close(after, usp.usp_moments(ref)) < 1e-9 and close(after, before) > 1e-3
    ctx.destroy()
    ref.destroy()


def _rest_error(U, c, off):
    """rms over the cells of a mean velocity's error in units of the speed's spread over
    sqrt(n), which is the size of the mean itself in a gas at rest."""
    W = np.longdouble
    e = []
    for i in range(len(off) - 1):
        v = c[:, off[i]:off[i + 1]]
        e.append((U[:, i] - W(v).mean(axis=1)).astype(float) / (v.std(axis=1) / np.sqrt(v.shape[1])))
    return float(np.sqrt(np.mean(np.square(e))))


@pytest.mark.parametrize("form", ["pool", "context"])
@pytest.mark.parametrize("ncell", [16, 640])
def test_mean_velocities_of_large_cells_at_rest(form, ncell):
    """About the mean the partial sums of n speeds are sqrt(n) large, and the mean is good to some
    6e-16 of itself; about a velocity a fifth of a thermal speed off they are up to sqrt(n) / 5
    times larger, and it is off by 4e-15 and more.  The bar lies between."""
    torch = pytest.importorskip("torch")
    sp = I.n2_vhs_relaxation_species()
    rng = np.random.default_rng(ncell)
    lo, hi = (10000, 40000) if ncell < 100 else (5000, 8000)
    off = np.concatenate([[0], np.cumsum(rng.integers(lo, hi, ncell))]).astype(np.int64)
    n = int(off[-1])
    c = 250.0 * rng.standard_normal((3, n))
    e, lev = rng.exponential(6e4, n), np.zeros(n, dtype=np.int32)
    if form == "context":
        ctx = usp.usp_init_homogeneous(sp, off, np.full(ncell, 1e23), np.full(ncell, 1e-10), *c, e,
                                       lev, precision=usp.USP_FP64)
        U = usp.usp_moments(ctx)[1:4]
        ctx.destroy()
    else:
        d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (off, *c, e, lev)]
        out = torch.empty((usp.USP_NMOM, ncell), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        usp.usp_moments_noalloc(sp, ncell, *[a.data_ptr() for a in d], out.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        U = out.cpu().numpy()[1:4]
    assert _rest_error(U, c, off) < 1.5e-15, _rest_error(U, c, off)


@pytest.mark.parametrize("ncell", [3, 700])
def test_moments_of_velocities_beyond_fp32(ncell):
    """The reference velocity is formed in FP32: what that has no number for leaves it finite."""
    torch = pytest.importorskip("torch")
    sp = I.n2_vhs_relaxation_species()
    rng = np.random.default_rng(ncell)
    off = np.arange(ncell + 1, dtype=np.int64) * 50
    n = int(off[-1])
    c = rng.standard_normal((3, n)) * np.repeat(10.0 ** rng.choice([-60, -41, 2, 37.5, 38.5, 60], ncell), 50)
    c[0, :50] = 0.0
    e, lev = rng.exponential(6e4, n), np.zeros(n, dtype=np.int32)
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (off, *c, e, lev)]
    out = torch.empty((usp.USP_NMOM, ncell), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    usp.usp_moments_noalloc(sp, ncell, *[a.data_ptr() for a in d], out.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    ref, scale = _moments(sp, off, c, e, lev)
    _near(out.cpu().numpy()[:13], ref[:13], 1.6e-11 * scale[:13] + 1e-300)
