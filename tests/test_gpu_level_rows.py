"""The FP64 jump tables cover every level that enters a step, also one that the
summation correction raised by picking the same particle more than once."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2508_05642_gb300 import inputs as I
from paper_2508_05642_gb300 import usp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncell", [2000, 140])
def test_levels_raised_twice_match_oracle(ncell):
    spd = I.n2_vhs_relaxation_species()
    sp = O.species(**spd)
    per = 600 if ncell > 152 else 520        # tabled cells; few cells take one launch
    off = np.arange(ncell + 1, dtype=np.int64) * per
    p = I.equilibrium_particles(np.random.default_rng(ncell), ncell * per, spd["m"],
                                spd["theta_v"], T_tr=15000.0, T_rot=800.0, T_vib=2500.0)
    nd = np.full(ncell, 1e23)
    dt = np.full(ncell, 0.5 * O.tau_c(sp, 1e23, 15000.0))
    st = O.State.from_arrays(p.cx, p.cy, p.cz, p.erot, p.lev)
    ctx = usp.usp_init_homogeneous(spd, off, nd, dt, p.cx, p.cy, p.cz, p.erot, p.lev,
                                   precision=usp.USP_FP64, seed=8)
    steps = 16 if ncell > 152 else 40
    for s in range(steps):
        O.homog_step(sp, 0, 8, s, 1, off, nd, dt, st)
        usp.usp_step(ctx, 1)
        assert np.array_equal(usp.usp_get_particles(ctx)[4], st.lev), s
    ctx.destroy()


@pytest.mark.parametrize("ncell,per,steps", [(20000, 4, 6), (20000, 6, 8), (150, 4, 30)])
def test_fp32_levels_raised_twice_match_oracle(ncell, per, steps):
    """FP32 form: in cells of a few particles the correction often raises one by two
    levels or more.  Levels equal the oracle's but for draws that fall between
    probabilities a rounding apart (1e-7 of each: below one cell in these runs); rows
    of an earlier step turn dozens."""
    spd = I.n2_vhs_relaxation_species()
    sp = O.species(**spd)
    off = np.arange(ncell + 1, dtype=np.int64) * per
    p = I.equilibrium_particles(np.random.default_rng(5), ncell * per, spd["m"], spd["theta_v"],
                                T_tr=15000.0, T_rot=800.0, T_vib=2500.0).astype_f32_exact()
    nd = np.full(ncell, 1e23)
    dt = np.full(ncell, 0.5 * O.tau_c(sp, 1e23, 15000.0))
    st = O.State.from_arrays(p.cx, p.cy, p.cz, p.erot, p.lev)
    ctx = usp.usp_init_homogeneous(spd, off, nd, dt, p.cx, p.cy, p.cz, p.erot, p.lev,
                                   precision=usp.USP_FP32, seed=8)
    O.homog_step(sp, 1, 8, 0, steps, off, nd, dt, st)
    usp.usp_step(ctx, steps)
    lev = usp.usp_get_particles(ctx)[4]
    ctx.destroy()
    assert (lev != st.lev).reshape(ncell, per).any(axis=1).sum() <= 1
