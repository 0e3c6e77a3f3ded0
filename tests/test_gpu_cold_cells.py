"""Cells so cold that a relaxation time overflows: the fraction over it is 0, as the
oracle's division gives, not an invalid number."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2508_05642_gb300 import inputs as I
from paper_2508_05642_gb300 import usp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [usp.USP_FP64, usp.USP_FP32])
def test_cells_near_zero_temperature_match_oracle(precision):
    """Two particles 1e-3 to 10 m/s apart: the vibrational collision number of
    Millikan and White overflows below some 0.03 K, and the relaxation fraction
    over it is 0."""
    w = I.cylinder_flow(nx=8, ny=8, ppc=2.0)
    spd, sp = w.species, O.species(**w.species)
    gap = np.array([1e-3, 1e-2, 0.1, 1.0, 3.0, 10.0])
    m = len(gap)
    off = np.arange(m + 1, dtype=np.int64) * 2
    c = np.zeros((3, 2 * m))
    c[:, 1::2] = gap * np.array([[1.0], [0.7], [-0.4]])
    er, lev = np.linspace(1e4, 3e4, 2 * m), np.zeros(2 * m, dtype=np.int32)
    form = 1 if precision == usp.USP_FP32 else 0
    if form:
        c, er = (a.astype(np.float32).astype(np.float64) for a in (c, er))
    nd, dt = np.full(m, 1e20), np.full(m, 1e-6)
    st = O.State.from_arrays(*c, er, lev)
    O.homog_step(sp, form, 5, 0, 3, off, nd, dt, st)
    ctx = usp.usp_init_homogeneous(spd, off, nd, dt, *c, er, lev, precision=precision, seed=5)
    usp.usp_step(ctx, 3)
    got = usp.usp_get_particles(ctx)
    assert all(np.all(np.isfinite(a)) for a in got[:4])
    tol = 1e-9 if form == 0 else 1e-4
    assert np.array_equal(got[4], st.lev)
    for a, b in zip(got[:4], (st.cx, st.cy, st.cz, st.erot)):
        assert np.max(np.abs(a - b)) <= tol * max(np.max(np.abs(b)), 1e-30)
    ctx.destroy()
