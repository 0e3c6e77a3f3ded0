"""The trial launches that pick a context's collision kernel work on a copy of
the state in a scratch buffer; nothing is written past the end of any buffer
that the context asked for, whatever the particle and cell counts round to."""
import numpy as np
import pytest

from paper_2508_05642_gb300 import inputs as I
from paper_2508_05642_gb300 import usp

pytestmark = pytest.mark.gpu

GUARD, MARK = 256, 0xA5


@pytest.mark.parametrize("precision", [usp.USP_FP32, usp.USP_FP64])
@pytest.mark.parametrize("ncell", [1, 2, 3])
@pytest.mark.parametrize("extra", [0, 1, 33])
def test_buffers_are_not_overrun(precision, ncell, extra):
    torch = pytest.importorskip("torch")
    spd = I.n2_vhs_relaxation_species()
    n = (1 << 20) + extra
    off = np.linspace(0, n, ncell + 1).astype(np.int64)
    p = I.equilibrium_particles(np.random.default_rng(0), n, spd["m"], spd["theta_v"],
                                T_tr=8000.0, T_rot=8000.0, T_vib=8000.0)
    arena = torch.full((1 << 29,), MARK, dtype=torch.uint8, device="cuda")
    base = arena.data_ptr()
    top, guards = [(-base) % 256], []
    torch.cuda.synchronize()

    @usp.ALLOC_FN
    def alloc(nbytes, user):
        a = top[0]
        if a + nbytes + GUARD > arena.numel():
            return None
        guards.append(a + nbytes)
        top[0] = (a + nbytes + GUARD + 255) // 256 * 256
        return base + a

    @usp.FREE_FN
    def free(ptr, user):
        pass

    ctx = usp.usp_init_homogeneous(spd, off, np.full(ncell, 1e23), np.full(ncell, 1e-10), p.cx,
                                   p.cy, p.cz, p.erot, p.lev, precision=precision,
                                   allocator=(alloc, free, None))
    torch.cuda.synchronize()
    assert len(guards) > 5
    for g in guards:
        assert bool((arena[g:g + GUARD] == MARK).all()), g
    ctx.destroy()
