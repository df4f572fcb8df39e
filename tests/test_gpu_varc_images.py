"""RK4 steps of the variable-speed wave, whose stages write their ghost zones
themselves: interior against the oracle, ghosts equal to the periodic images, on
grids at and below the ghost width, with stale ghosts on entry, one step and
several, and no step at all."""
import numpy as np
import pytest

from paper_1410_1764_gb300 import synth
from helpers import scaled_err, to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2), (1, 5, 3), (3, 2, 9), (33, 9, 6)])
@pytest.mark.parametrize("g,steps", [(2, 0), (2, 1), (2, 5), (3, 3)])
def test_rk4(orc, dims, g, steps):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_1764_gb300 import api
    nx, ny, nz = dims
    rng, h = np.random.default_rng(steps), 1.0 / max(dims)
    c = synth.pad(1.0 + 0.2 * rng.random((1, nz, ny, nx)), g)
    orc.fill_ghosts(c, g)
    s = (c * c)
    orc.fill_ghosts(s, g)
    st = synth.pad(rng.standard_normal((2, nz, ny, nx)), g)
    want = orc.rk4(orc.WAVE_VARC, st, g, h, 0.2 * h, steps, s=s[0]) if steps else st.copy()
    orc.fill_ghosts(want, g)
    stale = np.full_like(st, 7.0)
    synth.interior(stale, g)[...] = synth.interior(st, g)
    sysm = api.make_system(api.WAVE_VARC, *dims, h, nghost=g)
    sysm.set_speed(to_gpu(c[0]))
    t = to_gpu(stale)
    sysm.rk4_step(t, 0.2 * h, steps)
    got = to_np(t)
    assert scaled_err(got, want, g) <= 1e-12  # rounding of the steps
    filled = got.copy()
    orc.fill_ghosts(filled, g)
    assert np.array_equal(got, filled)
