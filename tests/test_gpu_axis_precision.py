"""Differences along one axis keep their digits where the values along the other
axes are far larger: the right-hand side is arranged so that one row's difference
alone reaches an output, and compared with the oracle relative to that row."""
import numpy as np
import pytest

from paper_1410_1764_gb300 import synth
from helpers import to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_1764_gb300 import api as A
    A.lib()
    return A


def _row(shape, axis, rng, small):
    """Values of order one with a row along `axis` (x 0, y 1, z 2) through the
    middle of the interior scaled by `small`, and the row's index."""
    u = rng.standard_normal(shape)
    at = [n // 2 for n in shape]
    at[2 - axis] = slice(None)
    u[tuple(at)] *= small
    return u, tuple(at)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("small", [2.0 ** -12, 2.0 ** -40])
def test_variable_speed(api, orc, axis, small):
    """Where the speed is zero but its gradient is not, rho_t = G_a D_a u."""
    dims, g = (14, 13, 12), 2
    h = 1.0 / 16
    shape = dims[::-1]
    rng = np.random.default_rng(axis)
    u, at = _row(shape, axis, rng, small)
    st = synth.pad(np.stack([u, np.zeros(shape)]), g)
    orc.fill_ghosts(st, g)
    along = [np.newaxis] * 3
    along[2 - axis] = slice(None)
    c = np.where(np.arange(shape[2 - axis]) % 2 == 0, 0.0, 1.0 + rng.random(shape[2 - axis]))
    c = synth.pad((np.ones(shape) * c[tuple(along)])[None], g)
    orc.fill_ghosts(c, g)
    s = c * c
    want = synth.interior(orc.varc_rhs(st, s[0], g, h), g)[1]
    sysm = api.make_system(api.WAVE_VARC, *dims, h)
    sysm.set_speed(to_gpu(c[0]))
    zero_speed = np.arange(shape[2 - axis]) % 2 == 0
    # a first difference and its product with G (at most 8 max s / 12 h + ...): some roundings of the row's values
    bound = 2.0 ** -52 * 20 * (20 * float(s.max()) / (12 * h)) * np.abs(u[at]).max() / (12 * h)
    for v in range(api.lib().chemora_variant_count(api.WAVE_VARC)):
        sysm.variant(v)
        got = synth.interior(to_np(sysm.rhs(to_gpu(st))), g)[1]
        d = np.abs(got - want)[at][zero_speed]
        assert np.abs(want[at][zero_speed]).max() > 0 and d.max() <= bound, (v, d.max(), bound)
