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


def _flat(shape):
    return synth.BSSN_FLAT[:, None, None, None] * np.ones((1,) + shape)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("small", [2.0 ** -12, 2.0 ** -40])
def test_bssn_first(api, orc, axis, small):
    """Flat space with beta^a = 1 alone, no damping and dissipation: (B^x)_t = D_a B^x."""
    dims, g, h = (19, 13, 12), 3, 1.0 / 16
    shape = dims[::-1]
    u, at = _row(shape, axis, np.random.default_rng(axis), small)
    st = _flat(shape)
    st[18 + axis], st[21] = 1.0, u
    st = synth.pad(st, g)
    orc.fill_ghosts(st, g)
    want = synth.interior(orc.bssn_rhs(st, g, h, orc.Params(0.0, 0.0, 0, 0)), g)[21]
    got = synth.interior(to_np(api.make_system(api.BSSN, *dims, h, params=api.default_params(0.0, 0.0, 0, 0))
                               .rhs(to_gpu(st))), g)[21]
    bound = 2.0 ** -52 * 20 * np.abs(u[at]).max() / (12 * h)  # some roundings of the row's values
    assert np.abs(got - want)[at].max() <= bound


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("small", [2.0 ** -12, 2.0 ** -40])
def test_bssn_second(api, orc, axis, small):
    """A constant metric of 1 along the axis and 2^60 across it: (Xt^a)_t is
    4/3 D_aa beta^a and 2^-60 of the other second derivatives."""
    dims, g, h = (19, 13, 12), 3, 1.0 / 16
    shape = dims[::-1]
    u, at = _row(shape, axis, np.random.default_rng(10 + axis), small)
    st = _flat(shape)
    for q, v in enumerate((1, 4, 6)):
        st[v] = 1.0 if q == axis else 2.0 ** 60
    st[18 + axis] = u
    st = synth.pad(st, g)
    orc.fill_ghosts(st, g)
    want = synth.interior(orc.bssn_rhs(st, g, h, orc.Params(0.0, 0.0, 0, 0)), g)[14 + axis]
    got = synth.interior(to_np(api.make_system(api.BSSN, *dims, h, params=api.default_params(0.0, 0.0, 0, 0))
                               .rhs(to_gpu(st))), g)[14 + axis]
    # the difference (weights 64), its scaling, the trace, the divergence's term and their sum, rounded on both
    # sides: eight roundings of at most 4/3 of the largest second difference
    bound = 8 * 2.0 ** -53 * 4 / 3 * 64 * np.abs(u[at]).max() / (12 * h * h)
    assert np.abs(want[at]).max() > 0 and np.abs(got - want)[at].max() <= bound
