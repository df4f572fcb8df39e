"""Kernels whose stencils run on the integer units, where the values make them
take another path: zeros, values far below their neighbours, numbers at the
ends of the FP64 range, Inf and NaN; and at the edges of their tiles."""
import numpy as np
import pytest

from paper_1410_1764_gb300 import synth
from helpers import scaled_err, to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_1764_gb300 import api as A
    A.lib()
    return A


def _field(kind, nv, dims, rng):
    nx, ny, nz = dims
    u = rng.standard_normal((nv, nz, ny, nx))
    if kind == "zeros":                       # one live point in a field of zeros
        u *= 0.0
        u[:, nz // 2, ny // 2, nx // 2] = 1.0
    elif kind == "wide":                      # neighbours up to 2^40 apart
        u *= np.exp2(rng.uniform(-40, 0, u.shape))
    elif kind == "tiny":                      # near the smallest normal numbers
        u *= 1e-300
    elif kind == "huge":
        u *= 1e300
    return u


@pytest.mark.parametrize("kind", ["zeros", "wide", "tiny", "huge"])
@pytest.mark.parametrize("dims", [(33, 9, 7), (5, 3, 4)])
def test_wave_values(api, orc, kind, dims):
    nx, ny, nz = dims
    g, h = 2, 1.0 / nx
    st = synth.pad(_field(kind, 2, dims, np.random.default_rng(1)), g)
    orc.fill_ghosts(st, g)
    want = orc.wave_rhs(st, g, h)
    sysm = api.make_system(api.WAVE, nx, ny, nz, h)
    for v in range(api.lib().chemora_variant_count(api.WAVE)):
        sysm.variant(v)
        # rounding of a 13-point sum relative to the field's largest derivative
        assert scaled_err(to_np(sysm.rhs(to_gpu(st))), want, g) <= 1e-14, v


def test_wave_nonfinite(api, orc):
    """Inf and NaN spread to exactly the points whose stencil reads them."""
    dims, g = (12, 8, 9), 2
    st = synth.pad(np.random.default_rng(2).standard_normal((2,) + dims[::-1]), g)
    st[0, g + 4, g + 3, g + 6] = np.inf
    st[0, g + 6, g + 5, g + 2] = np.nan
    orc.fill_ghosts(st, g)
    want = synth.interior(orc.wave_rhs(st, g, 1.0 / 12), g)
    sysm = api.make_system(api.WAVE, *dims, 1.0 / 12)
    got = synth.interior(to_np(sysm.rhs(to_gpu(st))), g)
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    ok = np.isfinite(want)
    assert np.abs(got[ok] - want[ok]).max() <= 1e-13 * np.abs(want[ok]).max()


@pytest.mark.parametrize("dims", [(31, 9, 3), (32, 8, 2), (33, 17, 3), (65, 3, 2), (1, 40, 2), (8, 33, 2), (2, 1, 1)])
def test_bssn_field_tiles(api, orc, dims):
    """The split BSSN right-hand side at its tiles' edges (tiles of at most 32
    x 32 points, 256 in all), with variables that are exactly constant, zero,
    and spread over 2^30."""
    nx, ny, nz = dims
    g, h = 3, 0.05
    rng = np.random.default_rng(nx)
    p = 1e-2 * rng.standard_normal((24, nz, ny, nx))
    p[0] = 0.0                                               # phi: all zero
    p[7] *= np.exp2(rng.uniform(-30, 0, p[7].shape))          # K: wide
    p[17] = 0.0                                              # alpha: constant
    st = synth.pad(synth.BSSN_FLAT[:, None, None, None] + p, g)
    orc.fill_ghosts(st, g)
    want = orc.bssn_rhs(st, g, h)
    sysm = api.make_system(api.BSSN, nx, ny, nz, h)
    for v in range(8):                                       # the algebra kernel's five blocks
        sysm.variant(v)
        assert scaled_err(to_np(sysm.rhs(to_gpu(st))), want, g) <= 1e-13, v


def test_bssn_flat_and_nonfinite(api, orc):
    """Exactly flat space has an exactly zero right-hand side; a NaN reaches
    the points whose stencils read it, and only those."""
    dims, g = (20, 11, 9), 3
    st = synth.pad(synth.BSSN_FLAT[:, None, None, None] + np.zeros((24,) + dims[::-1]), g)
    orc.fill_ghosts(st, g)
    sysm = api.make_system(api.BSSN, *dims, 0.05)
    assert not np.any(to_np(sysm.rhs(to_gpu(st))))
    st[5, g + 4, g + 5, g + 10] = np.nan
    orc.fill_ghosts(st, g)
    want = synth.interior(orc.bssn_rhs(st, g, 0.05), g)
    got = synth.interior(to_np(sysm.rhs(to_gpu(st))), g)
    assert np.array_equal(np.isnan(got), np.isnan(want))


def test_bssn_rhs_without_a_workspace(api, orc):
    """A first right-hand side on a stream that is being captured: it finds no
    workspace of the system's, and the graph replays it."""
    import torch
    dims, g = (21, 10, 8), 3
    rng = np.random.default_rng(5)
    st = synth.pad(synth.BSSN_FLAT[:, None, None, None] + 1e-2 * rng.standard_normal((24,) + dims[::-1]), g)
    orc.fill_ghosts(st, g)
    want = orc.bssn_rhs(st, g, 0.05)
    sysm = api.make_system(api.BSSN, *dims, 0.05)
    t, out = to_gpu(st), torch.zeros(st.shape, dtype=torch.float64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sysm.rhs(t, out)
    graph.replay()
    assert scaled_err(to_np(out), want, g) <= 1e-13
    assert scaled_err(to_np(sysm.rhs(t)), to_np(out), g) <= 1e-13
