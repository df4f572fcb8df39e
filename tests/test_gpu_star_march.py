"""The marching star kernels (scalar wave of every order, first-order form) at
the edges of their tiles and on values that take another path: zeros, values
far apart, the ends of the FP64 range, Inf and NaN."""
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
    if kind == "zeros":
        u *= 0.0
        u[:, nz // 2, ny // 2, nx // 2] = 1.0
    elif kind == "wide":
        u *= np.exp2(rng.uniform(-40, 0, u.shape))
    elif kind == "tiny":
        u *= 1e-300
    elif kind == "huge":
        u *= 1e300
    return u


def _systems(api, orc, kind, order, dims, field, seed):
    g, h = max(2, order // 2), 1.0 / dims[0]
    K, okind, nv = (api.WAVE, orc.WAVE, 2) if kind == "wave" else (api.WAVE1, orc.WAVE1, 5)
    st = synth.pad(_field(field, nv, dims, np.random.default_rng(seed)), g)
    orc.fill_ghosts(st, g)
    sysm = api.make_system(K, *dims, h, params=api.default_params(fd_order=order), nghost=g)
    return sysm, st, g, h, (lambda s: orc.rhs(okind, s, g, h, params=orc.default_params(order))), \
        api.lib().chemora_variant_count(K)


CASES = [("wave", 2), ("wave", 4), ("wave", 6), ("wave", 8), ("wave1", 2), ("wave1", 4), ("wave1", 6), ("wave1", 8)]


@pytest.mark.parametrize("kind,order", CASES)
@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 5, 70), (33, 9, 5), (65, 17, 2), (16, 31, 8)])
def test_tile_edges(api, orc, kind, order, dims):
    sysm, st, g, h, rhs, nvar = _systems(api, orc, kind, order, dims, "", dims[0])
    want = rhs(st)
    for v in range(nvar):
        sysm.variant(v)
        # rounding of a weighted sum relative to the field's largest derivative
        assert scaled_err(to_np(sysm.rhs(to_gpu(st))), want, g) <= 1e-14, v


@pytest.mark.parametrize("kind,order", CASES)
@pytest.mark.parametrize("field", ["zeros", "wide", "tiny", "huge"])
def test_values(api, orc, kind, order, field):
    sysm, st, g, h, rhs, nvar = _systems(api, orc, kind, order, (35, 10, 9), field, 4)
    want = rhs(st)
    for v in range(nvar):
        sysm.variant(v)
        assert scaled_err(to_np(sysm.rhs(to_gpu(st))), want, g) <= 1e-14, v


@pytest.mark.parametrize("kind,order", CASES)
def test_nonfinite(api, orc, kind, order):
    sysm, st, g, h, rhs, nvar = _systems(api, orc, kind, order, (20, 18, 19), "", 2)
    for v in range(len(st)):
        st[v, g + 4, g + 3 + v, g + 6] = np.inf
        st[v, g + 11, g + 14 - v, g + 12] = np.nan
    orc.fill_ghosts(st, g)
    want = synth.interior(rhs(st), g)
    for v in range(nvar):
        sysm.variant(v)
        got = synth.interior(to_np(sysm.rhs(to_gpu(st))), g)
        assert np.array_equal(np.isfinite(got), np.isfinite(want))
        ok = np.isfinite(want)
        assert np.abs(got[ok] - want[ok]).max() <= 1e-13 * np.abs(want[ok]).max()
