"""The marching kernels of the variable-speed wave and its adjoint at the edges
of their tiles, with quiescent regions (exact zeros), values far apart, the
ends of the FP64 range, and non-finite values."""
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


def _inputs(orc, dims, field, seed):
    nx, ny, nz = dims
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((2, nz, ny, nx))
    if field == "zeros":
        u *= 0.0
        u[:, nz // 2, ny // 2, nx // 2] = 1.0
    elif field == "wide":
        u *= np.exp2(rng.uniform(-40, 0, u.shape))
    elif field == "tiny":
        u *= 1e-300
    elif field == "huge":
        u *= 1e300
    c = synth.pad(1.0 + 0.3 * rng.random((1, nz, ny, nx)), 2)
    orc.fill_ghosts(c, 2)
    st = synth.pad(u, 2)
    orc.fill_ghosts(st, 2)
    return st, c[0]


def _square(orc, c):
    s = (c * c)[None].copy()
    orc.fill_ghosts(s, 2)
    return s[0]


CASES = [((1, 1, 1), ""), ((3, 5, 70), ""), ((33, 9, 5), ""), ((65, 17, 2), ""), ((16, 31, 8), ""),
         ((35, 10, 9), "zeros"), ((35, 10, 9), "wide"), ((35, 10, 9), "tiny"), ((35, 10, 9), "huge")]


@pytest.mark.parametrize("dims,field", CASES)
def test_varc_rhs(api, orc, dims, field):
    st, c = _inputs(orc, dims, field, dims[0])
    h = 1.0 / dims[0]
    want = orc.varc_rhs(st, _square(orc, c), 2, h)
    sysm = api.make_system(api.WAVE_VARC, *dims, h)
    sysm.set_speed(to_gpu(c))
    for v in range(api.lib().chemora_variant_count(api.WAVE_VARC)):
        sysm.variant(v)
        # rounding of the sums relative to the field's largest derivative
        assert scaled_err(to_np(sysm.rhs(to_gpu(st))), want, 2) <= 1e-14, v


def test_varc_nonfinite(api, orc):
    st, c = _inputs(orc, (20, 18, 19), "", 2)
    st[0, 6, 5, 8] = np.inf
    st[1, 9, 9, 9] = np.nan
    st[0, 13, 16, 14] = np.nan
    orc.fill_ghosts(st, 2)
    want = synth.interior(orc.varc_rhs(st, _square(orc, c), 2, 0.05), 2)
    sysm = api.make_system(api.WAVE_VARC, 20, 18, 19, 0.05)
    sysm.set_speed(to_gpu(c))
    got = synth.interior(to_np(sysm.rhs(to_gpu(st))), 2)
    assert np.array_equal(np.isfinite(got), np.isfinite(want))


@pytest.mark.parametrize("dims,field", [c for c in CASES if c[1] not in ("tiny", "huge")] + [((2, 3, 2), "")])
def test_adjoint(api, orc, dims, field):
    nx, ny, nz = dims
    st, c = _inputs(orc, dims, field, nx)
    h, rng = 1.0 / nx, np.random.default_rng(9)
    pts = rng.permutation(nx * ny * nz)[:3]
    recv = ((pts // (nx * ny) + 2) * (ny + 4) + (pts // nx) % ny + 2) * (nx + 4) + pts % nx + 2
    data = rng.standard_normal(len(recv))
    J, gy, gs = orc.varc_adjoint(st, _square(orc, c), 2, h, 0.2 * h, 3, 2, recv, data)
    sysm = api.make_system(api.WAVE_VARC, *dims, h)
    loss, g0, gc = api.adjoint_rk4(sysm, to_gpu(st), to_gpu(c), 0.2 * h, 3, 2, recv, data)
    assert abs(loss - J) <= 1e-13 * abs(J)
    # rounding of twelve transposed stages relative to the largest gradient
    assert scaled_err(to_np(g0), gy, 2) <= 1e-12
    assert scaled_err(to_np(gc)[None], (2 * c * gs)[None], 2) <= 1e-12
