"""GPU-vs-oracle parity of the fused stencil/RHS/RK4 kernels, through the
C ABI (ctypes binding).  Gate: scaled error <= 1e-12 after one RHS and
<= 1e-10 after many RK4 steps (per variable v: |a-b| / max(|b|, max|b_v|))."""
import numpy as np
import pytest

from paper_1410_1764_gb300 import synth
from helpers import scaled_err, to_gpu, to_np

pytestmark = pytest.mark.gpu

RHS_TOL = 1e-12
RK4_TOL = 1e-10


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_1764_gb300 import api as A
    A.lib()
    return A


@pytest.mark.parametrize("dims,g,nv", [((17, 9, 11), 3, 24), ((32, 32, 32), 2, 2), ((5, 7, 4), 3, 2)])
def test_ghost_fill_bitwise(api, orc, dims, g, nv):
    nx, ny, nz = dims
    kind = api.BSSN if nv == 24 else api.WAVE
    sysm = api.make_system(kind, nx, ny, nz, 1.0 / nx, nghost=g)
    rng = np.random.default_rng(0)
    a = rng.standard_normal((nv, nz + 2 * g, ny + 2 * g, nx + 2 * g))
    t = to_gpu(a)
    sysm.fill_ghosts(t)
    want = a.copy()
    orc.fill_ghosts(want, g)
    assert np.array_equal(to_np(t), want)


def _wave_cases():
    return [(12, 16, 20), (32, 32, 32), (33, 9, 7)]


@pytest.mark.parametrize("dims", _wave_cases())
def test_wave_rhs(api, orc, dims):
    nx, ny, nz = dims
    g, h = 2, 1.0 / nx
    rng = np.random.default_rng(1)
    st = synth.pad(rng.standard_normal((2, nz, ny, nx)), g)
    orc.fill_ghosts(st, g)
    want = orc.wave_rhs(st, g, h)
    sysm = api.make_system(api.WAVE, nx, ny, nz, h)
    got = to_np(sysm.rhs(to_gpu(st)))
    assert scaled_err(got, want, g) <= RHS_TOL


def test_wave_plane_100_steps(api, orc):
    """The 32^3 plane-wave workload: 100 RK4 steps, dt = h/4."""
    n, g = 32, 2
    y0, h = synth.plane_wave(n, g)
    want = orc.rk4(orc.WAVE, y0, g, h, 0.25 * h, 100)
    sysm = api.make_system(api.WAVE, n, n, n, h)
    t = to_gpu(y0)
    sysm.rk4_step(t, 0.25 * h, 100)
    got = to_np(t)
    assert scaled_err(got, want, g) <= RK4_TOL
    assert np.array_equal(got[:, :g], got[:, n:n + g])  # ghosts refilled on return


def test_wave_pulses(api, orc):
    n, g = 48, 2
    y0, h = synth.gaussian_pulses(n, g, seed=1)
    want = orc.rk4(orc.WAVE, y0, g, h, 0.25 * h, 20)
    sysm = api.make_system(api.WAVE, n, n, n, h)
    t = to_gpu(y0)
    sysm.rk4_step(t, 0.25 * h, 20)
    assert scaled_err(to_np(t), want, g) <= RK4_TOL


@pytest.mark.parametrize("dims", [(12, 16, 20), (32, 32, 32)])
def test_varc_rhs(api, orc, dims):
    nx, ny, nz = dims
    g, h = 2, 1.0 / nx
    rng = np.random.default_rng(2)
    st = synth.pad(rng.standard_normal((2, nz, ny, nx)), g)
    orc.fill_ghosts(st, g)
    c = synth.pad(1.0 + 0.2 * rng.uniform(-1, 1, (nz, ny, nx)), g)[0]
    s = (c * c).copy()
    orc.fill_ghosts(s, g)
    want = orc.varc_rhs(st, s, g, h)
    sysm = api.make_system(api.WAVE_VARC, nx, ny, nz, h)
    sysm.set_speed(to_gpu(c))
    got = to_np(sysm.rhs(to_gpu(st)))
    assert scaled_err(got, want, g) <= RHS_TOL


def _bssn_random(dims, amp, seed, g=3):
    nx, ny, nz = dims
    rng = np.random.default_rng(seed)
    st = synth.pad(synth.BSSN_FLAT[:, None, None, None] + amp * rng.standard_normal((24, nz, ny, nx)), g)
    return st


@pytest.mark.parametrize("dims,amp", [((17, 9, 11), 1e-10), ((17, 9, 11), 3e-2), ((32, 32, 32), 1e-10),
                                      ((40, 12, 9), 3e-2)])
def test_bssn_rhs(api, orc, dims, amp):
    nx, ny, nz = dims
    g, h = 3, 1.0 / nx
    st = _bssn_random(dims, amp, seed=3)
    orc.fill_ghosts(st, g)
    want = orc.bssn_rhs(st, g, h)
    sysm = api.make_system(api.BSSN, nx, ny, nz, h)
    got = to_np(sysm.rhs(to_gpu(st)))
    assert scaled_err(got, want, g) <= RHS_TOL


@pytest.mark.parametrize("slicing,shift", [(1, 1), (2, 1), (0, 1), (1, 0)])
def test_bssn_rhs_gauge_options(api, orc, slicing, shift):
    dims = (16, 12, 10)
    g, h = 3, 1.0 / 16
    st = _bssn_random(dims, 3e-2, seed=4)
    orc.fill_ghosts(st, g)
    prm_o = orc.Params(0.1, 1.5, slicing, shift)
    want = orc.bssn_rhs(st, g, h, prm_o)
    sysm = api.make_system(api.BSSN, *dims, h, params=api.default_params(0.1, 1.5, slicing, shift))
    got = to_np(sysm.rhs(to_gpu(st)))
    assert scaled_err(got, want, g) <= RHS_TOL


def test_bssn_rk4_noise(api, orc):
    n, g = 24, 3
    st, h = synth.bssn_noise(n, n, n, g, seed=2)
    want = orc.rk4(orc.BSSN, st, g, h, 0.25 * h, 20)
    sysm = api.make_system(api.BSSN, n, n, n, h)
    t = to_gpu(st)
    sysm.rk4_step(t, 0.25 * h, 20)
    assert scaled_err(to_np(t), want, g) <= RK4_TOL


def test_bssn_rk4_strong(api, orc):
    """Large perturbations drive every nonlinear term."""
    dims = (20, 14, 12)
    g, h = 3, 1.0 / 20
    st = _bssn_random(dims, 1e-2, seed=5)
    want = orc.rk4(orc.BSSN, st, g, h, 0.25 * h, 10)
    sysm = api.make_system(api.BSSN, *dims, h)
    t = to_gpu(st)
    sysm.rk4_step(t, 0.25 * h, 10)
    assert scaled_err(to_np(t), want, g) <= RK4_TOL


@pytest.mark.slow
def test_bssn_128_rhs_full_size(api, orc):
    """The BSSN 128^3 workload (flat + 1e-10 noise): one RHS, every point."""
    n, g = 128, 3
    st, h = synth.bssn_noise(n, n, n, g, seed=2)
    orc.fill_ghosts(st, g)
    want = orc.bssn_rhs(st, g, h)
    sysm = api.make_system(api.BSSN, n, n, n, h)
    got = to_np(sysm.rhs(to_gpu(st)))
    assert scaled_err(got, want, g) <= RHS_TOL


def test_bssn_100_steps_random(api, orc):
    """100 RK4 steps of 1e-3 random perturbations of flat space: every
    variable's perturbation is resolved far above one ulp of its background,
    so the 1e-10 gate applies."""
    n, g = 24, 3
    h = 1.0 / n
    st = _bssn_random((n, n, n), 1e-3, seed=7)
    want = orc.rk4(orc.BSSN, st, g, h, 0.25 * h, 100)
    sysm = api.make_system(api.BSSN, n, n, n, h)
    t = to_gpu(st)
    sysm.rk4_step(t, 0.25 * h, 100)
    assert scaled_err(to_np(t), want, g) <= RK4_TOL


def test_bssn_100_steps_gauge_wave(api, orc):
    """100 RK4 steps of the gauge wave (harmonic slicing, frozen zero shift)."""
    from test_oracle_bssn import gauge_wave_state
    st, h = gauge_wave_state(64, 6, 6, 0.0)
    prm_o = orc.Params(0.1, 2.0, 1, 1)
    want = orc.rk4(orc.BSSN, st, 3, h, 0.25 * h, 100, params=prm_o)
    sysm = api.make_system(api.BSSN, 64, 6, 6, h, params=api.default_params(0.1, 2.0, 1, 1))
    t = to_gpu(st)
    sysm.rk4_step(t, 0.25 * h, 100)
    assert scaled_err(to_np(t), want, 3) <= RK4_TOL


@pytest.mark.slow
def test_bssn_100_steps_noise(api, orc):
    """100 RK4 steps of the flat + 1e-10 noise workload (48^3).

    This case is ill-conditioned in FP64: one ulp of an O(1) background value
    (2.2e-16) is 2e-6 of the 1e-10 perturbation, and the zero-background
    variables (At_ij) inherit it.  The oracle run on the same input with ONE
    value moved by one ulp departs from itself by e_ulp ~ 1e-5 (scaled), so no
    two FP64 evaluations with different rounding orders can agree to 1e-10
    here.  The gate is the measured conditioning bound: the GPU must stay
    within 4 e_ulp of the oracle (and the 1e-10 gate holds on the
    well-conditioned cases above)."""
    n, g = 48, 3
    st, h = synth.bssn_noise(n, n, n, g, seed=2)
    want = orc.rk4(orc.BSSN, st, g, h, 0.25 * h, 100)
    st1 = st.copy()
    st1[1, g + n // 2, g + n // 3, g + n // 4] = np.nextafter(st1[1, g + n // 2, g + n // 3, g + n // 4], 2.0)
    e_ulp = scaled_err(orc.rk4(orc.BSSN, st1, g, h, 0.25 * h, 100), want, g)
    sysm = api.make_system(api.BSSN, n, n, n, h)
    t = to_gpu(st)
    sysm.rk4_step(t, 0.25 * h, 100)
    got = to_np(t)
    e = scaled_err(got, want, g)
    assert e <= 4 * e_ulp, (e, e_ulp)
    # the variables with O(1) backgrounds agree to a few ulps of the background
    bg = [1, 4, 6, 17]
    assert np.abs(got[bg] - want[bg]).max() <= 64 * 2.2e-16


@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 3, 1), (1, 5, 2), (3, 1, 1)])
def test_degenerate_grids(api, orc, dims):
    """Grids thinner than the stencil: the periodic images cover the ghosts."""
    nx, ny, nz = dims
    rng = np.random.default_rng(12)
    for kind in ("wave", "bssn"):
        if kind == "wave":
            K, g, nv = api.WAVE, 2, 2
            st = synth.pad(rng.standard_normal((nv, nz, ny, nx)), g)
        else:
            K, g, nv = api.BSSN, 3, 24
            st = synth.pad(synth.BSSN_FLAT[:, None, None, None] + 1e-2 * rng.standard_normal((nv, nz, ny, nx)), g)
        h = 0.1
        sysm = api.make_system(K, nx, ny, nz, h)
        t = to_gpu(st)
        sysm.fill_ghosts(t)
        want_g = st.copy()
        orc.fill_ghosts(want_g, g)
        assert np.array_equal(to_np(t), want_g)
        want = orc.rhs(orc.WAVE if kind == "wave" else orc.BSSN, want_g, g, h)
        assert scaled_err(to_np(sysm.rhs(t)), want, g) <= RHS_TOL
        y = orc.rk4(orc.WAVE if kind == "wave" else orc.BSSN, st, g, h, 0.25 * h, 3)
        t2 = to_gpu(st)
        sysm.rk4_step(t2, 0.25 * h, 3)
        assert scaled_err(to_np(t2), y, g) <= RK4_TOL


def _shapes_with(api, kind, sharing):
    return [v for v in range(api.lib().chemora_variant_count(kind)) if api.variant_info(kind, v)[3] == sharing]


@pytest.mark.parametrize("dims", [(64, 12, 20), (32, 7, 37), (33, 9, 11)])
def test_wave_xz_shapes(api, orc, dims):
    """The order-4 wave's marching shapes: every shape, ragged rows (ny = 7), nz
    not a multiple of the march's depth, and nx % 32 != 0; one RHS and RK4 steps
    against the oracle."""
    nx, ny, nz = dims
    g, h = 2, 1.0 / nx
    rng = np.random.default_rng(11)
    st = synth.pad(rng.standard_normal((2, nz, ny, nx)), g)
    orc.fill_ghosts(st, g)
    want = orc.wave_rhs(st, g, h)
    y = orc.rk4(orc.WAVE, st, g, h, 0.25 * h, 8)
    shapes = _shapes_with(api, api.WAVE, 4)
    assert shapes
    for v in shapes:
        sysm = api.make_system(api.WAVE, nx, ny, nz, h)
        sysm.variant(v)
        assert scaled_err(to_np(sysm.rhs(to_gpu(st))), want, g) <= RHS_TOL, v
        t = to_gpu(st)
        sysm.rk4_step(t, 0.25 * h, 8)
        assert scaled_err(to_np(t), y, g) <= RK4_TOL, v


def test_wave_xz_plane_wave_100_steps(api, orc):
    """The 32^3 plane-wave workload, 100 RK4 steps, on a marching shape."""
    n, g = 32, 2
    y0, h = synth.plane_wave(n, g)
    want = orc.rk4(orc.WAVE, y0, g, h, 0.25 * h, 100)
    sysm = api.make_system(api.WAVE, n, n, n, h)
    sysm.variant(_shapes_with(api, api.WAVE, 4)[0])
    t = to_gpu(y0)
    sysm.rk4_step(t, 0.25 * h, 100)
    assert scaled_err(to_np(t), want, g) <= RK4_TOL
