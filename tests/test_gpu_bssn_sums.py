"""The split BSSN right-hand side's sums on the integer units (zero shift and
curvature, factors spread widely, ends of the FP64 range, every gauge) in every
block of the algebra kernel, and on both sides of the rule for its block."""
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


def _state(orc, dims, field, seed=3):
    nx, ny, nz = dims
    rng = np.random.default_rng(seed)
    p = 1e-2 * rng.standard_normal((24, nz, ny, nx))
    if field == "zero shift":
        p[18:] = 0.0
    elif field == "zero curvature":
        p[7:14] = 0.0
    elif field == "wide":
        p[8:14] *= np.exp2(rng.uniform(-40, 0, p[8:14].shape))
        p[18:] *= np.exp2(rng.uniform(-40, 0, p[18:].shape))
    elif field == "tiny":          # products below the normal range
        p[8:14] *= 1e-200
        p[18:] *= 1e-200
    elif field == "large":
        p[18:] *= 1e60
    st = synth.pad(synth.BSSN_FLAT[:, None, None, None] + p, 3)
    orc.fill_ghosts(st, 3)
    return st


@pytest.mark.parametrize("field", ["zero shift", "zero curvature", "wide", "tiny", "large"])
def test_values(api, orc, field):
    dims, h = (21, 10, 7), 0.05
    st = _state(orc, dims, field)
    want = orc.bssn_rhs(st, 3, h)
    sysm = api.make_system(api.BSSN, *dims, h)
    # rounding relative to each variable's largest value
    assert scaled_err(to_np(sysm.rhs(to_gpu(st))), want, 3) <= 1e-13


@pytest.mark.parametrize("slicing,shift", [(0, 0), (1, 0), (2, 0), (0, 1), (2, 1)])
def test_gauges(api, orc, slicing, shift):
    dims, h = (18, 9, 8), 0.05
    st = _state(orc, dims, "")
    want = orc.bssn_rhs(st, 3, h, orc.Params(0.1, 1.5, slicing, shift))
    sysm = api.make_system(api.BSSN, *dims, h, params=api.default_params(0.1, 1.5, slicing, shift))
    assert scaled_err(to_np(sysm.rhs(to_gpu(st))), want, 3) <= 1e-13


@pytest.mark.parametrize("dims", [(64, 44, 55), (64, 44, 56)])   # below and above the rule's 155,648 points
def test_block_rule(api, orc, dims):
    st = _state(orc, dims, "")
    want = orc.bssn_rhs(st, 3, 0.05)
    sysm = api.make_system(api.BSSN, *dims, 0.05)
    for v in range(4):
        sysm.variant(v)
        assert scaled_err(to_np(sysm.rhs(to_gpu(st))), want, 3) <= 1e-13, v
