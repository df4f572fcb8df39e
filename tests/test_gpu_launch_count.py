"""chemora_launch_count: a replayed step counts the kernels of a plain one, and
capturing it counts none."""
import pytest

from paper_1410_1764_gb300 import synth
from helpers import to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_1764_gb300 import api as A
    A.lib()
    return A


def _count(api, f):
    n = api.launch_count()
    f()
    return api.launch_count() - n


# launches of a step: ghost fills, then a stage's kernels (BSSN: two field launches and one
# algebra launch per 2^20 points)
@pytest.mark.parametrize("kind,dims,chain,step", [("WAVE", (12, 9, 8), 0, 8), ("WAVE", (12, 9, 8), 1, 4),
                                                  ("WAVE_VARC", (12, 9, 8), 0, 4), ("BSSN", (12, 9, 8), 0, 16),
                                                  ("BSSN", (128, 128, 70), 0, 28)])
def test_steps(api, kind, dims, chain, step):
    import torch
    k = getattr(api, kind)
    sysm = api.make_system(k, *dims, 0.1)
    g = sysm.grid.nghost
    y = torch.zeros(sysm.grid.shape, dtype=torch.float64, device="cuda")
    if kind == "BSSN":
        y += to_gpu(synth.BSSN_FLAT)[:, None, None, None]
    if kind == "WAVE_VARC":
        sysm.set_speed(torch.ones(sysm.grid.shape[1:], dtype=torch.float64, device="cuda"))
    if kind == "WAVE":
        sysm.set_chain(chain)
    assert g >= 2
    for n in (1, 5, 5, 9):  # plain, captured and replayed, replayed; one fill besides the steps
        assert _count(api, lambda: sysm.rk4_step(y, 1e-3, n)) == n * step + 1, n


@pytest.mark.parametrize("kind,dims,step", [("WAVE", [(9, 8, 7), (5, 6, 4)], 8), ("BSSN", [(9, 8, 7), (5, 6, 4)], 16),
                                            ("BSSN", [(128, 128, 70)], 28)])
def test_batch(api, kind, dims, step):
    b = api.Batch(dims, 3 if kind == "BSSN" else 2, 0.1, kind=getattr(api, kind))
    for p in range(len(dims)):
        v = b.state(p)
        v.zero_()
        if kind == "BSSN":
            v += to_gpu(synth.BSSN_FLAT)[:, None, None, None]
    base = _count(api, lambda: b.step(1e-3, 1)) - step
    for n in (1, 4):
        assert _count(api, lambda: b.step(1e-3, n)) == n * step + base
    assert 0 <= base <= 1
