"""A deviation that one window of the settled path sees and its neighbour
relies on: an outlier just before the second window begins (in the first
window's rows only), and at nx = 32 one in the block of the first eight
chunks.  The models settle slowly, so that 256 steps leave a visible part of
it; such a call has to go through the scans.  The filter alone, whose calls
have no adjoint that would meet the same deviation."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu
GENERAL = 5      # header word: the general scans ran


@pytest.fixture(scope="module")
def ks():
    from paper_1905_13002_gb300 import _build
    _build.build()
    import paper_1905_13002_gb300 as ks
    return ks


def run(ks, m, y, polls=0):
    model = ks.Model.create(m.F, m.Q, m.H, m.R, m.m0, m.P0, device="cuda")
    yt = torch.as_tensor(y, dtype=torch.float32, device="cuda")
    ws = ks.alloc_workspace(model, len(y))
    if polls:
        ks.set_waits(ws, wait_polls=polls)
    out = ks.smooth(model, yt, ws, filter_only=True)[:2]
    assert ks.status(ws) == ks.KS_OK
    return out, int(ws[:64].view(torch.int32)[GENERAL])


# rows 1664.. are the second window's first; 1663 belongs to the first alone
@pytest.mark.parametrize("nx", [2, 4, 6])
@pytest.mark.parametrize("at", [1650, 1663])
def test_before_the_second_window(ks, nx, at):
    m = workloads.wiener_velocity(nx // 2, q=0.2, r=1.0)
    y = np.random.default_rng(nx).standard_normal((6000, nx // 2))
    out, general = run(ks, m, y)
    assert general == 0
    y[at] = 1e6
    out, general = run(ks, m, y)
    assert general == 1
    for a, b in zip(out, run(ks, m, y, 1000000)[0]):
        assert torch.allclose(a, b, rtol=1e-5, atol=1e-5 * float(b.abs().max()))


# rows 128.. 383 are the first eight chunks
@pytest.mark.parametrize("at", [200, 383])
def test_in_the_first_chunks_nx32(ks, at):
    m = workloads.random_stable(32, 8, np.random.default_rng(32), q=0.03, lo=0.95)
    y = np.random.default_rng(5).standard_normal((3000, 8))
    out, general = run(ks, m, y)
    assert general == 0
    y[at] = 1e6
    out, general = run(ks, m, y)
    assert general == 1
    for a, b in zip(out, run(ks, m, y, 1000000)[0]):
        assert torch.allclose(a, b, rtol=1e-4, atol=1e-5 * float(b.abs().max()))
