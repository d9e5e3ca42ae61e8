"""The settled path's head under priors far wider than the settled covariance:
no smoothed covariance may lose the digits by which the prior exceeds it, and
where a prior is wide along coordinates the call stays on the settled path."""
import numpy as np
import pytest
import torch

import oracle
import parity
import workloads

pytestmark = pytest.mark.gpu
GENERAL = 5      # header word: the general scans ran


@pytest.fixture(scope="module")
def ks():
    from paper_1905_13002_gb300 import _build
    _build.build()
    import paper_1905_13002_gb300 as ks
    return ks


def run(ks, m, y):
    model = ks.Model.create(m.F, m.Q, m.H, m.R, m.m0, m.P0, u=m.u, d=m.d, device="cuda")
    yt = torch.as_tensor(y, dtype=torch.float32, device="cuda")
    ws = ks.alloc_workspace(model, len(y))
    out = ks.smooth(model, yt, ws)
    assert ks.status(ws) == ks.KS_OK
    return [t.cpu().numpy() for t in out], int(ws[:64].view(torch.int32)[GENERAL])


# In 64 bits the head's Skeel condition is at most 40 for these models, so that
# its FP32 inverse and products lose at most 40 x 2 eps32 = 1e-5 (the difference
# P_k - P_k (I + O D)^-1 O P_k lost 1.4e-4 at P_0 = 1000 I)
@pytest.mark.parametrize("nx", [2, 4, 6])
@pytest.mark.parametrize("p0", [30.0, 1e3, 1e5])
@pytest.mark.parametrize("T", [20, 128, 300, 3000])
def test_wide_along_coordinates(ks, nx, p0, T):
    m = workloads.wiener_velocity(nx // 2, q=1.0, r=1.0, P0=p0 * np.eye(nx))
    _, y = workloads.simulate(m, T, np.random.default_rng(nx + T))
    out, general = run(ks, m, y)
    assert general == 0
    ref = oracle.kf_rts(m, y)
    assert parity.cov_err(out[1], ref[1]) < 1e-5 and parity.cov_err(out[3], ref[3]) < 1e-5
    parity.check_all(out, ref)


# wide across coordinates: P_0 itself in FP32 leaves p0 eps32 of the observed
# directions, in the scans as in the head
@pytest.mark.parametrize("nx", [8, 32])
@pytest.mark.parametrize("p0", [10.0, 100.0])
def test_wide_across_coordinates(ks, nx, p0):
    m = workloads.random_stable(nx, {8: 4, 32: 8}[nx], np.random.default_rng(nx), q=0.1)
    m.P0 = p0 * np.eye(nx)
    _, y = workloads.simulate(m, 500, np.random.default_rng(7))
    out, _ = run(ks, m, y)
    ref = oracle.kf_rts(m, y)
    assert parity.cov_err(out[1], ref[1]) < 16 * p0 * 2.0 ** -23
    assert parity.cov_err(out[3], ref[3]) < 64 * p0 * 2.0 ** -23
