"""The settled path's head from a known start, far more certain than the
settled covariance: every variance keeps its own digits."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu
GENERAL = 5      # header word: the general scans ran

# The powers of the bits of k: at most seven inverses, whose Skeel condition is at
# most 10 here in 64 bits, each followed by sums of non-negative parts:
# 7 x 10 eps32 = 8e-6; at most 20 for the nx = 32 model: 7 x 20 eps32 = 1.7e-5.
# P + D_k was 5e-5 and 1e-4 off for these models.
TOL, TOL32 = 1e-5, 1.7e-5


@pytest.fixture(scope="module")
def ks():
    from paper_1905_13002_gb300 import _build
    _build.build()
    import paper_1905_13002_gb300 as ks
    return ks


def run(ks, m, y, **kw):
    model = ks.Model.create(m.F, m.Q, m.H, m.R, m.m0, m.P0, device="cuda")
    yt = torch.as_tensor(y, dtype=torch.float32, device="cuda")
    ws = ks.alloc_workspace(model, len(y))
    out = ks.smooth(model, yt, ws, **kw)
    assert ks.status(ws) == ks.KS_OK and int(ws[:64].view(torch.int32)[GENERAL]) == 0
    return [None if t is None else t.cpu().numpy() for t in out]


def entry_err(got, ref):
    """Largest error of an entry in units of its two standard deviations."""
    sd = np.sqrt(np.einsum("tii->ti", ref))
    return float((np.abs(got - ref) / (sd[:, :, None] * sd[:, None, :])).max())


def check(out, ref, tol=TOL):
    assert entry_err(out[1], ref[1]) < tol and entry_err(out[3], ref[3]) < tol
    for i in (0, 2):
        sd = np.sqrt(np.einsum("tii->ti", ref[i + 1]))
        assert (np.abs(out[i] - ref[i]) / sd).max() < 0.01


@pytest.mark.parametrize("nx", [2, 4, 6])
@pytest.mark.parametrize("p0", [0.0, 1e-8, 1e-4])
@pytest.mark.parametrize("T", [3, 128, 300, 2500])
def test_known_start(ks, nx, p0, T):
    m = workloads.wiener_velocity(nx // 2, dt=0.02, q=20.0, r=1.0, P0=p0 * np.eye(nx))
    _, y = workloads.simulate(m, T, np.random.default_rng(T + nx))
    y = y * (1.0 if T < 2000 else 0.0)      # long positions would leave FP32's resolution of an sd
    check(run(ks, m, y), oracle.kf_rts(m, y))
    f = run(ks, m, y, filter_only=True)
    assert entry_err(f[1], oracle.kf(m, y)[1]) < TOL


def tracking32():
    """Eight axes of position and velocity and sixteen damped states."""
    w = workloads.wiener_velocity(8, dt=0.03, q=40.0, r=1.0)
    F, Q = np.zeros((32, 32)), np.eye(32)
    F[:16, :16], Q[:16, :16] = w.F, w.Q
    F[16:, 16:] = 0.5 * np.eye(16)
    H = np.hstack([w.H, 0.02 * np.ones((8, 16))])
    return workloads.make_model(F, Q, H, np.eye(8), np.zeros(32), 1e-8 * np.eye(32))


@pytest.mark.parametrize("T", [256, 700])
def test_known_start_nx32(ks, T):
    m = tracking32()
    _, y = workloads.simulate(m, T, np.random.default_rng(T))
    check(run(ks, m, y), oracle.kf_rts(m, y), TOL32)


def test_known_start_nx8(ks):
    w = workloads.wiener_velocity(3, dt=0.02, q=20.0, r=1.0)
    F, Q, H = np.zeros((8, 8)), np.eye(8), np.zeros((4, 8))
    F[:6, :6], Q[:6, :6], H[:3, :6] = w.F, w.Q, w.H
    F[6:, 6:] = 0.5 * np.eye(2)
    H[3, 6:] = 1.0
    m = workloads.make_model(F, Q, H, np.eye(4), np.zeros(8), np.zeros((8, 8)))
    _, y = workloads.simulate(m, 400, np.random.default_rng(1))
    check(run(ks, m, y), oracle.kf_rts(m, y))
