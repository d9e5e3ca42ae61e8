"""GPU parity of the settled path (constant covariances after the head of a
sequence) at the edges of its head, windows and sequence ends, and of the
calls that have to leave it for the general scans."""
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


def model_of(nx, rng):
    if nx <= 6:
        m = workloads.wiener_velocity(nx // 2, dt=0.1, q=float(rng.uniform(0.5, 2)), r=float(rng.uniform(0.1, 1)))
    else:
        m = workloads.random_stable(nx, {8: 4, 32: 8}[nx], rng)
    m.u = workloads._f32(0.01 * rng.standard_normal(nx))
    m.d = workloads._f32(rng.standard_normal(m.ny))
    return m


def call(ks, m, y, **kw):
    model = ks.Model.create(m.F, m.Q, m.H, m.R, m.m0, m.P0, u=m.u, d=m.d, device="cuda")
    yt = torch.as_tensor(np.asarray(y), dtype=torch.float32, device="cuda")
    purpose = ks.KS_WS_SMOOTH if kw.get("keep_filtered", True) else ks.KS_WS_ELEMENTS
    ws = ks.alloc_workspace(model, yt.shape[0], purpose)
    out = ks.smooth(model, yt, ws, **kw)
    torch.cuda.synchronize()
    return out, ws, int(ws[:64].view(torch.int32)[GENERAL])


# 128: the head's rows; 2176 = 128 + a window; 1536: an inner window's own rows
@pytest.mark.parametrize("nx", [2, 4, 6, 8])
@pytest.mark.parametrize("T", [1, 2, 127, 128, 129, 144, 255, 256, 257, 1000, 2175, 2176, 2177, 3712, 3713, 5300])
def test_edges(ks, nx, T):
    rng = np.random.default_rng(7000 + 10 * T + nx)
    m = model_of(nx, rng)
    _, y = workloads.simulate(m, T, rng)
    out, ws, general = call(ks, m, y)
    assert ks.status(ws) == ks.KS_OK and general == 0
    ref = oracle.kf_rts(m, np.asarray(y, dtype=np.float64))
    parity.check_all(out, ref)
    f, ws, general = call(ks, m, y, filter_only=True)
    assert general == 0 and f[2] is None
    assert torch.equal(f[0], out[0]) and torch.equal(f[1], out[1])
    s, ws, general = call(ks, m, y, keep_filtered=False)
    assert general == 0 and s[0] is None
    assert torch.equal(s[2], out[2]) and torch.equal(s[3], out[3])


def scans(ks, m, y):
    """The same call through the general scans: a workspace with look-back
    wait settings never takes the settled path."""
    model = ks.Model.create(m.F, m.Q, m.H, m.R, m.m0, m.P0, u=m.u, d=m.d, device="cuda")
    yt = torch.as_tensor(np.asarray(y), dtype=torch.float32, device="cuda")
    ws = ks.alloc_workspace(model, yt.shape[0])
    ks.set_waits(ws, wait_polls=1000000)
    out = ks.smooth(model, yt, ws)
    torch.cuda.synchronize()
    assert int(ws[:64].view(torch.int32)[GENERAL]) == 1
    return out, ws


# a process noise too small to settle in 128 steps, and a prior far too wide:
# the call gives what the scans give (to the rounding of their tiles' grouping)
@pytest.mark.parametrize("nx,q,p0", [(2, 1e-6, 1.0), (4, 1e-6, 1.0), (6, 1e-5, 1.0), (4, 1.0, 1e7)])
def test_unsettled_models_take_the_scans(ks, nx, q, p0):
    rng = np.random.default_rng(40 + nx)
    m = workloads.wiener_velocity(nx // 2, dt=0.1, q=q, r=1.0, P0=p0 * np.eye(nx))
    _, y = workloads.simulate(workloads.wiener_velocity(nx // 2, dt=0.1, q=q, r=1.0), 3000, rng)
    out, ws, general = call(ks, m, y)
    assert ks.status(ws) == ks.KS_OK and general == 1
    ref, _ = scans(ks, m, y)
    for a, b in zip(out, ref):
        assert torch.allclose(a, b, rtol=1e-5, atol=1e-5 * float(b.abs().max()))


# one sequence of a batch that does not settle takes the whole batch to the scans
@pytest.mark.parametrize("nx", [4, 8])
def test_unsettled_sequence_in_a_batch(ks, nx):
    rng = np.random.default_rng(60 + nx)
    ms = [model_of(nx, rng) for _ in range(5)]
    if nx == 4:
        ms[2] = workloads.wiener_velocity(2, q=1e-6, r=1.0)
    else:
        ms[2] = workloads.random_stable(8, 4, rng, q=1e-7)
    lengths = [300, 1, 900, 2500, 128]
    ys = [workloads.simulate(m, T, rng)[1] for m, T in zip(ms, lengths)]
    batch = ks.ModelBatch.create(ms, lengths)
    y = torch.as_tensor(np.concatenate(ys), dtype=torch.float32, device="cuda")
    ws = torch.zeros(ks.workspace_bytes_batch(nx, nx // 2, 5, int(y.shape[0])), dtype=torch.uint8, device="cuda")
    out = [t.cpu().numpy() for t in ks.smooth_batch(batch, y, ws)]
    assert int(ws[:64].view(torch.int32)[GENERAL]) == 1 and ks.status(ws) == ks.KS_OK
    o = 0
    for m, T, yy in zip(ms, lengths, ys):
        parity.check_all([x[o:o + T] for x in out], oracle.kf_rts(m, yy))
        o += T


@pytest.mark.parametrize("nx", [2, 4, 6, 8])
@pytest.mark.parametrize("value", [np.nan, np.inf, 3e38])
@pytest.mark.parametrize("at", [0, 100, 1500, 6999])
def test_non_finite_measurement_takes_the_scans(ks, nx, value, at):
    """As through the scans alone: the same status, the same elements finite."""
    rng = np.random.default_rng(80 + nx)
    m = workloads.wiener_velocity(nx // 2, q=1.0, r=0.5) if nx <= 6 else workloads.random_stable(8, 4, rng)
    _, y = workloads.simulate(m, 7000, rng)
    y = y.copy()
    y[at, 0] = value
    out, ws, general = call(ks, m, y)
    ref, wr = scans(ks, m, y)
    assert ks.status(ws) == ks.status(wr)
    assert all(torch.equal(torch.isfinite(a), torch.isfinite(b)) for a, b in zip(out, ref))
    if value != 3e38:
        assert general == 1


# nx = 32 takes the settled path from 256 rows on: edges of its chunks of 32,
# of the eight chunks behind a chunk, and of a block's eight chunks
@pytest.mark.parametrize("T", [256, 257, 383, 384, 385, 416, 767, 768, 769, 799, 800, 801, 1153, 2000, 5000])
def test_edges_nx32(ks, T):
    rng = np.random.default_rng(9000 + T)
    m = model_of(32, rng)
    _, y = workloads.simulate(m, T, rng)
    out, ws, general = call(ks, m, y)
    assert ks.status(ws) == ks.KS_OK and general == 0
    parity.check_all(out, oracle.kf_rts(m, np.asarray(y, dtype=np.float64)), parity.TOL_NX32)
    f, ws, general = call(ks, m, y, filter_only=True)
    assert general == 0 and torch.equal(f[0], out[0]) and torch.equal(f[1], out[1])
    s, ws, general = call(ks, m, y, keep_filtered=False)
    assert general == 0 and torch.equal(s[2], out[2]) and torch.equal(s[3], out[3])


@pytest.mark.parametrize("at", [0, 100, 1500, 2999])
def test_nx32_leaves_for_the_scans(ks, at):
    rng = np.random.default_rng(95)
    m = workloads.random_stable(32, 8, rng)
    _, y = workloads.simulate(m, 3000, rng)
    y = y.copy()
    y[at, 0] = np.nan
    out, ws, general = call(ks, m, y)
    ref, wr = scans(ks, m, y)
    assert general == 1 and ks.status(ws) == ks.status(wr)
    assert all(torch.equal(torch.isfinite(a), torch.isfinite(b)) for a, b in zip(out, ref))
    slow = workloads.random_stable(32, 8, rng, q=1e-8)      # does not settle
    _, y = workloads.simulate(slow, 3000, rng)
    out, ws, general = call(ks, slow, y)
    ref, wr = scans(ks, slow, y)
    assert general == 1
    for a, b in zip(out, ref):
        assert torch.allclose(a, b, rtol=1e-4, atol=1e-5 * float(b.abs().max()))


def test_unaligned_outputs_nx8(ks):
    """nx = 8 takes any 4-byte aligned posterior buffer (the settled path's row
    copies need 16 bytes, so these go through the scans)."""
    rng = np.random.default_rng(90)
    m = workloads.random_stable(8, 4, rng)
    _, y = workloads.simulate(m, 1000, rng)

    def buf(*s):
        n = int(np.prod(s))
        return torch.empty(n + 1, dtype=torch.float32, device="cuda")[1:].view(*s)

    out, ws, general = call(ks, m, y, fmean=buf(1000, 8), fcov=buf(1000, 8, 8), smean=buf(1000, 8),
                            scov=buf(1000, 8, 8))
    assert ks.status(ws) == ks.KS_OK
    parity.check_all(out, oracle.kf_rts(m, np.asarray(y, dtype=np.float64)))
