"""GPU parity of short sequences (at most 128 steps, a settled path's head)
whose model has not settled within them: alone, in a batch and in a mixed
batch.  The head's closed forms hold around the Riccati fixed point only."""
import numpy as np
import pytest
import torch

import oracle
import parity
import workloads

pytestmark = pytest.mark.gpu
GENERAL = 5      # header word: the general scans ran

SLOW = [dict(q=1.0, r=1.0, dt=0.01), dict(q=1e-4, r=1.0, dt=0.1), dict(q=1e-3, r=10.0, dt=0.1),
        dict(q=1e-3, r=10.0, dt=0.1, p0=0.01)]


@pytest.fixture(scope="module")
def ks():
    from paper_1905_13002_gb300 import _build
    _build.build()
    import paper_1905_13002_gb300 as ks
    return ks


def slow_model(nx, kind):
    if nx == 8:
        return workloads.random_stable(8, 4, np.random.default_rng(11), q=1e-4, lo=0.98, hi=0.998)
    kw = dict(SLOW[kind])
    return workloads.wiener_velocity(nx // 2, P0=kw.pop("p0", 1.0) * np.eye(nx), **kw)


@pytest.mark.parametrize("T", [2, 64, 100, 127, 128])
@pytest.mark.parametrize("nx,kind", [(2, 0), (2, 1), (2, 2), (2, 3), (4, 0), (4, 3), (6, 1), (6, 3), (8, 0)])
def test_alone(ks, nx, kind, T):
    m = slow_model(nx, kind)
    _, y = workloads.simulate(m, T, np.random.default_rng(300 + T))
    model = ks.Model.create(m.F, m.Q, m.H, m.R, m.m0, m.P0, device="cuda")
    yt = torch.as_tensor(y, dtype=torch.float32, device="cuda")
    ws = ks.alloc_workspace(model, T)
    out = ks.smooth(model, yt, ws)
    assert ks.status(ws) == ks.KS_OK and int(ws[:64].view(torch.int32)[GENERAL]) == 1
    parity.check_all(out, oracle.kf_rts(m, y))


def settled_model(nx, rng):
    return workloads.wiener_velocity(nx // 2, q=1.0, r=0.3) if nx <= 6 else workloads.random_stable(8, 4, rng)


def group(nx, kind, rng):
    ms = [settled_model(nx, rng), slow_model(nx, kind), settled_model(nx, rng), slow_model(nx, kind)]
    lengths = [300, 100, 64, 128]
    return ms, lengths, [workloads.simulate(m, T, rng)[1] for m, T in zip(ms, lengths)]


def check_group(out, ms, lengths, ys):
    o = 0
    for m, T, y in zip(ms, lengths, ys):
        parity.check_all([x[o:o + T].cpu().numpy() for x in out], oracle.kf_rts(m, y))
        o += T


@pytest.mark.parametrize("nx,kind", [(2, 3), (4, 0), (6, 2), (8, 0)])
def test_in_a_batch(ks, nx, kind):
    ms, lengths, ys = group(nx, kind, np.random.default_rng(400 + nx))
    y = torch.as_tensor(np.concatenate(ys), dtype=torch.float32, device="cuda")
    out = ks.smooth_batch(ks.ModelBatch.create(ms, lengths), y)
    check_group(out, ms, lengths, ys)


def test_in_a_mixed_batch(ks):
    gs = [group(nx, kind, np.random.default_rng(500 + nx)) for nx, kind in [(2, 1), (4, 3), (6, 0)]]
    call = [(ks.ModelBatch.create(ms, lengths), torch.as_tensor(np.concatenate(ys), dtype=torch.float32, device="cuda"))
            for ms, lengths, ys in gs]
    for (ms, lengths, ys), out in zip(gs, ks.smooth_batched(call)):
        check_group(out, ms, lengths, ys)
