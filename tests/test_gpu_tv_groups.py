"""GPU: time-varying nx = 8 where a chain (8 steps), a tile (4 chains) or the
spine's first levels end; the constants and measurements of the next step are
staged while a step is combined, so the last step of each has none to stage."""
import numpy as np
import pytest
import torch

import workloads
from test_gpu_tv import check, ks  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [2, 7, 8, 9, 31, 32, 33, 40, 64, 97, 1025])
def test_chain_and_tile_edges(ks, T):  # noqa: F811
    check(ks, workloads.random_time_varying(8, 4, T, np.random.default_rng(8100 + T)))


@pytest.mark.parametrize("T", [9, 70])
def test_measurements_at_any_word(ks, T):  # noqa: F811
    """y needs no more than its own 4-byte alignment: bit for bit the same."""
    seq = workloads.random_time_varying(8, 4, T, np.random.default_rng(8200 + T))
    m = seq.model
    model = ks.Model.create(m.F, m.Q, m.H, m.R, m.m0, m.P0, u=m.u, d=m.d, device="cuda")
    y = torch.as_tensor(seq.y, dtype=torch.float32, device="cuda").contiguous()
    flat = torch.zeros(y.numel() + 1, device="cuda")
    flat[1:] = y.flatten()
    for a, b in zip(ks.smooth(model, y), ks.smooth(model, flat[1:].view(T, -1))):
        assert torch.equal(a, b)
