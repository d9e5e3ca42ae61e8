"""Likelihood rows at the ends of FP32's range (the largest accepted maximum is
3e38): scaled by powers of two, not lost."""
import numpy as np
import pytest
import torch

import workloads
from oracle import hmm as ohmm

pytestmark = pytest.mark.gpu
TOL = 1e-4      # absolute, per probability


@pytest.fixture(scope="module")
def ks():
    from paper_1905_13002_gb300 import _build
    _build.build()
    import paper_1905_13002_gb300 as ks
    return ks


@pytest.mark.parametrize("K", [2, 4, 8, 16, 32])
@pytest.mark.parametrize("peak", [1.6e38, 1.8e38, 2.9e38, 1e-37])
def test_row_maximum(ks, K, peak):
    T = 300
    seq = workloads.hmm_sequence(K, T, seed=40 + K)
    lik = seq.lik.copy()
    rows = np.arange(5, T, 37)
    lik[rows] *= (peak / lik[rows].max(axis=1))[:, None]
    lik = lik.astype(np.float32).astype(np.float64)
    model = ks.HmmModel.create(seq.pi, seq.Pi)
    filt, smooth, ll, ws = ks.hmm_smooth(model, torch.as_tensor(lik, dtype=torch.float32, device="cuda"))
    assert ks.status(ws) == ks.KS_OK
    rf, rs, rll = ohmm.forward_backward(seq.pi, seq.Pi, lik)
    assert np.abs(filt.cpu().numpy() - rf).max() < TOL and np.abs(smooth.cpu().numpy() - rs).max() < TOL
    assert (np.abs(ll.cpu().numpy() - rll) / np.maximum(1.0, np.abs(rll))).max() < TOL
