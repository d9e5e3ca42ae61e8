"""Discrete-state calls either side of the lengths at which the chains become
longer, against the FP64 oracle."""
import numpy as np
import pytest
import torch

import workloads
from oracle import hmm as ohmm

pytestmark = pytest.mark.gpu
TOL = 1e-4      # absolute, per probability; the log-likelihood relative


@pytest.mark.parametrize("K,T", [(8, 786431), (8, 786433), (16, 262143), (16, 262145), (32, 81919), (32, 81921)])
def test_line(K, T):
    import paper_1905_13002_gb300 as ks
    seq = workloads.hmm_sequence(K, T, seed=T)
    model = ks.HmmModel.create(seq.pi, seq.Pi)
    filt, smooth, ll, ws = ks.hmm_smooth(model, torch.as_tensor(seq.lik, dtype=torch.float32, device="cuda"))
    assert ks.status(ws) == ks.KS_OK
    rf, rs, rll = ohmm.forward_backward(seq.pi, seq.Pi, seq.lik)
    assert np.abs(filt.cpu().numpy() - rf).max() < TOL and np.abs(smooth.cpu().numpy() - rs).max() < TOL
    assert (np.abs(ll.cpu().numpy() - rll) / np.maximum(1.0, np.abs(rll))).max() < TOL
