"""Absorbing states that are never measured: a short sequence is one chain that
starts from p(x_1), so that states which cannot give the measurements do not
fail it, whatever the lane groups beside it fold."""
import numpy as np
import pytest
import torch

from oracle import hmm as ohmm

pytestmark = pytest.mark.gpu
TOL = 1e-4      # absolute, per probability


@pytest.fixture(scope="module")
def ks():
    from paper_1905_13002_gb300 import _build
    _build.build()
    import paper_1905_13002_gb300 as ks
    return ks


@pytest.mark.parametrize("K,T", [(8, 1), (8, 4), (8, 32), (16, 1), (16, 20), (16, 33), (16, 64), (32, 2), (32, 33),
                                 (32, 64)])
def test_one_chain(ks, K, T):
    rng = np.random.default_rng(K + T)
    Pi = rng.dirichlet(np.ones(K), size=K)
    Pi[-2:] = np.eye(K)[-2:]                             # two absorbing states
    Pi = Pi.astype(np.float32).astype(np.float64)
    pi = np.full(K, 1.0 / K)
    lik = rng.uniform(0.1, 1.0, size=(T, K)).astype(np.float32).astype(np.float64)
    lik[:, -2:] = 0.0                                    # that give none of the measurements
    model = ks.HmmModel.create(pi, Pi)
    t = torch.as_tensor(lik, dtype=torch.float32, device="cuda")
    filt, smooth, ll, ws = ks.hmm_smooth(model, t)
    assert ks.status(ws) == ks.KS_OK
    rf, rs, rll = ohmm.forward_backward(pi, Pi, lik)
    assert np.abs(filt.cpu().numpy() - rf).max() < TOL and np.abs(smooth.cpu().numpy() - rs).max() < TOL
    assert (np.abs(ll.cpu().numpy() - rll) / np.maximum(1.0, np.abs(rll))).max() < TOL
