"""Discrete-state prefixes over a long, static chain: the differences of
log g between states have to survive prefixes whose log g itself is -1e5 and
beyond."""
import numpy as np
import pytest
import torch

from oracle import hmm as ohmm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ks():
    from paper_1905_13002_gb300 import _build
    _build.build()
    import paper_1905_13002_gb300 as ks
    return ks


@pytest.mark.parametrize("K,T", [(8, 1 << 20), (16, 1 << 18), (32, 1 << 18)])
def test_static(ks, K, T):
    """A chain that never moves (its products with Pi are exact), states of near-equal
    evidence, undecided throughout.  What is left rounds each step's
    weights by about three eps32, by amounts that the random evidence makes
    independent: 4 sqrt(3 T) eps32 in the log odds, a quarter of it in a marginal."""
    rng = np.random.default_rng(K)
    Pi = np.eye(K)
    pi = np.full(K, 1.0 / K)
    odds = rng.standard_normal((T, K))
    odds -= odds.mean(axis=0)
    lik = 0.5 * np.exp(odds / np.sqrt(T))
    lik = lik.astype(np.float32).astype(np.float64)
    model = ks.HmmModel.create(pi, Pi)
    filt, smooth, ll, ws = ks.hmm_smooth(model, torch.as_tensor(lik, dtype=torch.float32, device="cuda"))
    assert ks.status(ws) == ks.KS_OK
    rf, rs, rll = ohmm.forward_backward(pi.astype(np.float32), Pi, lik)
    tol = np.sqrt(3.0 * T) * np.finfo(np.float32).eps
    assert 0.3 / K < rf[-1].min() and rf[-1].max() < 3.0 / K
    assert np.abs(filt.cpu().numpy() - rf).max() < tol
    assert np.abs(smooth.cpu().numpy() - rs).max() < tol
    assert (np.abs(ll.cpu().numpy() - rll) / np.maximum(1.0, np.abs(rll))).max() < 1e-6
