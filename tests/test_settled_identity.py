"""The closed forms of the settled path against the oracle, in FP64: the fixed
point by doubling Lemma 4, the covariances of the head and of a sequence's end
from the tables Phi^n and O_n, and the means' adjoint form."""
import numpy as np
import pytest

import oracle
import workloads


def settled(m, n_double=10):
    F, Q, H, R = m.F, m.Q, m.H, m.R
    S = H @ Q @ H.T + R
    K = Q @ H.T @ np.linalg.inv(S)
    A, C, J = F - K @ H @ F, Q - K @ S @ K.T, F.T @ H.T @ np.linalg.inv(S) @ H @ F
    for _ in range(n_double):
        Mi = np.linalg.inv(np.eye(m.nx) + C @ J)
        A, C, J = A @ Mi @ A, A @ Mi @ C @ A.T + C, A.T @ Mi.T @ J @ A + J
    P = C
    Pm = F @ P @ F.T + Q
    S = H @ Pm @ H.T + R
    K = Pm @ H.T @ np.linalg.inv(S)
    return P, K, F - K @ H @ F, F.T @ H.T @ np.linalg.inv(S)


def model(kind, seed):
    rng = np.random.default_rng(seed)
    if kind == "wiener4":
        return workloads.wiener_velocity(2, q=1.3, r=0.4, P0=3.0 * np.eye(4)), rng
    if kind == "wiener2":
        return workloads.wiener_velocity(1, q=0.6, r=0.9), rng
    return workloads.random_stable(8, 4, rng), rng


@pytest.mark.parametrize("kind", ["wiener2", "wiener4", "stable8"])
@pytest.mark.parametrize("T", [3, 100, 200, 400])
def test_closed_forms(kind, T):
    m, rng = model(kind, 5)
    _, y = workloads.simulate(m, T, rng)
    fm, fP, sm, sP = oracle.kf_rts(m, y)
    P, K, Phi, B = settled(m)
    n = m.nx
    pw, O = [np.eye(n)], [np.zeros((n, n))]
    for _ in range(T):
        O.append(O[-1] + pw[-1].T @ (B @ m.H @ m.F) @ pw[-1])
        pw.append(Phi @ pw[-1])
    for h, k in [(1, 1), (2, 1), (64, 30)]:           # the doubling of the tables
        if h + k <= T:
            assert np.allclose(O[h + k], O[h] + pw[h].T @ O[k] @ pw[h], rtol=1e-9, atol=1e-12)
    D0 = fP[0] - P
    for k in range(T):
        D = pw[k] @ np.linalg.inv(np.eye(n) + D0 @ O[k]) @ D0 @ pw[k].T
        assert np.allclose(P + D, fP[k], rtol=1e-8, atol=1e-10), k
        Pk = P + D
        later = O[T - 1 - k]
        assert np.allclose(Pk - Pk @ np.linalg.inv(np.eye(n) + later @ D) @ later @ Pk, sP[k], rtol=1e-7, atol=1e-9), k
    # means: s_k = m_k + P_k l_k, l_k = Phi_{k+1}^T l_{k+1} + F^T H^T S_{k+1}^-1 e_{k+1}
    lam = np.zeros(n)
    for k in range(T - 2, -1, -1):
        Pm = m.F @ fP[k] @ m.F.T + m.Q
        Si = np.linalg.inv(m.H @ Pm @ m.H.T + m.R)
        e = y[k + 1] - m.d - m.H @ (m.F @ fm[k] + m.u)
        Kk = Pm @ m.H.T @ Si
        lam = (m.F - Kk @ m.H @ m.F).T @ lam + m.F.T @ m.H.T @ Si @ e
        assert np.allclose(fm[k] + fP[k] @ lam, sm[k], rtol=1e-7, atol=1e-7), k
