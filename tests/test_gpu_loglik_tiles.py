"""GPU: ks_loglik where a block's tile of 32 or 128 steps ends (nx = 8, 32: lanes
of a group form a step's S, one thread takes its density in FP64)."""
import numpy as np
import pytest
import torch

from test_gpu_loglik import gpu_model, ks, make  # noqa: F401

pytestmark = pytest.mark.gpu


def density(m, y, fm, fc):
    """log p(y_k | y_1:k-1) in FP64 from the given filtered moments."""
    f = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)
    F, Q, H, R, u, d = f(m.F), f(m.Q), f(m.H), f(m.R), f(m.u), f(m.d)
    m0, P0 = np.asarray(m.m0, float), np.asarray(m.P0, float)
    mean = np.concatenate([m0[None], fm[:-1]]) @ F.T + u
    P = np.concatenate([P0[None], fc[:-1]])
    S = H @ (F @ P @ F.T + Q) @ H.T + R
    e = f(y) - mean @ H.T - d
    sign, ld = np.linalg.slogdet(S)
    return -0.5 * (np.einsum("ti,ti->t", e, np.linalg.solve(S, e[..., None])[..., 0]) + ld
                   + H.shape[0] * np.log(2 * np.pi)), np.linalg.norm(H, 2) * np.linalg.norm(F, 2), S, e


@pytest.mark.parametrize("nx,ny", [(8, 4), (32, 8)])
@pytest.mark.parametrize("T", [1, 2, 31, 33, 127, 128, 129, 300])
def test_tile_edges(ks, nx, ny, T):  # noqa: F811
    """S and the residual are FP32 sums of at most 2 nx + 1 terms from FP32
    constants (another nx terms): relative errors c = 4 (nx + 1) 2^-24 of the sums
    of absolute values, which change a density by at most 1/2 (|S^-1| dS ny +
    |z|^2 |S^-1| dS) + |z| |S^-1/2| de, z = S^-1/2 e.  The FP64 tail adds
    nothing at that scale; the result is one FP32 rounding."""
    m, y = make("stable", nx, ny, T, 40 + nx + T)
    model = gpu_model(ks, m)
    yt = torch.as_tensor(y, dtype=torch.float32, device="cuda")
    fm, fc, _, _ = ks.smooth(model, yt)
    ll, total, st = ks.loglik(model, yt, fm, fc)
    assert int(st.item()) == 0
    fm, fc = fm.cpu().numpy().astype(np.float64), fc.cpu().numpy().astype(np.float64)
    ref, g, S, e = density(m, y, fm, fc)
    c = 4 * (nx + 1) * 2.0 ** -24
    ev = np.linalg.eigvalsh(S)
    si = 1 / ev[:, 0]
    P = np.concatenate([np.asarray(m.P0, float)[None], fc[:-1]])
    mean = np.concatenate([np.asarray(m.m0, float)[None], fm[:-1]])
    dS = c * (np.sqrt(nx) * g * g * np.linalg.norm(P, axis=(1, 2)) + np.linalg.norm(m.H) ** 2 * np.linalg.norm(m.Q)
              + np.linalg.norm(m.R))
    de = c * (np.sqrt(nx) * g * np.linalg.norm(mean, axis=1) + np.linalg.norm(e, axis=1)
              + np.linalg.norm(m.H) * np.linalg.norm(m.u) + np.linalg.norm(m.d) + np.linalg.norm(y, axis=1))
    z2 = np.einsum("ti,ti->t", e, e) * si
    tol = 0.5 * si * dS * (ny + z2) + np.sqrt(z2 * si) * de + 2.0 ** -23 * np.abs(ref)
    got = ll.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= tol)
    assert abs(total.item() - ref.sum()) <= tol.sum()
