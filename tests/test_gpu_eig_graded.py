"""POD of windows whose singular values fall evenly to the rank cut and beyond it."""
import numpy as np
import pytest

import pr_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("K", [24, 33, 64])
def test_pod_down_to_the_rank_cut(gpu, prec, K):
    bd, torch = gpu
    n, B, tau = 8, 3, 1e-13   # the level-1 cut on the eigenvalues
    w = pi.Workload("graded", n, pi.Flow("abc"), 0.05, 1.0, B, 1.0 / (B * (K - 1)), n_snap=K, m_cap=min(K, 32))
    lam = 10.0 ** -np.linspace(0.0, 16.0, K)
    lam = np.where(abs(np.log10(lam / tau)) < 0.15, lam * 2.0, lam)   # none at the cut itself
    rank = int(np.sum(lam > tau))
    rng = np.random.default_rng(K)
    W = np.stack([(np.linalg.qr(rng.standard_normal((n ** 3, K)))[0] * np.sqrt(lam)) @
                  np.linalg.qr(rng.standard_normal((K, K)))[0].T for _ in range(B)])
    s = bd.Parareal.from_workload(w, precision=prec)
    Wt = torch.from_numpy(np.ascontiguousarray(np.swapaxes(W, 1, 2))).cuda().reshape(B, K, n, n, n)
    R, m = s.op_pod(Wt, 1.0, min(K, 32))
    R = R.cpu().numpy().reshape(B, -1, n ** 3)
    s.close()
    # the Gram's and the sweeps' rounding on every eigenvalue, at the size of the largest
    noise = 4 * K * (2.2e-16 if prec == 0 else 3.6e-15)
    for b in range(B):
        if lam[rank - 1] - noise > tau > lam[rank] + noise:
            assert m[b] == min(rank, 32)
        V = R[b, : m[b]]
        assert np.abs(V @ V.T - np.eye(m[b])).max() < 1e-12
        # what the basis leaves of the window: the values it cut, and the rounding of those it kept
        left = W[b] - V.T @ (V @ W[b])
        assert np.linalg.norm(left) ** 2 <= lam[m[b]:].sum() + (K + 4) * noise
