"""The POD's batched eigensolver: windows with a known singular value decomposition, over the
cluster sizes (few and many windows) and the matrix sizes where its slots split unevenly."""
import numpy as np
import pytest

import pr_inputs as pi

pytestmark = pytest.mark.gpu


# B windows of K columns: one slot, an odd player, fewer slots than CTAs, slots over several
# CTAs unevenly, a warp of angles and more, the largest window; B from 1 to more than the SMs
@pytest.mark.parametrize("B,K", [(1, 1), (2, 2), (1, 3), (2, 5), (1, 16), (3, 31), (1, 33), (4, 64), (20, 34), (30, 37),
                                 (40, 24), (80, 17), (160, 8), (2, 71), (1, 96)])
def test_pod_of_windows_with_known_svd(gpu, B, K):
    bd, torch = gpu
    n, rng, cap = 6, np.random.default_rng(B * 1000 + K), min(K, 32)
    w = pi.Workload("eig", n, pi.Flow("abc"), 0.05, 1.0, B, 1.0 / (B * max(1, K - 1)), n_snap=max(2, K), m_cap=cap)
    s = bd.Parareal.from_workload(w, precision=0)
    sig = np.logspace(0.0, -1.0, K) if K > 1 else np.ones(1)
    lam = sig ** 2
    gap = float(np.min(-np.diff(lam))) if K > 1 else 1.0
    # eigenvectors of a symmetric matrix known to a few K eps ||A|| (the Jacobi sweeps' end and
    # the Gram's own rounding), divided by the gap to the next eigenvalue
    tol = 16.0 * K * 2.22e-16 / gap + 1e-13
    Q, W = [], []
    for b in range(B):
        q, _ = np.linalg.qr(rng.standard_normal((n ** 3, K)))
        y, _ = np.linalg.qr(rng.standard_normal((K, K)))
        Q.append(q)
        W.append(((q * sig) @ y.T).T)
    Wt = torch.from_numpy(np.ascontiguousarray(np.stack(W) * 2.0 ** -300)).cuda().reshape(B, K, n, n, n)   # any scale
    R, m = s.op_pod(Wt, 1.0, cap)
    R = R.cpu().numpy().reshape(B, -1, n ** 3)
    s.close()
    for b in range(B):
        assert m[b] == cap
        G = R[b, :cap] @ Q[b][:, :cap]
        assert np.abs(np.abs(np.diag(G)) - 1.0).max() < tol, b
        assert np.abs(G - np.diag(np.diag(G))).max() < tol, b
