"""The FP32 mode's snapshot projection over its output counts (blocks of two) and two points a
thread with a ragged end: POD of windows with a known singular value decomposition."""
import numpy as np
import pytest

import pr_inputs as pi

pytestmark = pytest.mark.gpu


# n, B: one point a thread; two points a thread (enough CTAs), odd number of points
@pytest.mark.parametrize("n,B", [(9, 2), (47, 3)])
@pytest.mark.parametrize("K", [2, 3, 5, 8, 11, 13, 16, 19, 32])
def test_projection_of_windows_with_known_svd(gpu, n, B, K):
    bd, torch = gpu
    w = pi.Workload("tsmm", n, pi.Flow("abc"), 0.05, 1.0, B, 1.0 / (B * (K - 1)), n_snap=K, m_cap=K)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    sig = np.logspace(0.0, -1.0, K)
    gap = float(np.min(-np.diff(sig ** 2)))
    # as for the eigensolver, with double-float Grams and projections (2^-48 a value)
    tol = 16.0 * K * 3.6e-15 / gap + 1e-12
    rng = np.random.default_rng(n + K)
    Q = [np.linalg.qr(rng.standard_normal((n ** 3, K)))[0] for _ in range(B)]
    Y = [np.linalg.qr(rng.standard_normal((K, K)))[0] for _ in range(B)]
    W = np.ascontiguousarray(np.stack([((q * sig) @ y.T).T for q, y in zip(Q, Y)]))
    R, m = s.op_pod(torch.from_numpy(W).cuda().reshape(B, K, n, n, n), 1.0, K)
    R = R.cpu().numpy().reshape(B, -1, n ** 3)
    s.close()
    for b in range(B):
        assert m[b] == K
        G = R[b, :K] @ Q[b]
        assert np.abs(np.abs(G) - np.eye(K)).max() < tol, b
