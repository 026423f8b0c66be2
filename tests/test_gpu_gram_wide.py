"""The tensor-core Gram of 33 to 64 columns over its units, accumulation windows and stages:
ragged ends, columns on 8-byte boundaries, several windows a unit, several waves of units."""
import numpy as np
import pytest

import pr_inputs as pi
from test_gpu_gram_tc import _exact_dot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K,B", [
    (4, 40, 1),     # 64 points: one stage
    (9, 33, 2),     # 729 points (odd): odd columns only 8-byte aligned, a 25-point tail
    (11, 64, 4),    # 1,331 points, all columns
    (40, 57, 3),    # several units a CTA, chunks of 640 points
    (72, 64, 5),    # 373,248 points: units of four windows, the last one ragged
])
def test_wide_tensor_gram(gpu, n, K, B):
    bd, torch = gpu
    w = pi.Workload("gram", n, pi.Flow("abc"), 0.05, 1.0, 5, 1e-3, n_snap=64, m_cap=32)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    rng = np.random.default_rng(n * K)
    Ng = n ** 3
    # columns of scales 1e-12 .. 1e12, some nearly parallel
    W = rng.standard_normal((B, K, Ng)) * 10.0 ** rng.integers(-12, 13, (B, K, 1))
    W[:, 1] = W[:, 0] * (1.0 + 1e-7 * rng.standard_normal(Ng))
    G = s.op_gram(torch.from_numpy(W).cuda(), tensor=True).cpu().numpy()
    s.close()
    assert np.array_equal(G, np.swapaxes(G, 1, 2))
    for b in {0, B - 1}:
        for i, j in [(0, 0), (0, 1), (1, K - 1), (K // 2, K // 2), (7, 31), (K - 1, K - 1)]:
            x, y = W[b, i], W[b, j]
            # the values are cut at 2^-54 of their column's largest, dropped digit pairs weigh
            # below 2^-57 of the product of the two largest; the sums are exact, a chunk and the
            # item round once each
            ref, mx = _exact_dot(x, y), np.abs(x).max() * np.abs(y).max()
            cut = 2.0 ** -53 * (np.abs(x).sum() * np.abs(y).max() + np.abs(y).sum() * np.abs(x).max())
            tol = cut + 8 * 2.0 ** -57 * Ng * mx + 128 * 2.0 ** -53 * np.abs(x * y).sum()
            assert abs(G[b, i, j] - ref) <= tol, (b, i, j, G[b, i, j], ref, tol)


# 33 to 54 columns: the tensor cores from 262,144 points in all, double-float below and where
# waits may not last
@pytest.mark.parametrize("n,B,K,opts", [(64, 1, 33, {}), (63, 1, 40, {}), (63, 2, 40, {}), (64, 1, 54, {"spin_limit": 0}),
                                        (64, 1, 54, {"spin_limit": 4096})])
def test_pod_of_middle_widths(gpu, n, B, K, opts):
    bd, torch = gpu
    w = pi.Workload("mid", n, pi.Flow("abc"), 0.05, 1.0, B, 1.0 / (B * (K - 1)), n_snap=K, m_cap=16)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32, **opts)
    sig = np.logspace(0.0, -1.0, K)
    gap = float(np.min(-np.diff(sig ** 2)))
    tol = 16.0 * K * 3.6e-15 / gap + 1e-12   # double-float accuracy over the eigenvalues' gap
    rng = np.random.default_rng(n + K)
    Q = [np.linalg.qr(rng.standard_normal((n ** 3, K)))[0] for _ in range(B)]
    Y = np.linalg.qr(rng.standard_normal((K, K)))[0]
    W = np.ascontiguousarray(np.stack([((q * sig) @ Y.T).T for q in Q]))
    R, m = s.op_pod(torch.from_numpy(W).cuda().reshape(B, K, n, n, n), 1.0, 16)
    R = R.cpu().numpy().reshape(B, -1, n ** 3)
    s.close()
    for b in range(B):
        assert m[b] == 16
        assert np.abs(np.abs(R[b] @ Q[b][:, :16]) - np.eye(16)).max() < tol, b
