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
