"""Tensor-core Grams of windows that hold a NaN or an infinity: NaN in that column's products, as
the FP64 and double-float kernels give, and nothing else changes."""
import numpy as np
import pytest

import pr_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 24, 32, 40, 64])   # the narrow form, the wide one
@pytest.mark.parametrize("n,value", [(4, np.nan), (32, np.inf), (32, -np.nan)])
def test_non_finite_columns(gpu, K, n, value):
    bd, torch = gpu
    B = 3
    w = pi.Workload("gram", n, pi.Flow("abc"), 0.05, 1.0, B, 1e-3, n_snap=64, m_cap=8)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    W = torch.from_numpy(np.random.default_rng(K).standard_normal((B, K, n ** 3))).cuda()
    clean = s.op_gram(W, tensor=True).cpu().numpy()
    W[1, K // 2, n ** 3 - 3] = value
    G = s.op_gram(W, tensor=True).cpu().numpy()
    ref = s.op_gram(W, tensor=False).cpu().numpy()
    s.close()
    bad = np.zeros((B, K, K), bool)
    bad[1, K // 2, :] = bad[1, :, K // 2] = True
    assert np.isnan(G[bad]).all() and np.array_equal(G[~bad], clean[~bad])
    assert not np.isfinite(ref[bad]).any() and np.isfinite(ref[~bad]).all()


def test_pod_of_a_non_finite_window(gpu):
    bd, torch = gpu
    n, K, B = 64, 40, 2
    w = pi.Workload("pod", n, pi.Flow("abc"), 0.05, 1.0, B, 1.0 / (B * (K - 1)), n_snap=K, m_cap=8)
    W = torch.from_numpy(np.random.default_rng(1).standard_normal((B, K, n, n, n))).cuda()
    m = []
    for mode in (bd.PR_GRAM_DF, bd.PR_GRAM_AUTO):
        s = bd.Parareal.from_workload(w, precision=bd.PR_FP32, gram_mode=mode)
        W[1, 3, 2, 1, 0] = float("nan")
        m.append(s.op_pod(W, 1.0, 8)[1])
        s.close()
    assert m[0][0] == 8 and m[0][1] == 0 and np.array_equal(m[0], m[1]), m
