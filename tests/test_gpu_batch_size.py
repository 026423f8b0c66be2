"""An item's POD does not depend on how many items share the call: wave mode and requests that
are run together give the bits of the single launch (for a fixed group_ctas)."""
import numpy as np
import pytest

import pr_inputs as pi
from test_gpu_gram_tc import _columns
from test_gpu_waves import _iterates

pytestmark = pytest.mark.gpu


def same_alone_and_together(fn, Wt):
    """fn on all items, and on each of the first and last alone and the first two together."""
    whole = fn(Wt)
    B = Wt.shape[0]
    for lo, hi in [(0, 1), (0, 2), (B - 1, B)]:
        part = fn(Wt[lo:hi].contiguous())
        for x, y in zip(whole, part):
            assert np.array_equal(x[lo:hi], y), (lo, hi)


# chunks of one share and of three, ragged ones, several groups of rows a CTA and one
@pytest.mark.parametrize("n,K,B", [(64, 16, 5), (45, 40, 6), (41, 3, 9), (37, 33, 4), (64, 60, 3)])
def test_double_float_gram(gpu, n, K, B):
    bd, torch = gpu
    w = pi.Workload("gram", n, pi.Flow("abc"), 0.05, 1.0, B, 1e-3, n_snap=64, m_cap=32)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    Wt = torch.from_numpy(np.ascontiguousarray(_columns(n, K, B, seed=n * K))).to("cuda")
    same_alone_and_together(lambda x: [s.op_gram(x, tensor=False, df=True).cpu().numpy()], Wt)
    s.close()


# contexts of one or two items, whose chunks are shared by clusters
@pytest.mark.parametrize("n,K,B", [(41, 3, 1), (47, 17, 2), (45, 33, 1), (64, 16, 1), (41, 60, 1)])
def test_double_float_gram_in_clusters(gpu, n, K, B):
    bd, torch = gpu
    w = pi.Workload("gram", n, pi.Flow("abc"), 0.05, 1.0, B, 1e-3, n_snap=64, m_cap=32)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    Wt = torch.from_numpy(np.ascontiguousarray(_columns(n, K, B, seed=n + K))).to("cuda")
    Gd = s.op_gram(Wt, tensor=False, df=True).cpu().numpy()
    G64 = s.op_gram(Wt, tensor=False).cpu().numpy()
    s.close()
    for b in range(B):   # the bound of the double-float Gram on smaller grids
        assert np.abs(Gd[b] - G64[b]).max() < 1e-14 * np.abs(G64[b]).max()


# the wide form over units of one item to several: a single unit, ragged ones, 33 columns to 64
@pytest.mark.parametrize("n,K,B", [(9, 64, 3), (45, 64, 6), (64, 40, 5), (72, 33, 4), (37, 50, 12),
                                   (64, 54, 16)])
def test_tensor_gram(gpu, n, K, B):
    bd, torch = gpu
    w = pi.Workload("gram", n, pi.Flow("abc"), 0.05, 1.0, B, 1e-3, n_snap=64, m_cap=32)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    Wt = torch.from_numpy(np.random.default_rng(n * K).standard_normal((B, K, n ** 3))).cuda()
    same_alone_and_together(lambda x: [s.op_gram(x, tensor=True).cpu().numpy()], Wt)
    s.close()


# a middle width whose kernel is chosen by the context's points: 3 items of 45^3 are 273,375
@pytest.mark.parametrize("n,K,B", [(45, 40, 3), (40, 54, 5)])
def test_pod_of_middle_widths(gpu, n, K, B):
    bd, torch = gpu
    w = pi.Workload("mid", n, pi.Flow("abc"), 0.05, 1.0, B, 1.0 / (B * (K - 1)), n_snap=K, m_cap=16)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    Wt = torch.from_numpy(np.ascontiguousarray(_columns(n, K, B, seed=n))).cuda().reshape(B, K, n, n, n)

    def pod(x):
        R, m = s.op_pod(x, 1.0, 16)
        return [R.cpu().numpy(), m]

    same_alone_and_together(pod, Wt)
    s.close()


# the eigensolver's cluster of CTAs follows the number of matrices: 1, 2, 4 and 8 of them
@pytest.mark.parametrize("K,B", [(64, 20), (34, 40), (17, 80), (71, 30)])
def test_eigensolver(gpu, K, B):
    bd, torch = gpu
    n, cap = 6, min(K, 32)
    w = pi.Workload("eig", n, pi.Flow("abc"), 0.05, 1.0, B, 1.0 / (B * (K - 1)), n_snap=K, m_cap=cap)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP64)
    rng = np.random.default_rng(K)
    W = np.stack([(np.linalg.qr(rng.standard_normal((n ** 3, K)))[0] * np.logspace(0, -5, K)) @
                  np.linalg.qr(rng.standard_normal((K, K)))[0] for _ in range(B)])
    Wt = torch.from_numpy(np.ascontiguousarray(np.swapaxes(W, 1, 2))).cuda().reshape(B, K, n, n, n)

    def pod(x):
        R, m = s.op_pod(x, 1.0, cap)
        return [R.cpu().numpy(), m]

    same_alone_and_together(pod, Wt)
    s.close()


# waves whose last one holds one or two windows, against the single launch
@pytest.mark.parametrize("precision,n,N,ns,wave", [(1, 45, 7, 40, 3), (0, 45, 5, 12, 2), (1, 64, 5, 64, 2), (1, 64, 4, 40, 3)])
def test_wave_form(gpu, precision, n, N, ns, wave):
    bd, torch = gpu
    dt = 1e-3
    w = pi.Workload("waves", n, pi.Flow("kolmogorov", k=2), 0.02, N * (ns - 1) * dt, N, dt, n_snap=ns, m_cap=16, f_seed=3)
    s1, U1 = _iterates(bd, w, N, precision, group_ctas=9)
    m1 = s1.diagnostics()
    s1.close()
    s2, U2 = _iterates(bd, w, N, precision, group_ctas=9, wave=wave)
    m2 = s2.diagnostics()
    s2.close()
    for k in range(N + 1):
        assert np.array_equal(U1[k], U2[k]), (k, float(np.max(np.abs(U1[k] - U2[k]))))
    # the subintervals of the last iteration (older entries are an earlier iteration's)
    assert np.array_equal(m1["m1"][N - 1:], m2["m1"][N - 1:]) and np.array_equal(m1["m2"][N:], m2["m2"][N:])
