"""An item's POD does not depend on how many items share the call: wave mode and requests that
are run together give the bits of the single launch (for a fixed group_ctas)."""
import numpy as np
import pytest

import pr_inputs as pi
from test_gpu_gram_tc import _columns

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
@pytest.mark.parametrize("n,K,B", [(9, 64, 3), (45, 64, 6), (64, 40, 5), (72, 33, 4)])
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
