"""Double-float Grams of one or two items, whose chunks are shared by clusters of CTAs, and the
coarse update that forms them, on grids whose chunks end raggedly."""
import numpy as np
import pytest

import oracle as O
import pr_inputs as pi
from test_gpu_gram_tc import _columns
from test_gpu_parity import dev, rel, solver

pytestmark = pytest.mark.gpu


# columns: fewer tiles than a warp, several row groups, one group a thread (64-row blocks),
# two passes over the chunk; two items: fewer CTAs a cluster
@pytest.mark.parametrize("n,K,B", [(41, 3, 1), (44, 16, 1), (47, 17, 2), (45, 33, 1), (64, 16, 1), (41, 60, 1)])
def test_double_float_gram_of_few_items(gpu, n, K, B):
    bd, torch = gpu
    w = pi.Workload("gram", n, pi.Flow("abc"), 0.05, 1.0, 4, 1e-3, n_snap=64, m_cap=32)
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    Wt = torch.from_numpy(np.ascontiguousarray(_columns(n, K, B, seed=n + K))).to("cuda")
    Gd = s.op_gram(Wt, tensor=False, df=True).cpu().numpy()
    G64 = s.op_gram(Wt, tensor=False).cpu().numpy()
    s.close()
    for b in range(B):   # the bound of the double-float Gram on smaller grids
        assert np.abs(Gd[b] - G64[b]).max() < 1e-14 * np.abs(G64[b]).max()
        assert np.array_equal(Gd[b], Gd[b].T)


@pytest.mark.parametrize("n,m", [(41, 5), (44, 16), (45, 31)])
def test_coarse_update_on_larger_grids_matches_oracle(gpu, n, m):
    bd, torch = gpu
    w = pi.Workload("cu", n, pi.Flow("kolmogorov", k=2), 0.03, 1.0, 4, 1e-3, m_cap=32, f_seed=3)
    s = solver(bd, w, precision=1)
    op = O.make_operator(w)
    rng = np.random.default_rng(m)
    R = np.linalg.qr(rng.standard_normal((w.Ng, m)))[0]
    U = pi.initial_state(n, seed=7).reshape(-1)
    Up = U + 0.05 * pi.forcing(n, seed=8).reshape(-1)
    F = pi.initial_state(n, seed=9).reshape(-1)
    out = s.op_coarse_update(dev(torch, R.T), m, dev(torch, U), dev(torch, Up), dev(torch, F)).cpu().numpy()
    V, _ = O.augment(R, U)
    g1, _ = O.coarse_propagate(op, V, U, 0.0, s.Lc, s.DeltaT / s.Lc)
    g2, _ = O.coarse_propagate(op, V, Up, 0.0, s.Lc, s.DeltaT / s.Lc)
    ref = g1 + F - g2
    s.close()
    assert rel(out, ref) < 1e-10, rel(out, ref)   # the FP32 mode's bound on smaller grids
