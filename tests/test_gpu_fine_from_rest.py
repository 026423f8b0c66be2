"""FP32 steps whose residual falls several hundredfold in half an iteration (a first step from
rest under a forcing, with a small dt L): the on-chip kernel stops where the streaming kernel,
which sums the residual itself, does."""
import numpy as np
import pytest

import oracle as O
import pr_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dt", [(8, 1e-5), (8, 1e-4), (16, 1e-5), (16, 1e-4), (32, 1e-5), (45, 1e-5), (45, 1e-4)])
def test_iterations_from_rest(gpu, n, dt):
    bd, torch = gpu
    B = 6
    w = pi.Workload("rest", n, pi.Flow("kolmogorov", k=2), 0.02, B * 10 * dt, B, dt, n_snap=0, m_cap=4, f_seed=3)
    u = np.stack([1e-6 * b * pi.initial_state(n, seed=3 + b) for b in range(B)])
    op = O.make_operator(w)
    counts = []
    for kw in (dict(), dict(group_ctas=1, spin_limit=0)):   # spin_limit = 0 keeps the streaming kernel
        s = bd.Parareal.from_workload(w, precision=bd.PR_FP32, **kw)
        s.set_initial(u[0], w.f())
        out, _ = s.op_fine(torch.from_numpy(u).cuda(), 1)
        out = out.cpu().numpy()
        counts.append(s.lin_stats()[0][:B])
        s.close()
        for b in (0, B - 1):
            ue, _ = O.fine_propagate(op, u[b], 0.0, 1, dt, tol=1e-14)
            # the increment is a float: three roundings of 2^-24 a point, and the residual's 1e-9
            assert np.linalg.norm(out[b] - ue) < (3 * 2.0 ** -24 + 4e-9) * np.linalg.norm(ue)
    assert np.array_equal(*counts), counts
