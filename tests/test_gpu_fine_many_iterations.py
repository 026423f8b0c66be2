"""FP64 fine steps that take many BiCGStab iterations (a large step against the advection time
of a cell): they converge, in about the oracle's number of iterations, to its states."""
import numpy as np
import pytest

import oracle as O
import pr_inputs as pi

pytestmark = pytest.mark.gpu


# on chip: the smallest grids, an even and an odd one, the largest; from 36 on the streaming
# kernel (two points a thread, and one).  10 to 40 iterations a step; a small state beside the
# forcing starts far from its solution
@pytest.mark.parametrize("n,flow,eps,dt,scale", [
    (8, "abc", 0.05, 0.1, 1e-3), (16, "abc", 0.002, 0.1, 1.0), (24, "abc", 0.2, 0.1, 1e-3), (24, "kolmogorov", 0.2, 0.1, 1.0),
    (33, "abc", 0.01, 0.03, 1.0), (36, "abc", 0.05, 0.1, 1.0), (45, "abc", 0.01, 0.03, 1e-3), (48, "abc", 0.002, 0.03, 1.0)])
def test_many_iterations_converge_to_the_oracle(gpu, n, flow, eps, dt, scale):
    bd, torch = gpu
    B, steps = 2, 5
    w = pi.Workload("many", n, pi.Flow(flow, k=2), eps, B * 10 * dt, B, dt, n_snap=0, m_cap=4, f_seed=3)
    u = np.stack([scale * pi.initial_state(n, seed=3 + b) for b in range(B)])
    s = bd.Parareal.from_workload(w, precision=0)
    s.set_initial(u[0], w.f())
    out, _ = s.op_fine(torch.from_numpy(u).cuda(), steps)
    out = out.cpu().numpy()
    total, most = s.lin_stats()
    s.close()
    op = O.make_operator(w)
    for b in range(B):
        its = []
        ue, _ = O.fine_propagate(op, u[b], 0.0, steps, dt, tol=1e-14, stats=its)
        # L is positive semidefinite, so a step adds at most the two residuals of 1e-14 of its
        # right-hand side; the rounding of dt L u (dt ||L|| up to 10) is below 1e-13 over the steps
        assert np.linalg.norm(out[b] - ue) < 1e-12 * np.linalg.norm(ue)
        # BiCGStab's path responds to rounding: the counts agree to about a tenth
        assert 0.7 * sum(its) - steps <= total[b] <= 1.3 * sum(its) + steps, (total[b], its)
        assert most[b] <= 1.5 * max(its) + 3
