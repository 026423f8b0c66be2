"""Steps of two and three iterations stay in the FP32 mode's two-pass kernel: its states are the
four-pass kernel's and its sweep is the faster one; steps of more iterations are resumed."""
import ctypes

import numpy as np
import pytest

import pr_inputs as pi
from test_gpu_fine_fused import rel, step_tol
from test_gpu_tune_kernels import best_ms

pytestmark = pytest.mark.gpu


# iterations a step: 2, 3, and more than the two-pass kernel keeps
@pytest.mark.parametrize("n,eps,dt,its", [(64, 0.05, 3e-3, 2), (64, 0.05, 1e-2, 3), (96, 0.02, 3e-3, 2), (64, 0.05, 3e-2, 5)])
def test_two_pass_keeps_steps_of_few_iterations(gpu, n, eps, dt, its):
    bd, torch = gpu
    B, steps = 8, 16
    w = pi.Workload("two", n, pi.Flow("abc"), eps, B * steps * dt, B, dt, n_snap=0, m_cap=4, f_seed=3)
    u = torch.from_numpy(np.stack([pi.initial_state(n, seed=3 + b) for b in range(B)])).cuda()
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    s.set_initial(u[0].cpu().numpy(), w.f())
    out = s.op_fine(u, steps)[0]
    total = s.lin_stats()[0][:B]
    x = u.clone()

    def four_pass():   # in place: the four-pass kernel does all steps
        x.copy_(u)
        p = ctypes.c_void_p(x.data_ptr())
        s._check(s._lib.pr_op_fine(s.ctx, p, p, None, B, 0.0, steps, 1, 0))

    four_pass()
    for b in range(B):
        assert rel(out[b].cpu().numpy(), x[b].cpu().numpy()) < steps * step_tol(w, dt), b
    if its > 3:
        assert total.min() > its * steps
    else:
        assert abs(total - its * steps).max() <= steps // 4 + 4, total
        assert best_ms(torch, lambda: s.op_fine(u, steps)) < 0.9 * best_ms(torch, four_pass)
    s.close()
