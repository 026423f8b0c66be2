"""Which kernel a fine sweep takes (told by its launches: one on chip, three in two passes), and its
states there: uneven slabs of the 4-wide on-chip form, the two-pass kernel's tiles of large grids."""
import ctypes

import numpy as np
import pytest

import oracle as O
import pr_inputs as pi
from test_gpu_fine_fused import rel, step_tol

pytestmark = pytest.mark.gpu


# a positive group size on small grids is the cluster's: any up to 36, beyond it one that fits
@pytest.mark.parametrize("n,G,launches", [(36, 11, 1), (36, 40, 1), (40, 9, 1), (40, 6, 3), (44, 16, 1), (48, 9, 3), (48, 16, 1),
                                          (52, 9, 3), (64, 0, 3)])
def test_kernel_of_a_group_size(gpu, n, G, launches):
    bd, torch = gpu
    B, steps, dt = 2, 3, 1e-3
    w = pi.Workload("route", n, pi.Flow("abc"), 0.02, B * 10 * dt, B, dt, n_snap=0, m_cap=4, f_seed=5)
    u = np.stack([pi.initial_state(n, seed=20 + b) for b in range(B)])
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32, group_ctas=G)
    s.set_initial(u[0], w.f())
    x = torch.from_numpy(u).cuda()
    s.op_fine(x, steps)
    before = bd.launch_count()
    out = s.op_fine(x, steps)[0].cpu().numpy()
    assert bd.launch_count() - before == launches
    s.close()
    op = O.make_operator(w)
    for b in range(B):
        ue, _ = O.fine_propagate(op, u[b], 0.0, steps, dt, tol=1e-14)
        assert rel(out[b], ue) < steps * step_tol(w, dt), b


# tiles of 16, 8 and 32 rows (96, 128 and 256, 64): against the four-pass kernel, which an in-place
# call takes; groups that end within a tile's column
@pytest.mark.parametrize("n,G", [(64, 5), (96, 7), (96, 0), (128, 9), (128, 0), (256, 0)])
def test_two_pass_tiles_of_large_grids(gpu, n, G):
    bd, torch = gpu
    B, steps, dt = (1 if n == 256 else 2), 4, 5e-4
    w = pi.Workload("tiles", n, pi.Flow("abc"), 0.005, B * 10 * dt, B, dt, n_snap=0, m_cap=2, f_seed=3)
    u = torch.from_numpy(np.stack([pi.initial_state(n, seed=3 + b) for b in range(B)])).cuda()
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32, group_ctas=G)
    s.set_initial(u[0].cpu().numpy(), w.f())
    out = s.op_fine(u, steps)[0]
    p = ctypes.c_void_p(u.data_ptr())
    s._check(s._lib.pr_op_fine(s.ctx, p, p, None, B, 0.0, steps, 1, 0))
    s.close()
    for b in range(B):
        err, ref = (out[b] - u[b]).abs(), u[b]
        assert float((out[b] - ref).norm() / ref.norm()) < steps * step_tol(w, dt), b
        # no plane or row of a tile stands out: pointwise within the residual's and the float
        # increment's bounds at the size of the largest value
        assert float(err.max() / ref.abs().max()) < 40 * steps * step_tol(w, dt), b
