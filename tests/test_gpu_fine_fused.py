"""The FP32 mode's two-pass fine kernel on large grids against the oracle and against the
four-pass kernel, which also takes over the steps it leaves."""
import numpy as np
import pytest

import oracle as O
import pr_inputs as pi

pytestmark = pytest.mark.gpu

# Each step stops at a residual of 1e-9 of the right-hand side (see test_gpu_fine_chip.py), and
# the FP32 mode's residual leaves out dt L of the operand's rounding to a float (2^-25 of it).
TOL32_STEP = 4e-9


def step_tol(w, dt):
    h = 2 * np.pi / w.n
    return TOL32_STEP + 2.0 ** -25 * dt * (12 * w.eps / h ** 2 + 3 / h)


def rel(a, b):
    return float(np.linalg.norm(a.reshape(-1) - b.reshape(-1)) / np.linalg.norm(b.reshape(-1)))


def propagate(bd, torch, w, u, steps, dM=1, n_snap=0, **kw):
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32, **kw)
    s.set_initial(u[0], w.f())
    out, snap = s.op_fine(torch.from_numpy(u).cuda(), steps, dM, n_snap)
    tot, mx = s.lin_stats()
    r = out.cpu().numpy(), None if snap is None else snap.cpu().numpy(), tot[: len(u)], mx[: len(u)]
    s.close()
    return r


# one tile that wraps on both sides (40), tiles of even and odd rows, fewer threads than
# arrays' warps (68), the largest tile rows (64); groups that split a column and that cross it
@pytest.mark.parametrize("n,G,forced", [(40, 3, True), (52, 1, False), (52, 5, True), (64, 7, True), (68, 4, False),
                                        (76, 9, True)])
def test_two_pass_fine_matches_oracle(gpu, n, G, forced):
    bd, torch = gpu
    B, steps, dM, dt = 2, 4, 2, 1e-3
    w = pi.Workload("two", n, pi.Flow("abc"), 0.02, B * 10 * dt, B, dt, n_snap=0, m_cap=4, f_seed=5 if forced else None)
    u = np.stack([pi.initial_state(n, seed=20 + b) for b in range(B)])
    out, snap, _, _ = propagate(bd, torch, w, u, steps, dM, 3, group_ctas=G)
    op = O.make_operator(w)
    for b in range(B):
        ue, W = O.fine_propagate(op, u[b], 0.0, steps, dt, dM, 3, tol=1e-14)
        assert rel(out[b], ue) < steps * TOL32_STEP, (b, rel(out[b], ue))
        for j in range(3):
            assert rel(snap[b, j], W[:, j]) < steps * TOL32_STEP, (b, j)


# spin_limit = 0 keeps the four-pass kernel, which waits for nobody with one CTA a group.
# dt = 0.01: two or three iterations in every step, so the four-pass kernel resumes the items
# after a few; 0.1: many iterations; one step, fewer steps than a snapshot stride, and a last
# step that is a snapshot
@pytest.mark.parametrize("n", [40, 52])
@pytest.mark.parametrize("dt,steps,dM", [(1e-3, 12, 5), (1e-2, 9, 3), (1e-1, 3, 1), (1e-3, 1, 1)])
def test_two_pass_fine_matches_four_pass(gpu, n, dt, steps, dM):
    bd, torch = gpu
    B = 5
    w = pi.Workload("two", n, pi.Flow("kolmogorov", k=4), 0.02, B * 10 * dt, B, dt, n_snap=0, m_cap=4, f_seed=3)
    u = np.stack([pi.initial_state(n, seed=30 + b) for b in range(B)])
    n_snap = steps // dM + 1
    a, sa, ta, ma = propagate(bd, torch, w, u, steps, dM, n_snap, group_ctas=1, spin_limit=0)
    for G in (1, 4, 40):
        b, sb, tb, mb = propagate(bd, torch, w, u, steps, dM, n_snap, group_ctas=G)
        for i in range(B):
            assert rel(b[i], a[i]) < steps * step_tol(w, dt), (G, i, rel(b[i], a[i]))
            for j in range(n_snap):
                assert rel(sb[i, j], sa[i, j]) < steps * step_tol(w, dt), (G, i, j)
        # the same stopping rule: counts differ only where a residual sits at the threshold
        assert abs(tb - ta).max() <= 1 + steps // 4 and abs(mb - ma).max() <= 1, (ta, tb, ma, mb)


def test_two_pass_fine_in_place(gpu):
    # out = in: the state of the first step may not replace u_0 under the second launch
    bd, torch = gpu
    import ctypes
    n, B = 52, 2
    w = pi.Workload("two", n, pi.Flow("abc"), 0.02, 0.04, B, 1e-3, n_snap=0, m_cap=4)
    u = np.stack([pi.initial_state(n, seed=b) for b in range(B)])
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    out, _ = s.op_fine(torch.from_numpy(u).cuda(), 5)
    x = torch.from_numpy(u).cuda()
    p = ctypes.c_void_p(x.data_ptr())
    s._check(s._lib.pr_op_fine(s.ctx, p, p, None, B, 0.0, 5, 1, 0))
    assert rel(x.cpu().numpy(), out.cpu().numpy()) < 5 * TOL32_STEP
    s.close()


def test_two_pass_fine_at_rest_and_failures(gpu):
    bd, torch = gpu
    n = 52
    w = pi.Workload("two", n, pi.Flow("abc"), 0.05, 0.04, 4, 1e-3, n_snap=0, m_cap=4)
    u = np.stack([pi.initial_state(n, seed=b) for b in range(3)])
    u[1] = 0.0   # nothing to solve
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32)
    out, _ = s.op_fine(torch.from_numpy(u).cuda(), 3)
    assert not bool(out[1].any()) and bool(torch.isfinite(out).all())
    bad = u.copy()
    bad[2, 3, 2, 1] = np.nan
    with pytest.raises(bd.PRError) as e:
        s.op_fine(torch.from_numpy(bad).cuda(), 3)
    assert e.value.status == 7
    again, _ = s.op_fine(torch.from_numpy(u).cuda(), 3)   # the context stays usable
    assert torch.equal(again, out)
    s.close()
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32, lin_maxit=1)
    with pytest.raises(bd.PRError) as e:
        s.op_fine(torch.from_numpy(u).cuda(), 3)
    assert e.value.status == 4
    s.close()
