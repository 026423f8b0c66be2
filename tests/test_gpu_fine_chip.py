"""The on-chip fine propagator (one thread-block cluster a subinterval) against the oracle
and against the streaming kernel it replaces on small grids."""
import numpy as np
import pytest

import oracle as O
import pr_inputs as pi

pytestmark = pytest.mark.gpu

# FP64: the parity bar.  FP32 mode: each step stops at a residual of 1e-9 of the right-hand
# side, so S steps are off by S * 1e-9 at the size of the state, with a factor for the norm of
# (I + dt L)^-1 and the float-pair rounding
TOL64, TOL32_STEP = 1e-12, 4e-9


def propagate(bd, torch, w, prec, u, steps, dM=1, n_snap=0, **kw):
    s = bd.Parareal.from_workload(w, precision=prec, **kw)
    s.set_initial(u[0], w.f())
    out, snap = s.op_fine(torch.from_numpy(u).cuda(), steps, dM, n_snap)
    tot, mx = s.lin_stats()
    r = out.cpu().numpy(), None if snap is None else snap.cpu().numpy(), tot[: len(u)], mx[: len(u)]
    s.close()
    return r


def rel(a, b):
    return float(np.linalg.norm(a.reshape(-1) - b.reshape(-1)) / np.linalg.norm(b.reshape(-1)))


# n: smallest, below and at a warp's width, odd, the largest that fits in each mode; C: one
# CTA, slabs of unequal height, the largest cluster; dt = 0.02: several BiCGStab iterations
@pytest.mark.parametrize("prec,n,G,dt,pert", [
    (0, 4, 0, 1e-3, 0), (0, 5, 3, 2e-2, 0), (0, 16, 16, 2e-2, 0), (0, 17, 5, 1e-3, 2), (0, 28, 7, 2e-2, 0),
    (0, 34, 0, 1e-3, 0), (1, 4, 4, 1e-3, 0), (1, 7, 2, 2e-2, 3), (1, 16, 1, 2e-2, 0), (1, 31, 11, 1e-3, 0),
    (1, 32, 16, 2e-2, 2), (1, 40, 9, 1e-3, 0), (1, 47, 0, 1e-3, 0), (1, 48, 0, 1e-3, 0)])
def test_cluster_fine_matches_oracle(gpu, prec, n, G, dt, pert):
    bd, torch = gpu
    flow = pi.Flow("abc", pert_seed=pert)
    B, steps, dM = 3, 4, 2
    w = pi.Workload("chip", n, flow, 0.02, B * 10 * dt, B, dt, n_snap=0, m_cap=4, f_seed=5)
    u = np.stack([pi.initial_state(n, seed=20 + b) for b in range(B)])
    out, snap, _, _ = propagate(bd, torch, w, prec, u, steps, dM, 3, group_ctas=G)
    op = O.make_operator(w)
    tol = TOL64 if prec == 0 else steps * TOL32_STEP
    for b in (0, B - 1):
        ue, W = O.fine_propagate(op, u[b], 0.0, steps, dt, dM, 3, tol=1e-14)
        assert rel(out[b], ue) < tol, (b, rel(out[b], ue))
        for j in range(3):
            assert rel(snap[b, j], W[:, j]) < tol, (b, j)


# spin_limit = 0 keeps the streaming kernel, which waits for nobody with one CTA a group
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,dt,forced", [(6, 5e-3, True), (16, 1e-3, False), (16, 3e-2, True), (24, 1e-2, True)])
def test_cluster_fine_matches_streaming_kernel(gpu, prec, n, dt, forced):
    bd, torch = gpu
    B, steps = 5, 6
    w = pi.Workload("chip", n, pi.Flow("kolmogorov", k=2), 0.05, B * 10 * dt, B, dt, n_snap=0, m_cap=4,
                    f_seed=3 if forced else None)
    u = np.stack([pi.initial_state(n, seed=30 + b) for b in range(B)])
    u[2] = 0.0   # nothing to solve without forcing
    a, sa, ta, ma = propagate(bd, torch, w, prec, u, steps, 3, 2, group_ctas=1, spin_limit=0)
    for G in (0, 1, 4, 6):
        b, sb, tb, mb = propagate(bd, torch, w, prec, u, steps, 3, 2, group_ctas=G)
        tol = 1e-13 if prec == 0 else steps * TOL32_STEP
        for i in range(B):
            if np.any(a[i]):
                assert rel(b[i], a[i]) < tol, (G, i, rel(b[i], a[i]))
            else:
                assert not np.any(b[i])
            assert abs(sb[i] - sa[i]).max() <= tol * max(1.0, abs(sa[i]).max()) * 40
        # the same stopping rule: counts differ only where a residual sits at the threshold
        assert abs(tb - ta).max() <= 1 and abs(mb - ma).max() <= 1, (ta, tb)


def test_cluster_fine_reports_non_finite_states(gpu):
    bd, torch = gpu
    w = pi.Workload("chip", 16, pi.Flow("abc"), 0.05, 0.04, 4, 1e-3, n_snap=0, m_cap=4)
    u = np.stack([pi.initial_state(16, seed=b) for b in range(4)])
    u[1, 3, 2, 1] = np.inf
    for prec in (0, 1):
        s = bd.Parareal.from_workload(w, precision=prec)
        with pytest.raises(bd.PRError) as e:
            s.op_fine(torch.from_numpy(u).cuda(), 3)
        assert e.value.status == 7
        out, _ = s.op_fine(torch.from_numpy(u[2:3]).cuda(), 3)   # the context stays usable
        assert bool(torch.isfinite(out).all())
        s.close()
