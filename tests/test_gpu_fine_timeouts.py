"""Waits of the two-pass fine sweep that run out: the call returns PR_ERR_TIMEOUT or a correct
result, writes nothing outside of its outputs, and leaves the device usable.  The workspace is
filled with bytes that are no step number, as memory fresh from an allocator may be."""
import ctypes

import numpy as np
import pytest

import pr_inputs as pi
from test_gpu_fine_fused import rel, step_tol

pytestmark = pytest.mark.gpu

PR_ERR_TIMEOUT = 6


def filled(bd, torch, w, fill, **kw):
    """A context whose workspace holds `fill` in every byte when it is bound."""
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32, workspace=False, **kw)
    n = s.workspace_bytes()
    s.ws = torch.full((n + 256,), fill, dtype=torch.uint8, device="cuda")
    s._check(s._lib.pr_bind_workspace(s.ctx, ctypes.c_void_p((s.ws.data_ptr() + 255) // 256 * 256), n))
    return s


def fine_into(s, torch, u, steps, dM, n_snap):
    """op_fine into buffers with guard words around the snapshots; its status and results."""
    B, Ng = u.shape[0], u[0].numel()
    guard = 1 << 16
    out = torch.zeros_like(u)
    buf = torch.full((2 * guard + B * n_snap * Ng,), -7.0, dtype=torch.float64, device="cuda")
    snap = buf[guard: guard + B * n_snap * Ng]
    st = s._lib.pr_op_fine(s.ctx, ctypes.c_void_p(u.data_ptr()), ctypes.c_void_p(out.data_ptr()),
                           ctypes.c_void_p(snap.data_ptr()), B, 0.0, steps, dM, n_snap)
    assert bool((buf[:guard] == -7.0).all()) and bool((buf[-guard:] == -7.0).all())
    return st, out.cpu().numpy(), snap.cpu().numpy().reshape(B, n_snap, -1)


# polls: fewer than a barrier between two CTAs needs, about as many, more; group sizes from one CTA
# (which waits for its copies only) to every SM; dt = 0.01 leaves items to the third launch
@pytest.mark.parametrize("limit", [1, 2, 20, 300])
@pytest.mark.parametrize("G,dt", [(0, 1e-3), (1, 1e-3), (4, 1e-3), (40, 1e-2)])
def test_two_pass_waits_that_run_out(gpu, limit, G, dt):
    bd, torch = gpu
    n, B, steps, dM, n_snap = 52, 5, 9, 2, 5
    w = pi.Workload("two", n, pi.Flow("kolmogorov", k=4), 0.02, B * 10 * dt, B, dt, n_snap=0, m_cap=4, f_seed=3)
    u = torch.from_numpy(np.stack([pi.initial_state(n, seed=30 + b) for b in range(B)])).cuda()
    s = bd.Parareal.from_workload(w, precision=bd.PR_FP32, group_ctas=G)
    s.set_initial(u[0].cpu().numpy(), w.f())
    st, ref, sref = fine_into(s, torch, u, steps, dM, n_snap)
    assert st == 0
    s.close()
    for fill in (0x80, 0x01):   # negative and large positive entries
        s = filled(bd, torch, w, fill, group_ctas=G, spin_limit=limit)
        s.set_initial(u[0].cpu().numpy(), w.f())
        for _ in range(2):      # the second call finds what the first one left
            st, out, snap = fine_into(s, torch, u, steps, dM, n_snap)
            assert st in (0, PR_ERR_TIMEOUT), st
            if st == 0:
                for b in range(B):
                    assert rel(out[b], ref[b]) < steps * step_tol(w, dt), b
                    assert rel(snap[b], sref[b]) < steps * step_tol(w, dt), b
        s.close()
    s = filled(bd, torch, w, 0x80, group_ctas=G)
    s.set_initial(u[0].cpu().numpy(), w.f())
    st, out, snap = fine_into(s, torch, u, steps, dM, n_snap)
    assert st == 0 and np.array_equal(out, ref) and np.array_equal(snap, sref)
    s.close()


# one CTA a group waits for its copies only: at one poll a copy that has not landed ends the
# launch, with others of it in flight (one tile of 40 rows, tiles of 16)
@pytest.mark.parametrize("n,steps", [(40, 6), (128, 4)])
def test_two_pass_copies_in_flight_when_a_wait_gives_up(gpu, n, steps):
    bd, torch = gpu
    B, dt = 6, 5e-4
    w = pi.Workload("two", n, pi.Flow("abc"), 0.005, B * 10 * dt, B, dt, n_snap=0, m_cap=4)
    u = torch.from_numpy(np.stack([pi.initial_state(n, seed=30 + b) for b in range(B)])).cuda()
    s = filled(bd, torch, w, 0x80, group_ctas=1)
    s.set_initial(u[0].cpu().numpy(), None)
    st, ref, _ = fine_into(s, torch, u, steps, 1, 2)
    assert st == 0
    t = filled(bd, torch, w, 0x80, group_ctas=1, spin_limit=1)
    t.set_initial(u[0].cpu().numpy(), None)
    for _ in range(3):
        st, out, _ = fine_into(t, torch, u, steps, 1, 2)
        assert st == PR_ERR_TIMEOUT or (st == 0 and rel(out, ref) < steps * step_tol(w, dt)), st
        assert fine_into(s, torch, u, steps, 1, 2)[0] == 0   # the device is as it was
    st, again, _ = fine_into(s, torch, u, steps, 1, 2)
    assert st == 0 and np.array_equal(again, ref)
    s.close()
    t.close()
