"""The FP64 streaming fine propagator (weights of the operator in shared memory) against the
oracle, at the tile shapes where the tables and the row slots can go wrong."""
import numpy as np
import pytest

import oracle as O
import pr_inputs as pi

pytestmark = pytest.mark.gpu

# The solves stop at 1e-14 of the right-hand side (parity bar of the FP64 mode, as for the
# other FP64 propagators)
TOL64 = 1e-12


# n: below a tile's height with one CTA (spin_limit = 0 keeps the streaming kernel there), two
# points a thread with tiles of several heights, odd rows with one and two row slots, a
# row longer than half a CTA; dt = 0.02: several BiCGStab iterations, so that the operand of
# the first and of the later ones is formed
@pytest.mark.parametrize("n,dt,pert,flow", [
    (4, 2e-2, 0, "abc"), (5, 2e-2, 0, "abc"), (36, 1e-3, 0, "abc"), (36, 2e-2, 3, "kolmogorov"), (37, 2e-2, 0, "abc"),
    (50, 1e-3, 2, "abc"), (52, 2e-2, 0, "kolmogorov"), (66, 1e-3, 0, "abc"), (68, 1e-3, 0, "paper_abc"),
    (96, 1e-3, 0, "abc"), (130, 1e-3, 0, "kolmogorov"), (132, 1e-3, 0, "abc")])
def test_streaming_fp64_matches_oracle(gpu, n, dt, pert, flow):
    bd, torch = gpu
    B, steps = 2, 2
    kw = {"group_ctas": 1, "spin_limit": 0} if n < 35 else {}
    w = pi.Workload("f64", n, pi.Flow(flow, k=2, pert_seed=pert), 0.02, B * 10 * dt, B, dt, n_snap=0, m_cap=4,
                    f_seed=None if flow == "paper_abc" else 5)
    u = np.stack([pi.initial_state(n, seed=40 + b) for b in range(B)])
    s = bd.Parareal.from_workload(w, precision=0, **kw)
    s.set_initial(u[0], w.f())
    out, snap = s.op_fine(torch.from_numpy(u).cuda(), steps, 1, 2)
    out, snap = out.cpu().numpy(), snap.cpu().numpy()
    s.close()
    op = O.make_operator(w)
    rel = lambda a, b: float(np.linalg.norm((a - b.reshape(a.shape)).reshape(-1)) / np.linalg.norm(b.reshape(-1)))
    ue, W = O.fine_propagate(op, u[1], 0.0, steps, dt, 1, 2, tol=1e-14)
    assert rel(out[1], ue) < TOL64
    for j in range(2):
        assert rel(snap[1, j], W[:, j]) < TOL64, j
