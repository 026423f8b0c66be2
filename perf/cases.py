"""Timed cases of the library: the calls that a user's program makes, over the sizes it makes
them at.

* ``fine``   ``Parareal.op_fine``: the fine propagator on a batch of states, with snapshots;
* ``pod``    ``Parareal.op_pod``: POD_Mode of a batch of snapshot windows;
* ``coarse`` ``Parareal.op_coarse_update``: one augmented coarse update;
* ``apply``  ``Parareal.op_apply_L``: the advection-diffusion operator on grid functions;
* ``solve``  ``Parareal.solve``: all of Algorithm 2, run to its finite termination k = N, where
  the iterates are the sequential fine solution.  (Earlier iterates respond to rounding by
  many orders of magnitude, which is a property of the method: the kept POD subspaces move.)

Sizes are those of the workloads in ``pr_inputs`` (16^3, 64^3, 128^3; the serving stream's
32^3 to 128^3), of their snapshot windows and POD caps, and odd grids as in the tests.
"""
import math

import numpy as np
import torch

import pr_inputs as pi
from paper_2601_10981_gb300 import binding as bd


def listed():
    return [
        # the 16^3 workload: one whole FP64 solve, and its fine propagator alone.  Smallest
        # calls: what a user runs first, bound by latency
        dict(name="solve_abc16_fp64", kind="solve", n=16, N=8, steps=125, flow="abc", k=1, eps=0.05, dt=1e-3,
             n_snap=0, m_cap=8, fp32=False, forced=False),
        dict(name="fine_abc16_fp64", kind="fine", n=16, B=8, steps=125, flow="abc", k=1, eps=0.05, dt=1e-3,
             n_snap=26, fp32=False, forced=False, pert=False),
        # the 64^3 Kolmogorov workload: the fine sweep of its 64 windows with 32 snapshots
        # each (most of an iteration's time), and some steps of it in FP64
        dict(name="fine_kol64_fp32", kind="fine", n=64, B=64, steps=157, flow="kolmogorov", k=4, eps=0.01, dt=1e-3,
             n_snap=32, fp32=True, forced=True, pert=False),
        dict(name="fine_kol64_fp64", kind="fine", n=64, B=64, steps=16, flow="kolmogorov", k=4, eps=0.01, dt=1e-3,
             n_snap=4, fp32=False, forced=True, pert=False),
        # one wave of the 128^3 workload (38 windows), part of its steps
        dict(name="fine_abc128_fp32", kind="fine", n=128, B=38, steps=60, flow="abc", k=1, eps=0.005, dt=5e-4,
             n_snap=8, fp32=True, forced=False, pert=False),
        # a request of the serving stream on 96^3, with the shortest horizon it is served at
        dict(name="fine_kol96_fp32", kind="fine", n=96, B=16, steps=62, flow="kolmogorov", k=8, eps=0.02, dt=1e-3,
             n_snap=32, fp32=True, forced=False, pert=False),
        # an odd grid (no vector accesses) in the FP32 mode, with a stored perturbation
        dict(name="fine_odd45_fp32", kind="fine", n=45, B=16, steps=50, flow="kolmogorov", k=2, eps=0.01, dt=1e-3,
             n_snap=11, fp32=True, forced=True, pert=True),
        # level-1 POD of the 64^3 workload's windows (32 snapshots, cap 16) and of a few of the
        # 128^3 workload's (64 snapshots, cap 32)
        dict(name="pod_64_fp32", kind="pod", n=64, B=64, cols=32, cap=16, waves=3, fp32=True),
        dict(name="pod_128_fp32", kind="pod", n=128, B=4, cols=64, cap=32, waves=8, fp32=True),
        # one coarse update at the 64^3 workload's POD cap
        dict(name="coarse_64_fp32", kind="coarse", n=64, m=16, flow="kolmogorov", k=4, eps=0.01, fp32=True),
        # the operator on a basis of the 128^3 workload
        dict(name="apply_128_fp64", kind="apply", n=128, count=32, flow="abc", k=1, eps=0.005, transpose=False),
        # a whole FP32-mode solve on 64^3 with short windows (16 subintervals of 16 fine steps,
        # a serving request's horizon): fine sweeps, PODs and coarse sweeps weigh about alike
        dict(name="solve_kol64_fp32", kind="solve", n=64, N=16, steps=16, flow="kolmogorov", k=4, eps=0.01, dt=1e-3,
             n_snap=32, m_cap=16, fp32=True, forced=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fine", "fine", "fine", "pod", "coarse", "apply", "solve"])
    flow = rng.choice(["abc", "kolmogorov"])
    k = rng.choice([2, 4, 8]) if flow == "kolmogorov" else 1
    eps = math.exp(rng.uniform(math.log(0.002), math.log(0.05)))
    if kind == "fine":
        fp32 = rng.random() < 0.7
        n = _log(rng, 12, 128 if fp32 else 64)
        if n % 4 and rng.random() < 0.6:
            n = (n + 3) // 4 * 4
        # points x steps within the largest listed case (FP64 costs ten times as much)
        budget = (1.0e9 if fp32 else 1.0e8) * math.exp(-2.0 * rng.random())
        B = _log(rng, 2, 64)
        steps = max(4, min(160, int(budget / (B * n ** 3))))
        return dict(kind=kind, n=n, B=B if B * n ** 3 * steps < 2.0e9 else 2, steps=steps, flow=flow, k=k, eps=eps,
                    dt=5e-4 if n > 100 else 1e-3, n_snap=rng.choice([0, 2, min(steps, 11)]), fp32=fp32,
                    forced=rng.random() < 0.5, pert=rng.random() < 0.2)
    if kind == "pod":
        n = _log(rng, 16, 96)
        cols = rng.randint(6, 64)
        B = max(1, min(64, int(4.0e8 * rng.uniform(0.1, 1.0) / (cols * n ** 3))))
        waves = rng.randint(1, min(12, cols // 3))
        return dict(kind=kind, n=n, B=B, cols=cols, cap=min(32, max(2 * waves, 8)), waves=waves, fp32=rng.random() < 0.7)
    if kind == "coarse":
        return dict(kind=kind, n=_log(rng, 16, 128), m=rng.randint(2, 32), flow=flow, k=k, eps=eps, fp32=rng.random() < 0.7)
    if kind == "apply":
        n = _log(rng, 8, 128)
        return dict(kind=kind, n=n, count=_log(rng, 1, 64), flow=flow, k=k, eps=eps, transpose=rng.random() < 0.5)
    n = _log(rng, 8, 40)
    return dict(kind="solve", n=n, N=rng.randint(3, 8), steps=_log(rng, 5, 60), flow=flow, k=k, eps=eps, dt=1e-3,
                n_snap=rng.choice([0, 8, 32]), m_cap=rng.choice([4, 8, 16]) if n > 12 else 4, fp32=rng.random() < 0.6,
                forced=rng.random() < 0.5)


# ---------------------------------------------------------------------------------------
# inputs

def _flow(case, seed):
    if case.get("pert"):
        return pi.Flow(case["flow"], k=case["k"], pert_seed=1 + seed % 1000003, pert_amp=0.05)
    return pi.Flow(case["flow"], k=case["k"])


def _modes(rng, count, kmax=4):
    """`count` different wave vectors (one of each +-k pair) with |k| <= kmax."""
    every = pi.half_space_modes(kmax)
    return [every[i] for i in rng.choice(len(every), count, replace=False)]


def _waves(n, modes):
    """cos(k.x), sin(k.x) of the wave vectors on the grid: (2 len(modes), n^3), float64, on the GPU."""
    x = torch.arange(n, dtype=torch.float64, device="cuda") * (2.0 * math.pi / n)
    out = torch.empty((2 * len(modes), n, n, n), dtype=torch.float64, device="cuda")
    for j, (kx, ky, kz) in enumerate(modes):
        ph = (kz * x)[:, None, None] + (ky * x)[None, :, None] + (kx * x)[None, None, :]
        torch.cos(ph, out=out[2 * j])
        torch.sin(ph, out=out[2 * j + 1])
    return out.view(2 * len(modes), -1)


def _states(n, B, seed):
    """B smooth states, sin x sin y sin z plus seeded modes with |k| <= 3 of amplitude 0.1 (the
    initial states of the workloads)."""
    rng = np.random.default_rng(seed)
    modes = pi.half_space_modes(3)
    W = _waves(n, modes)
    c = torch.from_numpy(rng.uniform(-0.1, 0.1, (B, W.shape[0]))).cuda()
    s = torch.sin(torch.arange(n, dtype=torch.float64, device="cuda") * (2.0 * math.pi / n))
    base = s[:, None, None] * s[None, :, None] * s[None, None, :]
    return (c @ W).view(B, n, n, n) + base


def _windows(case, seed):
    """Snapshot windows: travelling, decaying waves sampled over the window (the solution of a
    constant-coefficient advection-diffusion problem), `waves` wave vectors each with phase
    speeds apart, so that the window has 2 `waves` modes well above rounding."""
    n, B, cols, nw = case["n"], case["B"], case["cols"], case["waves"]
    rng = np.random.default_rng(seed)
    t = np.linspace(0.0, 1.0, cols)
    W = torch.empty((B, cols, n ** 3), dtype=torch.float64, device="cuda")
    for b in range(B):
        modes = _modes(rng, nw)
        basis = _waves(n, modes)
        C = np.empty((cols, 2 * nw))
        for j in range(nw):
            amp = 0.8 ** (0.5 * j) * rng.uniform(0.95, 1.05)
            sweep, ph = math.pi * (1.0 + j) * rng.uniform(0.95, 1.05), rng.uniform(0.0, 2.0 * math.pi)
            C[:, 2 * j] = amp * np.exp(-0.2 * t) * np.cos(sweep * t + ph)
            C[:, 2 * j + 1] = amp * np.exp(-0.2 * t) * np.sin(sweep * t + ph)
        torch.matmul(torch.from_numpy(C).cuda(), basis, out=W[b])
    return W.view(B, cols, n, n, n)


def _coarse_inputs(case, seed):
    """An orthonormal basis of m smooth fields, U with a part of relative size 1e-3 outside of
    its span, the previous iterate near U, and the fine end state."""
    n, m = case["n"], case["m"]
    rng = np.random.default_rng(seed)
    modes = _modes(rng, (m + 1) // 2 + 6)
    W = _waves(n, modes) * math.sqrt(2.0 / n ** 3)
    R = W[:m].contiguous()
    amp = math.sqrt(n ** 3)

    def field(size, scale):
        c = np.zeros(W.shape[0])
        c[:m] = rng.uniform(-1.0, 1.0, m) * scale
        c[m:] = rng.uniform(-1.0, 1.0, W.shape[0] - m) * size * scale
        return (torch.from_numpy(c).cuda() @ W) * amp

    U = field(1e-3, 0.3)
    Up = U + field(1e-1, 1e-2)
    F = field(1e-2, 0.3)
    return R, U, Up, F


def _u0f(case, seed):
    u0 = pi.initial_state(case["n"], 1 + seed % 1000003)
    f = pi.forcing(case["n"], 2 + seed % 1000003) if case["forced"] else None
    return u0, f


def _solver(case, N, steps, flow, n_snap, m_cap, eps, dt):
    """A context over N subintervals of `steps` fine steps of size dt."""
    w = pi.Workload("case", case["n"], flow, eps, N * steps * dt, N, dt, n_snap=n_snap, m_cap=m_cap)
    return bd.Parareal.from_workload(w, precision=bd.PR_FP32 if case.get("fp32") else bd.PR_FP64)


def _dM(case):
    return max(1, case["steps"] // (case["n_snap"] - 1)) if case["n_snap"] > 1 else 1


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    st = {"case": case}
    if kind == "fine":
        # the context that a program keeps for this problem, its forcing set once
        s = _solver(case, case["B"], case["steps"], _flow(case, seed), max(2, case["n_snap"]), 4, case["eps"], case["dt"])
        u0, f = _u0f(case, seed)
        s.set_initial(u0, f)
        st.update(s=s, u=_states(n, case["B"], seed))
    elif kind == "pod":
        w = pi.Workload("case", n, pi.Flow("abc"), 0.05, 1.0, case["B"], 1.0 / (case["B"] * (case["cols"] - 1)),
                        n_snap=case["cols"], m_cap=case["cap"])
        s = bd.Parareal.from_workload(w, precision=bd.PR_FP32 if case["fp32"] else bd.PR_FP64)
        st.update(s=s, W=_windows(case, seed))
    elif kind == "coarse":
        s = _solver(case, 2, 20, _flow(case, seed), 12, max(12, case["m"]), case["eps"], 1e-3)
        R, U, Up, F = _coarse_inputs(case, seed)
        st.update(s=s, R=R, U=U, Up=Up, F=F)
    elif kind == "apply":
        s = _solver(case, 32, 2, _flow(case, seed), 2, 2, case["eps"], 1e-3)
        st.update(s=s, u=_states(n, case["count"], seed))
    else:
        s = _solver(case, case["N"], case["steps"], _flow(case, seed), case["n_snap"], case["m_cap"], case["eps"], case["dt"])
        u0, f = _u0f(case, seed)
        out = torch.empty((case["N"] + 1, n, n, n), dtype=torch.float64, pin_memory=True).numpy()
        st.update(s=s, u0=u0, f=f, out=out)
    return st


def run(st):
    case, s = st["case"], st["s"]
    kind = case["kind"]
    if kind == "fine":
        out, snap = s.op_fine(st["u"], case["steps"], dM=_dM(case), n_snap=case["n_snap"])
        return {"u": out} if snap is None else {"u": out, "snapshots": snap}
    if kind == "pod":
        R, m = s.op_pod(st["W"], 1.0 - 5e-6, cap=case["cap"])
        return {"R": R, "m": m}
    if kind == "coarse":
        return s.op_coarse_update(st["R"], case["m"], st["U"], st["Up"], st["F"])
    if kind == "apply":
        return s.op_apply_L(st["u"], transpose=case["transpose"])
    # a solve from the host's initial state to the host's copy of the interface states; the
    # tolerance is below what any iterate but the last one meets
    s.set_initial(st["u0"], st["f"])
    s.solve(1e-14, k_max=case["N"])
    return s.interfaces(out=st["out"])


def work(case):
    """Each input read and each output written once; the floating-point operations of the
    method itself (a seven-point operator: 14; an implicit step: a residual and, at least, the two
    operator applications, five dot products and three updates of one BiCGStab iteration)."""
    n3 = case["n"] ** 3
    kind = case["kind"]
    step = 20 + 2 * 14 + 5 * 2 + 3 * 4
    if kind == "fine":
        return {"bytes": 8.0 * n3 * case["B"] * (2 + case["n_snap"]), "flops": float(step) * n3 * case["B"] * case["steps"]}
    if kind == "pod":
        K, m, B = case["cols"], 2 * case["waves"], case["B"]
        return {"bytes": 8.0 * n3 * B * (K + min(m, case["cap"])), "flops": 2.0 * n3 * B * (K * (K + 1) / 2 + K * m)}
    if kind == "coarse":
        m = case["m"]
        # the basis, U, U', F and the result; L R and R^T L R, then the 7 m products of the update
        return {"bytes": 8.0 * n3 * (m + 4), "flops": float(n3) * (14 * m + 2 * m * m + 2 * 7 * m + 2 * 14)}
    if kind == "apply":
        return {"bytes": 16.0 * n3 * case["count"], "flops": 14.0 * n3 * case["count"]}
    N = case["N"]
    sweeps = N * (N + 1) / 2 + 1
    return {"bytes": 8.0 * n3 * (N + 3), "flops": float(step) * n3 * case["steps"] * sweeps}


# ---------------------------------------------------------------------------------------
# the same results in 64 bits, by plain torch

class _Op:
    """L u = b.grad u - eps Lap u with second-order central differences on the periodic cube."""

    def __init__(self, case, seed):
        n = case["n"]
        self.h, self.eps = 2.0 * math.pi / n, case["eps"]
        x = torch.arange(n, dtype=torch.float64, device="cuda") * self.h
        X, Y, Z = x[None, None, :], x[None, :, None], x[:, None, None]
        if case["flow"] == "abc":
            b = (torch.sin(Z) + torch.cos(Y), torch.sin(X) + torch.cos(Z), torch.sin(Y) + torch.cos(X))
        else:
            zero = torch.zeros(1, 1, 1, dtype=torch.float64, device="cuda")
            b = (torch.sin(case["k"] * Y), zero, zero)
        if case.get("pert"):
            p = torch.from_numpy(_flow(case, seed).pert(n)).cuda()
            b = tuple(b[d] + p[d] for d in range(3))
        self.b = b

    def L(self, u, transpose=False):
        lap = -6.0 * u
        adv = 0.0
        for d, axis in enumerate((-1, -2, -3)):
            if transpose:      # (L^T u)_i: the column of b_d u, with the opposite sign
                w = self.b[d] * u
                adv = adv - (torch.roll(w, -1, axis) - torch.roll(w, 1, axis))
                lap = lap + (torch.roll(u, -1, axis) + torch.roll(u, 1, axis))
            else:
                up, um = torch.roll(u, -1, axis), torch.roll(u, 1, axis)
                adv = adv + self.b[d] * (up - um)
                lap = lap + (up + um)
        return adv * (0.5 / self.h) - (self.eps / self.h ** 2) * lap

    def steps(self, u, f, dt, steps, dM=1, n_snap=0):
        """Implicit Euler, each step by the fixed point delta = dt (f - L u) - dt L delta."""
        vmax = sum(float(c.abs().max()) for c in self.b)
        rho = dt * (12.0 * self.eps / self.h ** 2 + vmax / self.h)
        its = max(3, int(math.ceil(math.log(1e-17) / math.log(min(0.9, rho)))))
        snaps = [u.clone()] if n_snap > 0 else []
        for j in range(1, steps + 1):
            r = -dt * self.L(u)
            if f is not None:
                r = r + dt * f
            d = r.clone()
            for _ in range(its):
                d = r - dt * self.L(d)
            u = u + d
            if j % dM == 0 and len(snaps) < n_snap:
                snaps.append(u.clone())
        return u, snaps


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "pod":
        # the sign of an eigenvector is free, so the basis has no value of its own
        return {"R": None, "m": np.full(case["B"], 2 * case["waves"], dtype=np.int32)}
    op = _Op(case, seed)
    if kind == "apply":
        return op.L(_states(n, case["count"], seed), transpose=case["transpose"])
    if kind == "fine":
        _, f = _u0f(case, seed)
        f = None if f is None else torch.from_numpy(f).cuda()
        u, snaps = op.steps(_states(n, case["B"], seed), f, case["dt"], case["steps"], _dM(case), case["n_snap"])
        return {"u": u, "snapshots": torch.stack(snaps, dim=1)} if snaps else {"u": u}
    if kind == "coarse":
        R, U, Up, F = _coarse_inputs(case, seed)
        d = U - R.T @ (R @ U)
        d = d - R.T @ (R @ d)
        V = torch.cat([R, (d / torch.linalg.norm(d))[None]])
        LV = op.L(V.view(-1, n, n, n)).reshape(V.shape[0], -1)
        M, A = V @ V.T, V @ LV.T
        DeltaT = 20 * 1e-3
        dT = DeltaT / 10
        x = torch.linalg.solve(M, V @ (U - Up))
        for _ in range(10):
            x = torch.linalg.solve(M + dT * A, M @ x)
        return F + V.T @ x
    u0, f = _u0f(case, seed)
    u = torch.from_numpy(u0).cuda()
    f = None if f is None else torch.from_numpy(f).cuda()
    out = []
    for _ in range(case["N"] + 1):      # [0, T0], then the N subintervals
        u, _ = op.steps(u, f, case["dt"], case["steps"])
        out.append(u)
    return torch.stack(out)
