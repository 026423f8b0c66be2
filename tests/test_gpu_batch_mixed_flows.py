"""A batched fine sweep of steady and time-dependent flows, whose kernels differ, gives each context
the bits of its sweep alone."""
import numpy as np
import pytest

import pr_inputs as pi
from test_gpu_serving import started

pytestmark = pytest.mark.gpu


# the on-chip kernel in both modes, and the FP32 mode's two-pass kernel
@pytest.mark.parametrize("prec,n", [(0, 16), (1, 16), (1, 52)])
def test_mixed_flows_sweep_as_alone(gpu, prec, n):
    bd, torch = gpu
    ws = [pi.Workload(name, n, flow, 0.02, 0.06, 3, 2e-3, n_snap=6, m_cap=4, f_seed=3)
          for name, flow in (("t", pi.Flow("paper_abc", w=1.3)), ("a", pi.Flow("abc")), ("k", pi.Flow("kolmogorov", k=2)))]
    alone = {}
    for w in ws:
        s = started(bd, w, prec, group_ctas=4)
        s.fine_sweep(1)
        alone[w.name] = [s.fine_end(i) for i in range(3)], [s.snapshots(i) for i in range(3)]
        s.close()
    ss = [started(bd, w, prec, group_ctas=4) for w in ws]
    bd.fine_sweep_batch(ss, [1, 1, 1])
    for s, w in zip(ss, ws):
        F, W = alone[w.name]
        for i in range(3):
            assert np.array_equal(s.fine_end(i), F[i]), (w.name, i)
            assert np.array_equal(s.snapshots(i), W[i]), (w.name, i)
        s.close()
