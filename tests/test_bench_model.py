"""bench.py's byte model follows the kernels: which grids take the two-pass fine sweep."""
import pytest

import bench
import pr_inputs as pi


@pytest.mark.parametrize("n,takes", [(48, False), (50, False), (52, True), (64, True), (92, False), (96, True), (116, False),
                                     (124, False), (128, True), (148, False), (164, False), (256, True)])
def test_grids_of_the_two_pass_sweep(n, takes):
    w = pi.Workload("w", n, pi.Flow("abc"), 0.05, 1.0, 4, 1e-3)
    assert bench.fine_two_pass("fp32", w) is takes
    assert not bench.fine_two_pass("fp64", w)
    assert not bench.fine_two_pass("fp32", pi.Workload("w", n, pi.Flow("abc", pert_seed=1), 0.05, 1.0, 4, 1e-3))
