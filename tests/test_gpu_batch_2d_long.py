"""Runs of more launches than the row sweeps of 2D batches number in 32 bits keep
the two-step sweep, whose step counter has 64 (planned only, not run)."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("periods,steps", [(200000, 2), (100000, 8)])
def test_very_long_runs_keep_the_two_step_sweep(periods, steps):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2404_02346_gb300 import build as B
    B.build()
    import paper_2404_02346_gb300 as W
    prob = workloads.problem(2, (64, 32), 0, 16.0, 4.0, (32.0, 16.0), cp=2.0 ** -9, c0=2.0 ** -10, n_surface=8,
                             n_periods=periods, n_avg_periods=1, interface_d=1.0)
    assert prob["period"] == 16384  # 2048 launches a period
    with W.Batch([prob]) as b:
        assert b.steps_per_launch() == steps
