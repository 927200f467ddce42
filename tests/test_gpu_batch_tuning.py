"""The autotuner's time per step of 2D row sweeps counts the steps that its
launches take: no launch beyond a run's end, and each width's own steps."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wlb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2404_02346_gb300 import build as B
    B.build()
    import paper_2404_02346_gb300 as W
    W.lib()
    return W


def _problem(nx, ny):
    # a period of 64 steps along x
    return workloads.problem(2, (nx, ny), 0, 16.0, 4.0, (nx / 2, ny / 2), cp=0.4, n_surface=8, n_periods=1,
                             n_avg_periods=0, interface_d=1.0, precision="f32")


def test_time_per_step_of_trials_longer_than_the_run(wlb):
    """64 steps of 17 M cells are eight launches of about 0.1 ms; a hundred times
    as many steps per trial reach the same eight.  Counting the empty launches
    would give a time per step at least four times shorter."""
    with wlb.Batch([_problem(128, 131072)]) as b:
        assert b.steps_per_launch() == 8
        short, long = b.autotune(64)["ms_per_step"], b.autotune(6400)["ms_per_step"]
    assert 0.5 * short < long < 2.0 * short


def test_time_per_step_of_mixed_widths(wlb):
    """A wide lattice that takes four steps in the launch in which a tiny one takes
    eight: the time per step is the wide one's own."""
    wide, tiny = _problem(256, 65536), _problem(64, 32)
    with wlb.Batch([wide]) as b:
        assert b.steps_per_launch() == 4
        alone = b.autotune(32)["ms_per_step"]
    with wlb.Batch([wide, tiny]) as b:
        assert (b.steps_per_launch(0), b.steps_per_launch(1)) == (4, 8)
        both = b.autotune(32)["ms_per_step"]
    assert 0.7 * alone < both < 1.4 * alone
