"""Sampler boxes of 2D lattices whose object lies beyond 2^22 cells on an axis,
where FP32 coordinates no longer resolve half a cell, and of objects given by an
image of their centre outside the lattice: forces of the tiles (single lattices)
and of the row sweeps (batches) against one step per launch, bit for bit."""
import ctypes

import numpy as np
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


def _problem(n, axis, center, precision):
    # the short axis carries the wave; periods of 48 or 96 steps
    return workloads.problem(2, n, axis, float(n[axis]), 3.0, center, cp=0.4, n_surface=200, n_periods=2,
                             n_avg_periods=1, interface_d=0.5, precision=precision)


@pytest.mark.parametrize("n,axis,center,precision", [
    ((12, 4400000), 0, (1.5, 4300000.25), "f32"),
    ((12, 4400000), 0, (1.5, 4300000.25), "f16"),
    ((20000000, 12), 1, (19999999.5, 1.5), "f32"),    # across the far edge
    ((64, 60), 0, (72.25, -1.5), "f32"),              # an image of the centre
    ((64, 60), 0, (72.25, -1.5), "f64"),
])
def test_tiles_sample_far_objects(wlb, n, axis, center, precision):
    prob = _problem(n, axis, center, precision)
    T = prob["period"]
    with wlb.Solver(prob) as s:
        assert s.launch_info().steps[1] > 1
        s.init()
        s.step(5)
        s.step(T, sample=True)
        F = s.force()
    with wlb.Solver(prob) as s:
        s.init()
        s.step(5)
        F1 = np.zeros(3)
        assert wlb.lib().wlb_average_noalloc(s._h, T, F1.ctypes.data_as(ctypes.POINTER(ctypes.c_double))) == wlb.WLB_OK
    assert np.all(np.isfinite(F)) and np.any(F != 0) and np.array_equal(F, F1)


@pytest.mark.parametrize("precision", ["f32", "f16"])
def test_row_sweeps_sample_far_objects(wlb, precision):
    probs = [_problem((24, 4400000), 0, (3.0, 4300000.25), precision), _problem((64, 60), 0, (72.25, -1.5), precision)]
    with wlb.Batch(probs) as b:
        assert b.steps_per_launch(0) == 8
        F = b.run()
        b.set_two_step(False)
        one = b.run()
    assert np.all(np.isfinite(F)) and np.all(np.any(F != 0, axis=1)) and np.array_equal(F, one)


@pytest.mark.parametrize("center", [(3.0e9, 30.0), (30.0, -3.0e9)])
def test_centres_beyond_32_bits_go_without_boxes(wlb, center):
    prob = _problem((64, 60), 0, center, "f32")
    with wlb.Solver(prob) as s:
        assert s.launch_info().steps[1] == 1 and s.launch_info().steps[0] > 1
    with wlb.Batch([prob]) as b:
        assert b.steps_per_launch(0) == 2
