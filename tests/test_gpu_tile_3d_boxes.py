"""The sampling grid of 3D tiles with few points on a large sphere: the geometry
allows many more boxes than there are points, and a block beyond the points must
not read a box's entries (the list holds 27 entries per point)."""
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


@pytest.mark.parametrize("precision", ["f32", "f16"])
@pytest.mark.parametrize("R,N", [(4.0, 1), (8.0, 5), (16.0, 20), (16.0, 700)])
def test_no_more_sampling_blocks_than_points(wlb, R, N, precision):
    prob = workloads.problem(3, (40, 44, 48), 2, 24.0, R, (20.0, 21.5, 3.25), cp=0.4, n_surface=N, n_periods=2,
                             n_avg_periods=1, interface_d=0.5, precision=precision)
    T = prob["period"]
    with wlb.Solver(prob) as s:
        i = s.launch_info()
        assert i.steps[1] == 2 and 0 < i.sampler_blocks <= N
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
