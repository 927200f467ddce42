"""Several steps per launch on 2D lattices (overlapped tiles, the default path
of a single 2D handle) against one step per launch (wlb_average_noalloc, which
launches the sampling and the update of every step on their own): fields and
forces bit for bit.  Shapes where the tiling ends: tiny lattices whose box
wraps onto itself, odd sizes, ragged last tiles, objects and sampler boxes
across the periodic edges, waves along x, walls and source sheet, one surface
point, more points than a sampler takes, step counts that are no multiple of
the steps per launch."""
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


def _one_step_launches(W, solver, n):
    F = np.zeros(3)
    st = W.lib().wlb_average_noalloc(solver._h, n, F.ctypes.data_as(ctypes.POINTER(ctypes.c_double)))
    assert st == W.WLB_OK
    return F


CASES = [
    # nx, ny, axis, lam, R, d, center, N
    (9, 8, 1, 8.0, 1.0, 0.25, (4.25, 5.0), 8),            # smaller than a box: it wraps
    (22, 24, 1, 24.0, 3.0, 1.0, (0.125, 23.5), 33),       # object across both edges
    (57, 64, 1, 32.0, 5.0, 4.0, (30.0, 4.25), 1),         # odd rows, one point
    (64, 57, 0, 64.0, 8.0, 4.0, (8.5, 28.25), 129),       # wave along x
    (130, 96, 1, 48.0, 6.5, 4.0, (129.5, 6.0), 700),      # dense points
    (301, 180, 1, 60.0, 40.0, 4.0, (150.25, 90.5), 90),   # sparse points on a large circle
    (600, 400, 1, 100.0, 10.0, 4.0, (300.5, 12.5), 300),  # several waves of tiles
]


@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
@pytest.mark.parametrize("nx,ny,axis,lam,R,d,center,N", CASES)
def test_tiles_equal_one_step_per_launch(wlb, nx, ny, axis, lam, R, d, center, N, precision):
    prob = workloads.problem(2, (nx, ny), axis, lam, R, center, cp=0.4, n_surface=N, n_periods=3, n_avg_periods=1,
                             interface_d=d, precision=precision)
    T = prob["period"]
    # whole periods (graphs) and pieces; the sampled window starts inside a period
    with wlb.Solver(prob) as s:
        s.init()
        s.step(T + 5)
        for n in (1, T - 2, 7):
            s.step(n, sample=True)
        F, (p1, u1) = s.force(), s.fields()
        s.step(13)
        q1, v1 = s.fields()
    with wlb.Solver(prob) as s:
        s.init()
        _one_step_launches(wlb, s, T + 5)
        F1 = _one_step_launches(wlb, s, T + 6)
        r1, w1 = s.fields()
        _one_step_launches(wlb, s, 13)
        t1, x1 = s.fields()
    assert np.array_equal(p1, r1) and np.array_equal(u1, w1)
    assert np.array_equal(q1, t1) and np.array_equal(v1, x1)
    assert np.all(np.isfinite(F)) and np.array_equal(F, F1)


@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
@pytest.mark.parametrize("nx,axis,length", [(64, 1, 35), (33, 1, 203), (61, 0, 30)])
def test_driven_tiles_equal_one_step_per_launch(wlb, nx, axis, length, precision):
    """The driven cavity: every step of a launch has its own source amplitude,
    and walls and sheet lie in tiles and in halos that wrap onto the far wall."""
    n = (nx, length) if axis == 1 else (nx, 30)
    span = n[axis]
    prob = workloads.problem(2, n, axis, 2.0 * (span - 3), 2.5, tuple(v / 2 + 0.25 for v in n), cp=0.375, n_surface=48,
                             n_periods=2, n_avg_periods=1, precision=precision, surface_radius=3.5, interface_d=2.0)
    prob.update(boundary="driven", wall_damping=0.99, source_amplitude=1e-3 / 0.0625)
    T = prob["period"]
    with wlb.Solver(prob) as s:
        s.init()
        s.step(T + 3)
        s.step(T - 3, sample=True)
        s.step(10, sample=True)
        F, (p1, u1) = s.force(), s.fields()
    with wlb.Solver(prob) as s:
        s.init()
        _one_step_launches(wlb, s, T + 3)
        F1 = _one_step_launches(wlb, s, T + 7)
        r1, w1 = s.fields()
    assert np.abs(p1).max() > 0
    assert np.array_equal(p1, r1) and np.array_equal(u1, w1) and np.array_equal(F, F1)
