"""Two steps per launch in 3D tiles (the default path of 3D lattices that the
slab kernel does not take: odd rows, FP64, the driven cavity) against one step
per launch (wlb_average_noalloc): fields and forces bit for bit.  Lattices
smaller and larger than a tile (tiles that span an axis wrap around it), ragged
last tiles, objects across the periodic edges, waves along every axis, walls
and source sheet, one surface point, dense points, odd step counts."""
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


def _compare(W, prob):
    T = prob["period"]
    with W.Solver(prob) as s:
        assert s.info().steps_per_launch == 1  # not the slab kernel
        s.init()
        s.step(T + 5)
        for n in (1, T - 2, 8):
            s.step(n, sample=True)
        F, (p1, u1) = s.force(), s.fields()
        s.step(9)
        q1, v1 = s.fields()
    with W.Solver(prob) as s:
        s.init()
        _one_step_launches(W, s, T + 5)
        F1 = _one_step_launches(W, s, T + 7)
        r1, w1 = s.fields()
        _one_step_launches(W, s, 9)
        t1, x1 = s.fields()
    assert np.abs(p1).max() > 0 and np.all(np.isfinite(F)) and np.any(F != 0)
    assert np.array_equal(p1, r1) and np.array_equal(u1, w1)
    assert np.array_equal(q1, t1) and np.array_equal(v1, x1)
    assert np.array_equal(F, F1)


@pytest.mark.parametrize("precision", ["f32", "f16", "f64"])
@pytest.mark.parametrize("n,axis,lam,R,d,center,N", [
    ((9, 9, 10), 2, 10.0, 1.0, 0.25, (4.25, 4.5, 8.75), 30),         # a tile spans every axis
    ((23, 26, 24), 2, 12.0, 3.0, 0.5, (0.125, 25.5, 3.0), 100),      # object across the edges
    ((57, 45, 64), 2, 32.0, 5.0, 4.0, (28.25, 22.5, 4.25), 500),
    ((40, 33, 35), 1, 33.0, 4.0, 1.0, (20.0, 32.75, 17.0), 1),       # one point, wave along y
    ((100, 41, 39), 0, 25.0, 8.0, 2.0, (3.5, 20.25, 19.0), 2000),    # dense points, wave along x
    ((130, 101, 66), 2, 22.0, 17.5, 4.0, (65.5, 50.0, 33.0), 300),   # a large sphere: many boxes
])
def test_tiles_equal_one_step_per_launch(wlb, n, axis, lam, R, d, center, N, precision):
    _compare(wlb, workloads.problem(3, n, axis, lam, R, center, cp=0.4, n_surface=N, n_periods=3, n_avg_periods=1,
                                    interface_d=d, precision=precision))


@pytest.mark.parametrize("precision", ["f32", "f16", "f64"])
@pytest.mark.parametrize("n,axis", [((64, 24, 41), 2), ((33, 29, 24), 1), ((35, 24, 32), 0), ((128, 24, 30), 2)])
def test_driven_tiles_equal_one_step_per_launch(wlb, n, axis, precision):
    span = n[axis]
    prob = workloads.problem(3, n, axis, 2.0 * (span - 3), 2.5, tuple(v / 2 + 0.25 for v in n), cp=0.375, n_surface=80,
                             n_periods=2, n_avg_periods=1, precision=precision, surface_radius=3.5, interface_d=1.0)
    prob.update(boundary="driven", wall_damping=0.99, source_amplitude=1e-3 / 0.0625)
    _compare(wlb, prob)


def test_sphere_too_large_for_the_point_boxes(wlb):
    """More than 16 boxes per axis: sampled steps go one per launch, unsampled
    ones in tiles."""
    prob = workloads.problem(3, (107, 108, 112), 2, 56.0, 47.0, (53.5, 54.0, 56.0), cp=0.4, n_surface=200,
                             n_periods=2, n_avg_periods=1, interface_d=0.25)
    _compare(wlb, prob)
