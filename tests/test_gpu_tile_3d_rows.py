"""Two steps per launch in 3D tiles, on lattices that the planner gives to them:
FP32 and FP16 rows of whole 16-byte vectors (4 and 8 cells) that neither the slab
kernel (multiples of 16 cells, periodic) nor the one-step kernel's whole-warp rows
(multiples of 128 and 256 cells) take.  Fields and forces bit for bit against one
step per launch (wlb_average_noalloc).

Rows longer than 320 (FP32) and 640 (FP16) cells are split, so that tiles have
faces along x; others span the row and wrap around it.  Ragged last tiles (down
to one vector), a tile that spans z, objects across the periodic edges and across
tile edges, waves along every axis, walls and source sheet along every axis, and a
sphere of more than 16 boxes per axis, whose sampled steps go one per launch."""
import ctypes

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

LONG = {"f32": 320, "f16": 640}  # longest row whose tiles span it


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


def _compare(W, prob, boxes=True):
    T, nx = prob["period"], prob["n"][0]
    with W.Solver(prob) as s:
        i = s.launch_info()
        assert tuple(i.steps) == (2, 2 if boxes else 1) and (i.sampler_blocks > 0) == boxes
        assert (i.tile[0][0] < nx) == (nx > LONG[prob["precision"]])
        s.init()
        s.step(T + 5)
        for n in (1, T - 2, 8):
            s.step(n, sample=True)
        F, (p1, u1) = s.force(), s.fields()
        s.step(9)
        q1, v1 = s.fields()
        tile = tuple(i.tile[0])
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
    return tile


CASES = [
    # precision, n, axis, lam, R, d, center, N
    ("f32", (12, 9, 10), 2, 10.0, 1.0, 0.25, (4.25, 4.5, 8.75), 30),          # three vectors a row
    ("f32", (20, 26, 24), 2, 12.0, 3.0, 0.5, (0.125, 25.5, 3.0), 100),        # object across the edges
    ("f32", (36, 45, 64), 2, 32.0, 5.0, 4.0, (18.25, 22.5, 4.25), 500),
    ("f32", (132, 101, 66), 2, 22.0, 17.5, 4.0, (65.5, 50.0, 33.0), 300),     # a large sphere: many boxes
    ("f32", (324, 24, 32), 1, 24.0, 5.0, 0.5, (36.25, 2.5, 31.5), 300),       # nine x tiles, object on an edge
    ("f32", (516, 20, 26), 0, 12.0, 3.0, 0.5, (104.25, 10.0, 13.0), 200),     # ragged last x tile
    ("f32", (1028, 24, 24), 2, 24.0, 5.0, 0.5, (1027.5, 12.25, 3.0), 300),    # last x tile of one vector
    ("f16", (24, 9, 10), 2, 10.0, 1.0, 0.25, (4.25, 4.5, 8.75), 30),
    ("f16", (40, 26, 24), 2, 12.0, 3.0, 0.5, (39.875, 0.5, 3.0), 100),
    ("f16", (200, 41, 39), 0, 25.0, 8.0, 2.0, (3.5, 20.25, 19.0), 2000),      # dense points, wave along x
    ("f16", (648, 24, 32), 1, 24.0, 5.0, 0.5, (72.25, 2.5, 31.5), 300),
    ("f16", (1032, 24, 24), 2, 24.0, 5.0, 0.5, (1031.5, 12.25, 3.0), 300),    # ragged last x tile
]


@pytest.mark.parametrize("precision,n,axis,lam,R,d,center,N", CASES)
def test_tiles_equal_one_step_per_launch(wlb, precision, n, axis, lam, R, d, center, N):
    _compare(wlb, workloads.problem(3, n, axis, lam, R, center, cp=0.4, n_surface=N, n_periods=3, n_avg_periods=1,
                                    interface_d=d, precision=precision))


@pytest.mark.parametrize("precision,n", [("f32", (60, 2000, 9)), ("f16", (40, 4000, 8))])
def test_tile_that_spans_z(wlb, precision, n):
    tile = _compare(wlb, workloads.problem(3, n, 2, float(n[2]), 1.0, (30.25, 0.5, 7.75), cp=0.4, n_surface=40,
                                           n_periods=3, n_avg_periods=1, interface_d=0.25, precision=precision))
    assert tile[2] == n[2]


@pytest.mark.parametrize("precision,n,axis", [
    ("f32", (16, 24, 32), 2), ("f32", (32, 29, 24), 1), ("f32", (36, 24, 32), 0),
    ("f32", (336, 24, 32), 2), ("f32", (336, 24, 32), 0), ("f32", (528, 24, 32), 1),
    ("f16", (64, 29, 24), 1), ("f16", (40, 24, 32), 0), ("f16", (656, 24, 32), 2), ("f16", (656, 24, 32), 0),
])
def test_driven_tiles_equal_one_step_per_launch(wlb, precision, n, axis):
    span = n[axis]
    prob = workloads.problem(3, n, axis, 2.0 * (span - 3), 2.5, tuple(v / 2 + 0.25 for v in n), cp=0.375, n_surface=80,
                             n_periods=2, n_avg_periods=1, precision=precision, surface_radius=3.5, interface_d=1.0)
    prob.update(boundary="driven", wall_damping=0.99, source_amplitude=1e-3 / 0.0625)
    _compare(wlb, prob)


@pytest.mark.parametrize("precision,n,R", [("f32", (108, 108, 112), 47.0), ("f16", (104, 108, 112), 46.0)])
def test_sphere_of_too_many_boxes(wlb, precision, n, R):
    _compare(wlb, workloads.problem(3, n, 2, 56.0, R, tuple(v / 2 for v in n), cp=0.4, n_surface=200, n_periods=2,
                                    n_avg_periods=1, interface_d=0.25, precision=precision), boxes=False)
