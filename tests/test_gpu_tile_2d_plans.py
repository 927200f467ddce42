"""Several steps per launch on 2D lattices that are asserted to run in tiles
(wlb_get_launch_info): lattices narrower than a tile's box, which wraps onto
itself, objects and sampler boxes across both edges of the narrow axis, and
driven cavities with walls along x and along y in tiles.  Fields and forces bit
for bit against one step per launch (wlb_average_noalloc)."""
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
        i = s.launch_info()
        assert i.steps[0] > 1 and i.steps[1] > 1 and i.sampler_blocks > 0
        s.init()
        s.step(T + 5)
        for n in (1, T - 2, 7):
            s.step(n, sample=True)
        F, (p1, u1) = s.force(), s.fields()
        s.step(13)
        q1, v1 = s.fields()
    with W.Solver(prob) as s:
        s.init()
        _one_step_launches(W, s, T + 5)
        F1 = _one_step_launches(W, s, T + 6)
        r1, w1 = s.fields()
        _one_step_launches(W, s, 13)
        t1, x1 = s.fields()
    assert np.abs(p1).max() > 0 and np.all(np.isfinite(F)) and np.any(F != 0)
    assert np.array_equal(p1, r1) and np.array_equal(u1, w1)
    assert np.array_equal(q1, t1) and np.array_equal(v1, x1)
    assert np.array_equal(F, F1)


@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
@pytest.mark.parametrize("n,axis,lam,center,N", [
    ((12, 600), 1, 60.0, (11.5, 599.25), 8),      # 12 columns, boxes of up to 26
    ((12, 2000), 0, 12.0, (1.5, 1999.5), 200),
    ((900, 12), 1, 12.0, (0.25, 11.75), 200),
    ((57, 64), 1, 32.0, (30.0, 4.25), 1),         # odd rows, one point
])
def test_narrow_lattices(wlb, n, axis, lam, center, N, precision):
    _compare(wlb, workloads.problem(2, n, axis, lam, 3.0, center, cp=0.4, n_surface=N, n_periods=3, n_avg_periods=1,
                                    interface_d=0.5, precision=precision))


@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
@pytest.mark.parametrize("n,axis", [((203, 33), 0), ((403, 24), 0), ((16, 403), 1), ((33, 203), 1)])
def test_driven_cavities(wlb, n, axis, precision):
    prob = workloads.problem(2, n, axis, 2.0 * (n[axis] - 3), 2.5, tuple(v / 2 + 0.25 for v in n), cp=0.375,
                             n_surface=48, n_periods=2, n_avg_periods=1, precision=precision, surface_radius=3.5,
                             interface_d=1.0)
    prob.update(boundary="driven", wall_damping=0.99, source_amplitude=1e-3 / 0.0625)
    _compare(wlb, prob)
