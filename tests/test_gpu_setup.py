"""The setup kernels where their fast paths end: cells classified from FP32
distances away from the band and in FP64 near it (large radii, sharp and wide
bands, centres at the box edge), rows that are and are not whole 16-byte
vectors, waves along every axis (tables along the wave), and batches (all
lattices in one set of launches) against single handles."""
import numpy as np
import pytest

import oracle
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


# p1 at t = 0 is c^2 times the sum of q populations rounded to the storage
# type: q + 2 roundings of values up to p_a / c^2, i.e. (q + 2) eps p_a / 2.
EPS = {"f32": 2.0 ** -24, "f64": 2.0 ** -53, "f16": 2.0 ** -11}


@pytest.mark.parametrize("precision", ["f32", "f64", "f16"])
@pytest.mark.parametrize("dim,n,axis,lam,R,d,center", [
    (3, (64, 48, 40), 2, 40.0, 6.0, 4.0, (31.75, 24.25, 5.0)),
    (3, (65, 47, 32), 0, 65.0, 9.5, 0.25, (0.125, 46.875, 16.0)),    # odd rows, wave along x, object across the edges
    (3, (30, 64, 33), 1, 16.0, 4.0, 1.0, (29.5, 0.0, 32.5)),
    (3, (160, 96, 96), 2, 48.0, 38.0, 4.0, (80.25, 47.5, 90.0)),      # a large object: many inner cells
    (2, (130, 64, 1), 1, 64.0, 8.0, 4.0, (129.0, 60.5)),
    (2, (33, 41, 1), 0, 33.0, 5.0, 2.0, (-3.25, 44.5)),              # centre outside the box: one image
])
def test_classes_points_and_initial_wave(wlb, precision, dim, n, axis, lam, R, d, center):
    prob = workloads.problem(dim, n, axis, lam, R, center, cp=0.4, n_surface=73, n_periods=1, n_avg_periods=1,
                             interface_d=d, antinode=0.3, precision=precision)
    with wlb.Solver(prob) as s:
        s.init()
        assert np.array_equal(s.mask(), oracle.mask(prob))
        assert np.array_equal(s.surface(), oracle.run(dict(prob, n_steps=prob["period"]))["points"])
        p1, u1 = s.fields()
        s.init()  # a second setup of the same handle gives the same state
        q1, v1 = s.fields()
    assert np.array_equal(p1, q1) and np.array_equal(u1, v1)
    k = 2 * np.pi / prob["wavelength"]
    wave = prob["p_a"] * np.cos(k * (np.arange(n[axis]) - prob["antinode"]))
    shape = [1, 1, 1]
    shape[2 - axis] = -1
    q = 2 * dim + 1
    bound = (q + 2) * EPS[precision] * prob["p_a"]
    assert np.abs(p1 - wave.reshape(shape)).max() <= bound + 1e-15 * prob["p_a"]
    assert np.abs(u1).max() <= bound / prob["c0"] + 1e-30


@pytest.mark.parametrize("precision", ["f32", "f16"])
def test_batch_setup_matches_single_handles(wlb, precision):
    """Uneven lattices and point counts set up together: the forces of a run
    equal each lattice's own, also on a second run of the batch."""
    specs = [((48, 40, 32), 16.0, 3.0, 1), ((96, 24, 48), 24.0, 3.5, 211), ((64, 64, 32), 32.0, 5.0, 64)]
    probs = [workloads.problem(3, n, 2, lam, R, (n[0] / 2 + 0.25, n[1] / 2 - 0.5, lam / 8), cp=0.35, n_surface=N,
                               n_periods=2, n_avg_periods=1, precision=precision) for n, lam, R, N in specs]
    with wlb.Batch(probs) as b:
        F, F2 = b.run(), b.run()
    assert np.array_equal(F, F2)
    for f, p in zip(F, probs):
        with wlb.Solver(p) as s:
            assert np.array_equal(f, s.run())
