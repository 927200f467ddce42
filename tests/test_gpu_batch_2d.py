"""Batches of 2D lattices, several steps per launch: the same bits as one step
per launch for rows of every number of cells per lane, covered exactly by the
lanes or staged with a halo, chunks of one row block or several, and periods
that leave a remainder of two, four or six steps."""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

torch = pytest.importorskip("torch")
import workloads  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wlb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2404_02346_gb300 as W

    return W


# (nx, ny, wavelength): periods of 4 wavelength steps
ROWS = {
    "f32": [[(24, 32, 16.0), (64, 33, 16.5), (52, 35, 17.5)],             # two cells per lane
            [(96, 34, 17.0), (76, 39, 19.5), (92, 147, 24.5)],            # three (exact, halo), four
            [(128, 36, 18.0), (100, 95, 19.0), (140, 35, 17.5), (144, 34, 17.0)],  # four, five (exact, halo)
            [(192, 150, 25.0), (176, 35, 17.5), (208, 33, 16.5), (224, 39, 19.5)],  # six (exact, halo), seven
            [(244, 33, 16.5), (256, 35, 17.5), (248, 63, 21.0)],          # eight
            [(252, 34, 17.0), (128, 38, 19.0)]],                          # no room for a halo: two steps per launch
    "f16": [[(24, 32, 16.0), (64, 33, 16.5), (40, 147, 24.5)],
            [(96, 34, 17.0), (128, 35, 17.5), (112, 95, 19.0)],
            [(192, 39, 19.5), (144, 35, 17.5), (176, 150, 25.0)],
            [(208, 33, 16.5), (256, 35, 17.5), (240, 63, 21.0)]],
}


@pytest.mark.parametrize("precision,rows", [(p, r) for p in ROWS for r in ROWS[p]])
def test_batch_2d_steps_per_launch_bit_identical(wlb, precision, rows):
    probs = []
    for i, (nx, ny, lam) in enumerate(rows):
        c = (nx / 2 + 0.3 * i, (0.25 if i % 2 else 1.25) * lam % ny)  # stencils and arcs across the periodic edges too
        probs.append(workloads.problem(2, (nx, ny), 1, lam, 3.0 + 0.5 * i, c, cp=0.32, n_surface=(9, 200, 61, 33)[i],
                                       n_periods=3 + i, n_avg_periods=i if i < 3 else 0, precision=precision))
    with wlb.Batch(probs) as b:
        assert b.info().steps_per_launch == 2  # several
        F = b.run()
        again = b.run()
        b.set_two_step(False)
        one = b.run()
    assert np.all(np.isfinite(F))
    assert np.array_equal(F, one) and np.array_equal(F, again)
    assert np.any(F[1] != 0.0)
