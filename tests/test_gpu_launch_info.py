"""wlb_get_launch_info and wlb_batch_steps_per_launch name the path that runs:
tiles of several steps, the two-step slab kernel, one step per launch, and the
row sweeps of 2D batches by row length."""
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


def _problem(n, precision, dim):
    axis = dim - 1
    return workloads.problem(dim, n, axis, float(n[axis]), 3.0, tuple(v / 2 for v in n), cp=0.4, n_surface=40,
                             n_periods=1, n_avg_periods=1, interface_d=1.0, precision=precision)


@pytest.mark.parametrize("n,precision,least,most,tiles", [
    ((192, 192), "f32", 2, 8, True),        # overlapped 2D tiles
    ((128, 128), "f64", 2, 8, True),
    ((40, 33, 36), "f32", 2, 2, True),      # 3D tiles: whole vectors, no multiple of 16 cells
    ((64, 32, 32), "f32", 2, 2, False),     # the slab kernel
    ((40, 33, 36), "f64", 1, 1, False),     # one step per launch
    ((41, 33, 36), "f32", 1, 1, False),
])
def test_launch_info_names_the_path(wlb, n, precision, least, most, tiles):
    with wlb.Solver(_problem(n, precision, len(n))) as s:
        i = s.launch_info()
    for sampled in range(2):
        assert least <= i.steps[sampled] <= most
        assert all((v > 0) == tiles for v in i.tile[sampled])
    assert (0 < i.sampler_blocks <= 40) if tiles else i.sampler_blocks == 0


@pytest.mark.parametrize("nx,precision,steps", [(96, "f32", 8), (128, "f16", 8), (192, "f32", 6), (256, "f32", 4),
                                                (208, "f16", 4), (252, "f32", 2), (128, "f64", 2)])
def test_batch_reports_its_steps_per_launch(wlb, nx, precision, steps):
    with wlb.Batch([_problem((nx, 32), precision, 2), _problem((64, 48), precision, 2)]) as b:
        assert b.steps_per_launch(0) == steps
        assert b.steps_per_launch(1) == (2 if steps == 2 else 8)
        b.set_two_step(False)
        assert b.steps_per_launch(0) == 1
        for i in (-1, 2):
            with pytest.raises(wlb.WlbError):
                b.steps_per_launch(i)
