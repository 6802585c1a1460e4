"""Gradients of shifted views where voxels that no pixel samples are not finite.

A thread holds two pixels of a column; with an odd height the last one's second pixel lies below the
image and samples a voxel row that no pixel of the image samples.
"""
import numpy as np
import pytest
import torch

import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("H,W,D,row", [(13, 64, 6, 7), (9, 33, 5, 3)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_voxels_that_no_pixel_samples_change_nothing(bad, H, W, D, row, dtype):
    import paper_2307_03017_gb300 as rl
    # the nearest plane is moved by -6.4 rows: pixel row H - 1 samples rows H - 8 and H - 7, so rows from H - 6 on
    # are free; the row below the image would sample the first of them
    assert row == H - 6
    sc = sg.make_scene(13, H, W, D, 2, n_layers=(1, 2), novel="none", f=64.0)
    src = [sg.Camera(sc.ref.K, np.eye(3), np.array([x, 0.1, 0.0])) for x in (-0.05, 0.02)]
    clean = torch.from_numpy(sc.coarse_mpi).to(dtype).cuda()
    clean[..., 3] *= 0.5  # every plane is seen
    clean[D - 1, row:] = 0
    holed = clean.clone()
    holed[D - 1, row:, :, 3] = bad
    images = torch.from_numpy(sc.images).cuda()
    rl.reallife_set_kernel_path(2)
    try:
        _, mask = rl.reallife_select(rl.make_mpi(clean, sc.near, sc.far, sc.ref), 3)
        want_l, want = rl.reallife_loss_grad(rl.make_mpi(clean, sc.near, sc.far, sc.ref), images, src, mask=mask, k=3)
        got_l, got = rl.reallife_loss_grad(rl.make_mpi(holed, sc.near, sc.far, sc.ref), images, src, mask=mask, k=3)
        torch.cuda.synchronize()
    finally:
        rl.reallife_set_kernel_path(0)
    assert want.abs().max().item() > 1e-3
    assert got_l.item() == want_l.item()
    # the same additions, in an order that differs from run to run
    assert bool(torch.isfinite(got).all())
    assert (got - want).abs().max().item() <= 1e-5
