"""Losses beyond the range of FP32: infinite, as the sum of squares is, and never NaN."""
import math

import numpy as np
import pytest
import torch

import scenegen as sg

pytestmark = pytest.mark.gpu


# image values of 1e20 overflow every square; 3e18 keeps each pixel's sum of squares (3 x 9e36) and a
# tile's (32 to 128 pixels: up to 3.5e39 for the per-pixel family) near or beyond FP32's 3.4e38, and a
# value of 5e17 keeps a tile's sum finite (128 x 7.5e35 = 1e38) while the image's 3072 pixels exceed it
@pytest.mark.parametrize("value", [1e20, 3e18, 5e17])
@pytest.mark.parametrize("path", [0, 2])
@pytest.mark.parametrize("poses", ["random", "grid4x2"])
def test_overflowing_loss_is_infinite(value, path, poses):
    import paper_2307_03017_gb300 as rl
    H, W, D, N, k = 48, 64, 8, 2, 3
    sc = sg.make_scene(41, H, W, D, N, n_layers=(1, 2), src_poses=poses, novel="none")
    images = torch.full((N, H, W, 3), value, device="cuda")
    coarse = torch.from_numpy(sc.coarse_mpi).cuda()
    ws = rl.workspace(N, D, H, W, k)
    losses = torch.zeros(2, device="cuda")
    rl.reallife_set_kernel_path(path)
    try:
        dense, _ = rl.reallife_loss_grad(rl.make_mpi(coarse, sc.near, sc.far, sc.ref), images, sc.src)
        rl.reallife_hsgd_step(rl.make_mpi(coarse.clone(), sc.near, sc.far, sc.ref), images, sc.src, k,
                              loss_out=losses[:1], ws=ws)
        m = rl.make_mpi(coarse.clone(), sc.near, sc.far, sc.ref)
        rl.reallife_hsgd_step_batch(rl.BatchTable(1), [rl.BatchItem(m, images, sc.src, k, ws, loss_out=losses[1:])])
        torch.cuda.synchronize()
    finally:
        rl.reallife_set_kernel_path(0)
    want = N * H * W * 3 * (np.float64(value) ** 2) * 0.5 / N
    assert want > np.finfo(np.float32).max
    got = [dense.item(), *losses.tolist()]
    assert all(math.isinf(v) and v > 0 for v in got), got
