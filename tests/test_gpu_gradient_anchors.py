"""Anchored gradients of few planes, whose blocks hold several tiles, against the FP64 oracle.

A short focal length and cameras turned by 33 degrees: an anchor shared by the tiles of a block lies
outside the image, where its ray is nearly parallel to the planes (positions 0.015 px off).  With an
anchor a tile, at most 8 pixels from its pixels, positions are off by d = 4e-6 px at most (the rays
spread the pixels by up to 1 / cos^2 60 = 4, so differences of 32 pixels at 1e-7).  Values change by at
most 1 a pixel and axis, and a voxel collects a few samples (about four) of gradients of at most 3, so
the gradient is off by 2 x 4 x 3 x d = 1e-4 at most.
"""
import math

import numpy as np
import pytest
import torch

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu
TOL = 1e-4
NEAR, FAR = 1.0, 100.0


def _scene(H, W, D, f):
    rng = np.random.default_rng(H * W + D)
    K = sg.intrinsics(W, H, f)
    src = []
    for deg, C in ((-33.5, (-3.0, 0.2, 0.1)), (33.5, (3.0, -0.2, 0.1)), (-14.1, (-3.0, 0.2, -0.1))):
        c, s = math.cos(math.radians(deg)), math.sin(math.radians(deg))
        R = np.array([[c, 0.0, s], [0.0, 1.0, 0.0], [-s, 0.0, c]])
        src.append(sg.Camera(K, R, -R @ np.array(C)))
    M = rng.uniform(0.0, 1.0, size=(D, H, W, 4)).astype(np.float32)
    M[..., 3] *= 0.7  # no plane hides all behind it
    images = rng.uniform(0.0, 1.0, size=(len(src), H, W, 3)).astype(np.float32)
    return sg.Camera(K, np.eye(3), np.zeros(3)), src, M, images


@pytest.mark.parametrize("H,W,D", [(24, 64, 1), (24, 64, 3), (24, 64, 4), (24, 64, 8), (13, 70, 4), (13, 97, 9), (24, 64, 17)])
@pytest.mark.parametrize("path", [0, 3, 4])
def test_anchored_gradient_of_few_planes(H, W, D, path):
    import paper_2307_03017_gb300 as rl
    ref, src, M, images = _scene(H, W, D, 64.0)
    k = min(3, D)
    data, imgs = torch.from_numpy(M).cuda(), torch.from_numpy(images).cuda()
    m = rl.make_mpi(data, NEAR, FAR, ref)
    rl.reallife_set_kernel_path(path)
    try:
        loss, G = rl.reallife_loss_grad(m, imgs, src)
        S, mask = rl.reallife_select(m, k)
        loss_s, Gs = rl.reallife_loss_grad(m, imgs, src, mask=mask, k=k)
        # one HSGD iteration alone and as a batch, which holds twice the tiles a block
        one, both = data.clone(), data.clone()
        la, lb = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
        rl.reallife_hsgd_step(rl.make_mpi(one, NEAR, FAR, ref), imgs, src, k, clamp=False, loss_out=la)
        ws = rl.workspace(len(src), D, H, W, k)
        rl.reallife_hsgd_step_batch(rl.BatchTable(1), [rl.BatchItem(rl.make_mpi(both, NEAR, FAR, ref), imgs, src, k, ws,
                                                                    clamp=False, loss_out=lb)])
        torch.cuda.synchronize()
    finally:
        rl.reallife_set_kernel_path(0)
    L_o, g_o, _ = oracle.loss_grad(M, NEAR, FAR, ref, src, images)
    kept = np.take_along_axis(g_o, S.cpu().numpy().astype(np.int64)[..., None], axis=0)
    step = np.zeros_like(g_o)
    np.put_along_axis(step, np.broadcast_to(S.cpu().numpy().astype(np.int64)[..., None], kept.shape), kept, axis=0)
    for v in (loss, loss_s, la, lb):
        assert abs(v.item() - L_o) <= TOL * L_o
    assert np.abs(G.cpu().numpy() - g_o).max() <= TOL
    assert np.abs(Gs.cpu().numpy() - kept).max() <= TOL
    for out in (one, both):
        assert np.abs(out.cpu().numpy() - (M - step)).max() <= TOL
