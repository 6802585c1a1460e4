"""Gradients of images wider than the plane-parallel kernel's grid of 16-pixel tiles (1,048,560 pixels).

Automatic dispatch sends them to the per-pixel kernel, whose tiles are 32 pixels wide.  Two rows and a width
just above a multiple of 32 are a shape for which 16 x 2 tiles would be the fewer.  FP32 tolerance 1e-5 as
for the other sizes.
"""
import numpy as np
import pytest
import torch

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [16 * 65535, 16 * 65535 + 17])
def test_gradient_of_a_very_wide_image(W):
    import paper_2307_03017_gb300 as rl
    H, D, k, f = 2, 17, 2, 300.0
    rng = np.random.default_rng(W)
    ref = sg.Camera(sg.intrinsics(W, H, f), np.eye(3), np.zeros(3))
    # a lens of 300 px and a depth offset of 1e-5: offsets up to 5 px at the ends of the image
    src = [sg.Camera(ref.K, np.eye(3), np.array([0.004, 0.001, 1e-5]))]
    M = rng.uniform(0.0, 1.0, size=(D, H, W, 4)).astype(np.float32)
    M[..., 3] *= 0.3
    images = rng.uniform(0.0, 1.0, size=(1, H, W, 3)).astype(np.float32)
    m = rl.make_mpi(torch.from_numpy(M).cuda(), 1.0, 100.0, ref)
    loss, G = rl.reallife_loss_grad(m, torch.from_numpy(images).cuda(), src)
    S, mask = rl.reallife_select(m, k)
    loss_s, Gs = rl.reallife_loss_grad(m, torch.from_numpy(images).cuda(), src, mask=mask, k=k)
    torch.cuda.synchronize()
    oracle.set_threads(True)
    try:
        L_o, g_o, _ = oracle.loss_grad(M, 1.0, 100.0, ref, src, images)
    finally:
        oracle.set_threads(False)
    for v in (loss, loss_s):
        assert abs(v.item() - L_o) <= 1e-5 * L_o
    G, Gs = G.cpu().numpy(), Gs.cpu().numpy()
    kept = np.take_along_axis(g_o, S.cpu().numpy().astype(np.int64)[..., None], axis=0)
    # FP32 positions: 1.2e-7 of the offset, and of the pixel's distance from the centre over the lens
    assert np.abs(G - g_o).max() <= 1e-5
    assert np.abs(Gs - kept).max() <= 1e-5
