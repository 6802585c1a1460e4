"""Gradients on both sides of the dispatch rule agree with each other, whichever kernel the rule takes.

From 2^19 pixel-views on the rule goes by the planes (the share of the plane-parallel kernel's warps that hold
some), so plane counts on both sides of it are taken, dense and compact, shifted and rotated views.  All values are
at most 1, a voxel collects a few taps a view: 1e-5 between two FP32 evaluations, as against the oracle.
"""
import pytest
import torch

import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [5, 17, 33, 42, 48])
@pytest.mark.parametrize("poses", ["random", "grid4x2"])
@pytest.mark.parametrize("H,W,N,dtype", [(361, 500, 3, torch.float32), (300, 447, 8, torch.bfloat16)])
def test_automatic_gradient_equals_both_families(D, poses, H, W, N, dtype):
    import paper_2307_03017_gb300 as rl
    assert H * W * N >= 1 << 19 and (H * W * N >= 1 << 20) == (N == 8)
    sc = sg.make_scene(61, 12, 16, D, N, n_layers=(1, 2), src_poses=poses, novel="none")
    K = sg.intrinsics(W, H)
    ref, src = sg.Camera(K, sc.ref.R, sc.ref.t), [sg.Camera(K, c.R, c.t) for c in sc.src]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(D)
    data = torch.rand((D, H, W, 4), generator=gen, device="cuda")
    data[..., 3] *= 0.3
    m = rl.make_mpi(data.to(dtype), sc.near, sc.far, ref)
    images = torch.rand((N, H, W, 3), generator=gen, device="cuda")
    _, mask = rl.reallife_select(m, 3)
    out = {}
    for path in (0, 2, 3):
        rl.reallife_set_kernel_path(path)
        try:
            out[path] = (*rl.reallife_loss_grad(m, images, src), *rl.reallife_loss_grad(m, images, src, mask=mask, k=3))
            torch.cuda.synchronize()
        finally:
            rl.reallife_set_kernel_path(0)
    for path in (2, 3):
        for got, want in zip(out[0], out[path]):
            scale = max(1.0, want.item()) if want.numel() == 1 else 1.0
            assert (got - want).abs().max().item() <= 1e-5 * scale
