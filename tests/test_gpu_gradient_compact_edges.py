"""The compact gradient of an HSGD step at the edges of its tiles and chunks against the FP64 oracle.

Shapes as for the dense gradient: 32 x 1 and 16 x 2 tiles and their ragged ends, short plane chunks, one to sixteen
warps a tile, images without interior samples, offsets that take the FP64 anchors; both storage types, both families, and
the batched step.  1e-5 on the gradient and relative 1e-5 on the loss, as there (the oracle gets the stored values).
"""
import numpy as np
import pytest
import torch

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu
TOL32 = 1e-5


@pytest.mark.parametrize("H,W,D,N,f", [(7, 33, 3, 2, None), (6, 48, 5, 1, None), (5, 40, 33, 2, None),
                                       (3, 3, 4, 1, None), (9, 64, 64, 2, None), (10, 97, 17, 3, None),
                                       (12, 70, 9, 2, 1500.0), (9, 31, 61, 2, 1500.0)])
@pytest.mark.parametrize("path", [0, 2, 4])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_compact_gradient_at_tile_and_chunk_edges(H, W, D, N, f, path, dtype):
    import paper_2307_03017_gb300 as rl
    sc = sg.make_scene(11, H, W, D, N, n_layers=(1, 2), novel="none", f=f)
    k = min(3, D)
    data = torch.from_numpy(sc.coarse_mpi).to(dtype).cuda()
    images = torch.from_numpy(sc.images).cuda()
    batch_loss = torch.zeros(1, device="cuda")
    ws = rl.workspace(N, D, H, W, k, dtype)
    rl.reallife_set_kernel_path(path)
    try:
        m = rl.make_mpi(data, sc.near, sc.far, sc.ref)
        S, mask = rl.reallife_select(m, k)
        loss, G = rl.reallife_loss_grad(m, images, sc.src, mask=mask, k=k)
        moved = data.clone()
        item = rl.BatchItem(rl.make_mpi(moved, sc.near, sc.far, sc.ref), images, sc.src, k, ws, clamp=False,
                            loss_out=batch_loss)
        rl.reallife_hsgd_step_batch(rl.BatchTable(1), [item])
        torch.cuda.synchronize()
    finally:
        rl.reallife_set_kernel_path(0)
    stored = data.float().cpu().numpy()
    at = S.cpu().numpy().astype(np.int64)[..., None]
    L_o, g_o, _ = oracle.loss_grad(stored, sc.near, sc.far, sc.ref, sc.src, sc.images)
    want = np.take_along_axis(g_o, at, axis=0)
    for v in (loss, batch_loss):
        assert abs(v.item() - L_o) <= 1e-5 * max(L_o, 1e-3)
    assert np.abs(G.cpu().numpy() - want).max() <= TOL32
    step = np.zeros_like(g_o)
    np.put_along_axis(step, np.broadcast_to(at, want.shape), want, axis=0)
    # the step's result is rounded to the storage type: half a BF16 step of values up to 2
    tol = TOL32 if dtype == torch.float32 else TOL32 + 2.0 ** -8
    assert np.abs(moved.float().cpu().numpy() - (stored - step)).max() <= tol
