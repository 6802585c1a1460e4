"""The gradient kernels at the edges of their tiles, chunks and dispatch rules against the FP64 oracle.

FP32 tolerance 1e-5 max-abs on the gradient and 1e-5 relative on the loss, as for the other sizes:
values and weights are at most 1 and a voxel collects at most a few taps a view.
"""
import numpy as np
import pytest
import torch

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu
TOL32 = 1e-5


@pytest.fixture(scope="module")
def rl():
    import paper_2307_03017_gb300 as rl
    yield rl
    rl.reallife_set_kernel_path(0)
    assert rl.reallife_device_status(clear=True) == 0


def _dev(a, dtype=torch.float32):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda").to(dtype)


# 32 x 1 and 16 x 2 tiles and their ragged ends, short plane chunks (D % 4), one to sixteen warps a
# tile, images too narrow for any interior sample, focal lengths whose offsets take the FP64 anchors
@pytest.mark.parametrize("H,W,D,N,f", [(7, 33, 3, 2, None), (6, 48, 5, 1, None), (5, 40, 33, 2, None),
                                       (3, 3, 4, 1, None), (9, 64, 64, 2, None), (10, 97, 17, 3, None),
                                       (12, 70, 9, 2, 1500.0), (9, 31, 61, 2, 1500.0)])
@pytest.mark.parametrize("path", [0, 2, 4])
def test_gradient_at_tile_and_chunk_edges(rl, H, W, D, N, f, path):
    sc = sg.make_scene(11, H, W, D, N, n_layers=(1, 2), novel="none", f=f)
    rl.reallife_set_kernel_path(path)
    try:
        m = rl.make_mpi(_dev(sc.coarse_mpi), sc.near, sc.far, sc.ref)
        loss, G = rl.reallife_loss_grad(m, _dev(sc.images), sc.src)
    finally:
        rl.reallife_set_kernel_path(0)
    L_o, g_o, _ = oracle.loss_grad(sc.coarse_mpi, sc.near, sc.far, sc.ref, sc.src, sc.images)
    assert abs(loss.item() - L_o) <= 1e-5 * max(L_o, 1e-3)
    assert np.abs(G.cpu().numpy() - g_o).max() <= TOL32


# views that are pure shifts share taps between two rows: shifts beyond the image, taps left of and
# above the first voxel of all (plane 0, column and row -1), odd widths and heights, a single plane
@pytest.mark.parametrize("H,W,D,f", [(9, 64, 5, None), (7, 33, 33, None), (12, 97, 50, 300.0), (6, 40, 1, None)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_gradient_of_shifted_views(rl, H, W, D, f, dtype):
    sc = sg.make_scene(12, H, W, D, 8, n_layers=(1, 2), src_poses="grid4x2", novel="none", f=f)
    rl.reallife_set_kernel_path(2)
    try:
        m = rl.make_mpi(_dev(sc.coarse_mpi, dtype), sc.near, sc.far, sc.ref)
        loss, G = rl.reallife_loss_grad(m, _dev(sc.images), sc.src)
        k = min(3, D)
        S, mask = rl.reallife_select(m, k)
        loss_s, Gs = rl.reallife_loss_grad(m, _dev(sc.images), sc.src, mask=mask, k=k)
    finally:
        rl.reallife_set_kernel_path(0)
    stored = m.data.float().cpu().numpy()
    L_o, g_o, _ = oracle.loss_grad(stored, sc.near, sc.far, sc.ref, sc.src, sc.images)
    assert abs(loss.item() - L_o) <= 1e-5 * max(L_o, 1e-3)
    assert np.abs(G.cpu().numpy() - g_o).max() <= TOL32
    assert abs(loss_s.item() - L_o) <= 1e-5 * max(L_o, 1e-3)
    want = np.take_along_axis(g_o, S.cpu().numpy().astype(np.int64)[..., None], axis=0)
    assert np.abs(Gs.cpu().numpy() - want).max() <= TOL32


# the two gradient families a batch may take: the automatic rule's small and large batches
@pytest.mark.parametrize("H,W,n", [(24, 34, 3), (256, 352, 3)])
def test_batch_family_by_size_equals_single_steps(rl, H, W, n):
    scenes = [sg.make_scene(20 + i, H, W, 6 + i, 2, n_layers=(1, 2), novel="none") for i in range(n)]
    items, want = [], []
    for sc in scenes:
        ws = rl.workspace(2, sc.D, H, W, 3)
        one, both = _dev(sc.coarse_mpi), _dev(sc.coarse_mpi)
        la, lb = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
        images = _dev(sc.images)
        rl.reallife_hsgd_step(rl.make_mpi(one, sc.near, sc.far, sc.ref), images, sc.src, 3, loss_out=la)
        items.append(rl.BatchItem(rl.make_mpi(both, sc.near, sc.far, sc.ref), images, sc.src, 3, ws, loss_out=lb))
        want.append((one, la, both, lb))
    rl.reallife_hsgd_step_batch(rl.BatchTable(n), items)
    for one, la, both, lb in want:
        assert (one - both).abs().max().item() <= TOL32
        assert abs(la.item() - lb.item()) <= 1e-5 * max(1.0, abs(la.item()))
