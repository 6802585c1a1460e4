"""Renders of few planes, which are taken one at a time, and on both sides of the rule, against the FP64 oracle.

FP32 accumulation of at most 33 terms of at most 1: 1e-5, as for the other sizes (BF16 storage: the oracle gets the
stored values).
"""
import numpy as np
import pytest
import torch

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu


# f = None: offsets of a few pixels; f = 1500: FP64 anchors
@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 32, 33])
@pytest.mark.parametrize("f", [None, 1500.0])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_render_of_few_planes(D, f, dtype):
    import paper_2307_03017_gb300 as rl
    H, W = 21, 130
    sc = sg.make_scene(17, H, W, D, 3, n_layers=(1, 2), novel="none", f=f)
    data = torch.from_numpy(sc.coarse_mpi).to(dtype).cuda()
    data[..., 3] *= 0.6  # several planes show through
    rl.reallife_set_kernel_path(2)
    try:
        views = rl.reallife_render(rl.make_mpi(data, sc.near, sc.far, sc.ref), sc.src)
        torch.cuda.synchronize()
    finally:
        rl.reallife_set_kernel_path(0)
    stored = data.double().cpu().numpy()
    for got, cam in zip(views.cpu().numpy(), sc.src):
        assert np.abs(got - oracle.render(stored, sc.near, sc.far, sc.ref, cam)).max() <= 1e-5
