"""The workspace of the gradient volume: no part reaches past the bytes that the library asks for.

The level's alphas lie behind the level's view weights, in the room of level 0's.  Both sizes are
rounded up to 256 bytes, so that the smallest volumes have no such room.
"""
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle
import scenegen as sg

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_03017_gb300", "csrc")
TOL32, TOL_BF16_LEVEL = 1e-5, 1e-2  # as in the volume's other tests: a coarse BF16 level is rounded on the GPU

PROGRAM = r"""
#include <stdio.h>
#include "rl_layout.h"
int main() {
    const int planes[] = {1, 2, 3, 4, 5, 8, 16, 33, 64};
    long with = 0, without = 0;
    for (int level = 0; level <= 4; ++level)
        for (int D : planes)
            for (int N = 1; N <= 16; ++N)
                for (int H = 1 << level; H <= 64; H += 1 << level)
                    for (int W = 1 << level; W <= 64; W += 1 << level)
                        for (size_t elt = 2; elt <= 4; elt += 2) {
                            const RLVolLayout L = rl_vol_layout(N, D, H, W, 1, elt);
                            const size_t at = rl_vol_alphas(L, N, D, H, W, level, elt);
                            if (at == RL_NO_ROOM) {
                                ++without;
                                continue;
                            }
                            ++with;
                            const size_t end = at + (size_t)D * (H >> level) * (W >> level) * elt;
                            // clear of what is live beside it: the selection and the view weights, the level MPI above level 0
                            const size_t weights = L.A + (size_t)N * D * (H >> level) * (W >> level) * 4;
                            if (at % 256 || end > L.total || (level ? at < weights : end > L.S)) {
                                printf("level %d D %d N %d H %d W %d elt %zu: %zu .. %zu of %zu\n", level, D, N, H, W,
                                       elt, at, end, L.total);
                                return 1;
                            }
                        }
    printf("%ld %ld\n", with, without);
    return 0;
}
"""


def test_alphas_lie_inside_the_workspace(tmp_path):
    src, exe = tmp_path / "layout.cpp", tmp_path / "layout"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    with_room, without = map(int, r.stdout.split())
    assert with_room > 0 and without > 0  # both outcomes are met


# the smallest volumes (no room), and the next larger ones (room)
@pytest.mark.gpu
@pytest.mark.parametrize("H,W,D,N,level", [(2, 2, 8, 1, 1), (2, 2, 8, 2, 1), (4, 4, 4, 1, 1), (4, 4, 4, 1, 2),
                                           (4, 4, 5, 1, 2), (4, 8, 8, 2, 1)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_nothing_is_written_behind_the_workspace(H, W, D, N, level, dtype):
    import paper_2307_03017_gb300 as rl
    sc = sg.make_scene(31, H, W, D, N, n_layers=(1, 2), novel="none")
    data = torch.from_numpy(sc.coarse_mpi).to(dtype).cuda()
    n = rl.reallife_gradient_volume_workspace_bytes(N, D, H, W, 2, dtype)
    room = torch.full((n + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    V, S = rl.reallife_gradient_volume(rl.make_mpi(data, sc.near, sc.far, sc.ref), torch.from_numpy(sc.images).cuda(),
                                       sc.src, 2, level, ws=room[:n])
    torch.cuda.synchronize()
    assert bool((room[n:] == 0xA5).all())
    S = S.cpu().numpy()
    Vo, So = oracle.gradient_volume(data.double().cpu().numpy(), sc.near, sc.far, sc.ref, sc.src, sc.images, 2, level,
                                    S_pin=S)
    assert np.array_equal(So, S)
    err = np.abs(V.double().cpu().numpy() - Vo)
    assert err[:3 * N].max() < TOL32
    assert err[3 * N:].max() < (TOL_BF16_LEVEL if dtype == torch.bfloat16 else TOL32)
