// rl_layout.h -- how reallife_gradient_volume divides its workspace (host arithmetic alone, so that
// it compiles and is checked without CUDA).
#pragma once
#include <stddef.h>

inline size_t rl_align256(size_t x) { return (x + 255) & ~(size_t)255; }

// The level MPI (levels >= 1), the selection and the view alpha weights [N][D][h][w] (largest at
// level 0), as byte offsets.
struct RLVolLayout {
    size_t Ml, S, A, total;
};

inline RLVolLayout rl_vol_layout(int N, int D, int H, int W, int k, size_t elt) {
    RLVolLayout L;
    size_t off = 0;
    L.Ml = off;
    if (H % 2 == 0 && W % 2 == 0) off += rl_align256((size_t)D * (H / 2) * (W / 2) * 4 * elt);
    L.S = off;
    off += rl_align256((size_t)k * H * W);
    L.A = off;
    off += rl_align256((size_t)N * D * H * W * sizeof(float));
    L.total = off;
    return L;
}

#define RL_NO_ROOM (~(size_t)0)

// Where the level's alphas alone [D][h][w] go, in the storage type of `elt` bytes: at level 0 in the
// place of the level MPI (unused there, and as large); above it behind the level's weights, which
// take at most a quarter of the room of level 0's.  Odd sizes have no room at level 0, and with
// N D H W <= 64 the rounding to 256 bytes leaves none above it: RL_NO_ROOM, and the weights are
// formed from the level MPI itself.
inline size_t rl_vol_alphas(const RLVolLayout& L, int N, int D, int H, int W, int level, size_t elt) {
    if (level == 0) return H % 2 == 0 && W % 2 == 0 ? L.Ml : RL_NO_ROOM;
    const size_t voxels = (size_t)D * (H >> level) * (W >> level);
    const size_t at = L.A + rl_align256((size_t)N * voxels * sizeof(float));
    return at + voxels * elt <= L.total ? at : RL_NO_ROOM;
}
