// grad.cu -- fused warp + composite + photometric residual + exact adjoint (one launch for
// all source views), the render backward used by autograd, and the loss reduction.
//
// Per view pixel q (one thread), with T_d = prod_{j>d}(1 - alpha_j) (Eq. eq_over):
//   pass 1, d = D-1 .. 0:  m_d = bilinear(M[d], p_d(q)); T_d of each group's nearest plane ->
//                           shared memory; C += T_d alpha_d c_d; T *= (1 - alpha_d)
//   residual:               r = (C - I(q)) / N  (loss mode; L = 1/(2N) sum |C - I|^2; I the
//                           level image: given at the level's resolution, img_level 0, or formed
//                           on the fly from its 2^l x 2^l full-resolution pixels)
//                           or r = dL/dC given by the caller (backward mode)
//   pass 2, d = 0 .. D-1:  dL/dc_d = T_d alpha_d r;  dL/dalpha_d = T_d <c_d - B_d, r>,
//                           B_d the composite of the planes below d (B_0 = 0,
//                           B_{d+1} = c_d alpha_d + (1 - alpha_d) B_d);
//                           the bilinear transpose adds w_tap * dL/dm_d to the 4 taps.
// Sparse mode adds only into voxels kept by the selection (Sec. 3.3): the slot map
// slots[d][y][x] gives the compact slot of a kept voxel (its rank among the kept planes of
// the pixel) or RL_SLOT_NONE.  No division by (1 - alpha).
//
// What bounds it: L1 wavefronts (two gathers a sample and the reductions onto the kept taps) and
// the latency of the gathers.  Warps whose samples all lie inside leave out the border tests.  With
// many planes both passes take them in pairs, whose loads are in flight together, and pass 2 forms
// T_d within a pair from the pair's stored one: half the shared memory, so that a launch of 64
// planes keeps 32 warps an SM instead of 24, and its L1.  Views that are pure shifts of the reference
// (display and camera grids) have the same offset and weights at every pixel of a plane: a block
// forms them once in FP64 and reads them from shared memory.  1920x1080, D = 64, 8 views, BF16:
// 6.69 ms as shifts, 8.23 ms with anchored coordinates (one plane at a time 11.56 ms, groups of four
// 10.8 ms; at the start, with border tests in every sample and a fenced loss reduction at the end of
// every block, 12.9 ms).  Issue bound (78%): of the 197 instructions a sample left as shifts, 32
// widen BF16, 16 blend and about 40 are the reductions of the taps.
#include <type_traits>

#include "rl_internal.h"

namespace {

constexpr int kGradBX = 32, kGradBY = 4, kGradThreads = kGradBX * kGradBY;
constexpr int kGroup = 2;          // planes whose samples are held together (grad_group, the batch)
constexpr int kGradMinBlocks = 8;  // resident blocks the registers must then allow

// How the taps of a sample are formed.
constexpr int kPlain = 0, kAnchored = 1, kShifts = 2;

// Views that are pure shifts of the reference: the offset p - q of plane d, the same for all pixels,
// split in FP64 into an integer and a fraction.
struct ShiftTable {
    float4 w[RL_DEV_MAX_PLANES];   // the taps' weights
    int off[RL_DEV_MAX_PLANES];    // iy W + ix
    int ix[RL_DEV_MAX_PLANES], iy[RL_DEV_MAX_PLANES];
    float fx[RL_DEV_MAX_PLANES], fy[RL_DEV_MAX_PLANES];

    __device__ __forceinline__ RLTaps taps(int d, int qx, int qy) const {
        RLTaps t;
        t.ok = ix[d] != RL_PLANE_NONE;
        t.x0 = qx + ix[d];
        t.y0 = qy + iy[d];
        t.fx = fx[d];
        t.fy = fy[d];
        return t;
    }
    // All four taps inside the plane.  The integer offset is monotone in d, so what holds for two
    // planes holds for those between them.
    __device__ __forceinline__ bool inside(int d, int qx, int qy, int H, int W) const {
        return ix[d] != RL_PLANE_NONE && (unsigned)(qx + ix[d]) < (unsigned)(W - 1) &&
               (unsigned)(qy + iy[d]) < (unsigned)(H - 1);
    }
};

struct ShiftTap {
    unsigned idx;  // voxel of the top-left tap within its plane
    float4 w;
};

// Fills S for view `view`; every thread of the block calls it.
__device__ __forceinline__ void shift_build(ShiftTable* S, const RLViews& V, int view, int D, int W, int tid) {
    if (tid < D) {
        const RLViewParam64& P = V.v64[view];
        const double rho = V.rho64[tid];
        const double kx = P.dcx + rho * (P.fxr * P.C[0]), ky = P.dcy + rho * (P.fyr * P.C[1]);
        const bool ok = fabs(kx) < 1e9 && fabs(ky) < 1e9;
        const double flx = floor(kx), fly = floor(ky);
        S->ix[tid] = ok ? (int)flx : RL_PLANE_NONE;
        S->iy[tid] = ok ? (int)fly : RL_PLANE_NONE;
        S->off[tid] = ok ? (int)((unsigned)(int)fly * (unsigned)W + (unsigned)(int)flx) : 0;
        S->fx[tid] = (float)(kx - flx);
        S->fy[tid] = (float)(ky - fly);
        S->w[tid] = rl_weights(S->fx[tid], S->fy[tid]);
    }
    __syncthreads();
}

// One block's tile of 32 x 4 view pixels of one view.  bid / nblocks index the block among
// the launch's (or the batch item's) blocks for the loss partials.
template <typename Tm, int GROUP, bool SPARSE, bool LOSS, int MODE>
__device__ __forceinline__ void grad_tile(const Tm* __restrict__ M, int D, int H, int W, const RLViews& views, int view,
                                          int qx, int qy, int tid, float* __restrict__ sT,
                                          const float* __restrict__ images, int img_level,
                                          const float* __restrict__ grad_out, const uint8_t* __restrict__ slots,
                                          float* __restrict__ G, float inv_n, float* __restrict__ partials,
                                          unsigned bid, unsigned nblocks) {
    constexpr bool ANCH = MODE == kAnchored, SHIFT = MODE == kShifts;
    float lsum = 0.f;
    __shared__ RLAnchor sA;  // the tile's anchor: its centre pixel
    __shared__ ShiftTable sS;
    if (SHIFT) shift_build(&sS, views, view, D, W, tid);
    if (ANCH)
        rl_anchor_build(&sA, views, view, (qx & ~(kGradBX - 1)) + kGradBX / 2, qy - qy % kGradBY + kGradBY / 2, D,
                        W, tid, kGradThreads);
    const unsigned act = __ballot_sync(0xffffffffu, qx < W && qy < H);
    if (qx < W && qy < H) {
        RLPixWarp<ANCH> w;
        if constexpr (!SHIFT) w = rl_pix_warp<ANCH>(sA, views.v[view], qx, qy);
        const size_t plane = (size_t)H * W * 4;
        const unsigned hw = (unsigned)(H * W);
        const unsigned base = SHIFT ? (unsigned)(qy * W + qx) : rl_fast_base(qx, qy, W);
        // warps whose samples of every plane lie inside it skip the border tests; with shifts the whole
        // tile row moves as one, and every kWalk planes are tested by themselves
        constexpr int kWalk = 8, kPer = kWalk / GROUP;
        const int n_chunks = (D + kWalk - 1) / kWalk;
        unsigned chunks = 0u;
        if constexpr (SHIFT) {
            for (int c = 0; c < n_chunks; ++c) {
                const int d0 = c * kWalk, d1 = min(d0 + kWalk, D) - 1;
                if (__all_sync(act, sS.inside(d0, qx, qy, H, W) && sS.inside(d1, qx, qy, H, W))) chunks |= 1u << c;
            }
        } else {
            chunks = __all_sync(act, rl_chunk_inside<ANCH>(w, sA, views, 0, D - 1, qx, qy, H, W)) ? 1u : 0u;
        }
        // the sample of plane d: top-left voxel and weights (inside), or footprint (anywhere)
        const auto tap_inside = [&](int d) {
            if constexpr (SHIFT) return ShiftTap{base + (unsigned)sS.off[d], sS.w[d]};
            else return rl_fast_tap<ANCH>(w, sA, d, views.rho[d], base, W);
        };
        const auto weights = [](const auto& t) {
            if constexpr (SHIFT) return t.w;
            else return rl_weights(t.fx, t.fy);
        };
        const auto tap_any = [&](int d) {
            if constexpr (SHIFT) return sS.taps(d, qx, qy);
            else return w.taps(sA, d, views.rho[d], qx, qy);
        };
        const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
        const int groups = (D + GROUP - 1) / GROUP;
        float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
        // the two kinds take separate loops: a branch in every group costs 15%
        const auto pass1 = [&](auto inside, int first, int end) {
#pragma unroll 1
            for (int j = end - 1; j >= first; --j) {
                float4 m[GROUP];
#pragma unroll
                for (int i = GROUP - 1; i >= 0; --i) {
                    const int d = j * GROUP + i, dc = GROUP == 1 ? d : min(d, D - 1);
                    if constexpr (decltype(inside)::value) {
                        const auto t = tap_inside(dc);
                        m[i] = RL_IN((long long)t.idx + W + 1, hw)
                                   ? rl_sample_at(M, (unsigned)dc * hw + t.idx, W, weights(t)) : none;
                    } else {
                        m[i] = rl_sample_fast(M + dc * plane, H, W, tap_any(dc));
                    }
                    if (GROUP > 1 && d >= D) m[i] = none;  // beyond the last plane
                }
                sT[j * kGradThreads + tid] = T;
#pragma unroll
                for (int i = GROUP - 1; i >= 0; --i) {
                    const float a = T * m[i].w;
                    c0 = fmaf(a, m[i].x, c0);
                    c1 = fmaf(a, m[i].y, c1);
                    c2 = fmaf(a, m[i].z, c2);
                    T = T * (1.f - m[i].w);
                }
            }
        };
        if constexpr (SHIFT) {
#pragma unroll 1
            for (int c = n_chunks - 1; c >= 0; --c) {
                if ((chunks >> c) & 1u) pass1(std::true_type(), c * kPer, min((c + 1) * kPer, groups));
                else pass1(std::false_type(), c * kPer, min((c + 1) * kPer, groups));
            }
        } else if (chunks) {
            pass1(std::true_type(), 0, groups);
        } else {
            pass1(std::false_type(), 0, groups);
        }
        float r0, r1, r2;
        if (LOSS) {
            // source image at this level: mean of the 2^l x 2^l full-resolution block
            const int s = 1 << img_level;
            const int Wf = W << img_level, Hf = H << img_level;
            const float* img = images + (size_t)view * Hf * Wf * 3;
            float i0 = 0.f, i1 = 0.f, i2 = 0.f;
            for (int yy = 0; yy < s; ++yy)
                for (int xx = 0; xx < s; ++xx) {
                    const float* px = img + ((size_t)(qy * s + yy) * Wf + (qx * s + xx)) * 3;
                    i0 += __ldg(px);
                    i1 += __ldg(px + 1);
                    i2 += __ldg(px + 2);
                }
            const float inv_area = 1.f / (float)(s * s);
            // the image mean is rounded on its own (as the level images of the pyramid pass are)
            const float e0 = c0 - __fmul_rn(i0, inv_area), e1 = c1 - __fmul_rn(i1, inv_area),
                        e2 = c2 - __fmul_rn(i2, inv_area);
            lsum = fmaf(e0, e0, fmaf(e1, e1, e2 * e2));
            r0 = e0 * inv_n;
            r1 = e1 * inv_n;
            r2 = e2 * inv_n;
        } else {
            const float* go = grad_out + (((size_t)view * H + qy) * W + qx) * 3;
            r0 = __ldg(go);
            r1 = __ldg(go + 1);
            r2 = __ldg(go + 2);
        }
        float b0 = 0.f, b1 = 0.f, b2 = 0.f;
        const unsigned ng = views.gplanes ? (unsigned)views.gplanes : (unsigned)D;  // checked in debug builds
        const auto pass2 = [&](auto inside, int first, int end) {
#pragma unroll 1
            for (int j = first; j < end; ++j) {
                float4 m[GROUP];
                float Td[GROUP];
                unsigned word[GROUP];
                decltype(tap_inside(0)) tap[GROUP];
#pragma unroll
                for (int i = GROUP - 1; i >= 0; --i) {
                    const int d = j * GROUP + i, dc = GROUP == 1 ? d : min(d, D - 1);
                    if constexpr (decltype(inside)::value) {
                        tap[i] = tap_inside(dc);
                        const unsigned e = (unsigned)dc * hw + tap[i].idx;
                        m[i] = none;
                        word[i] = 0xFFFFFFFFu;
                        if (RL_IN((long long)tap[i].idx + W + 1, hw)) {
                            if (SPARSE) word[i] = rl_slot_word(slots, e, W);
                            m[i] = rl_sample_at(M, e, W, weights(tap[i]));
                        }
                    } else {
                        m[i] = rl_sample_fast(M + dc * plane, H, W, tap_any(dc));
                    }
                    if (GROUP > 1 && d >= D) m[i] = none;
                }
                float Tg = sT[j * kGradThreads + tid];
#pragma unroll
                for (int i = GROUP - 1; i >= 0; --i) {
                    Td[i] = Tg;
                    Tg = Tg * (1.f - m[i].w);
                }
#pragma unroll
                for (int i = 0; i < GROUP; ++i) {
                    const int d = j * GROUP + i;
                    if (Td[i] != 0.f && d < D) {
                        const float gc = Td[i] * m[i].w;
                        const float4 g =
                            make_float4(gc * r0, gc * r1, gc * r2,
                                        Td[i] * fmaf(m[i].x - b0, r0, fmaf(m[i].y - b1, r1, (m[i].z - b2) * r2)));
                        if constexpr (decltype(inside)::value) {
                            // a pair forms its taps again (they cost registers); a single plane keeps them
                            const auto t = GROUP == 1 ? tap[i] : tap_inside(d);
                            rl_scatter_at<SPARSE>(G, word[i], (unsigned)d, t.idx, (unsigned)d * hw + t.idx, hw, W,
                                                  weights(t), g, ng);
                        } else {
                            const RLTaps t = tap_any(d);
                            if (t.ok) rl_scatter<SPARSE>(G, slots, (unsigned)d, hw, H, W, t, g, ng);
                        }
                    }
                    const float om = 1.f - m[i].w;
                    b0 = fmaf(m[i].x, m[i].w, om * b0);
                    b1 = fmaf(m[i].y, m[i].w, om * b1);
                    b2 = fmaf(m[i].z, m[i].w, om * b2);
                }
            }
        };
        if constexpr (SHIFT) {
#pragma unroll 1
            for (int c = 0; c < n_chunks; ++c) {
                if ((chunks >> c) & 1u) pass2(std::true_type(), c * kPer, min((c + 1) * kPer, groups));
                else pass2(std::false_type(), c * kPer, min((c + 1) * kPer, groups));
            }
        } else if (chunks) {
            pass2(std::true_type(), 0, groups);
        } else {
            pass2(std::false_type(), 0, groups);
        }
    }
    if (LOSS) {
        __shared__ float red[kGradThreads / 32];
        lsum = rl_warp_sum(lsum);
        if ((tid & 31) == 0) red[tid >> 5] = lsum;
        __syncthreads();
        if (tid == 0) {
            float blk = 0.f;
            for (int j = 0; j < kGradThreads / 32; ++j) blk += red[j];
            if (RL_IN(bid, nblocks)) partials[bid] = blk;
        }
    }
}

template <typename Tm, int GROUP, bool SPARSE, bool LOSS, int MODE>
__global__ void __launch_bounds__(kGradThreads, GROUP == 1 ? 10 : kGradMinBlocks)
k_grad(const Tm* __restrict__ M, int D, int H, int W, const __grid_constant__ RLViews views,
       const float* __restrict__ images, int img_level, const float* __restrict__ grad_out,
       const uint8_t* __restrict__ slots, float* __restrict__ G, float inv_n, float* __restrict__ partials) {
    extern __shared__ float sT[];  // [ceil(D / GROUP)][kGradThreads]
    // view-fastest block order: the N views of a tile run together and share M through L2
    grad_tile<Tm, GROUP, SPARSE, LOSS, MODE>(M, D, H, W, views, blockIdx.x, blockIdx.y * kGradBX + threadIdx.x,
                                blockIdx.z * kGradBY + threadIdx.y, threadIdx.y * kGradBX + threadIdx.x, sT, images,
                                img_level, grad_out, slots, G, inv_n, partials,
                                blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z),
                                gridDim.x * gridDim.y * gridDim.z);
}

// Batched gradient, per-pixel gather family: one persistent launch walks the gradient units of
// the batch table's items that take this family (a unit is one 32 x 4 tile of one view of one
// item, in the order of k_grad's grid), each writing its own loss partial.  The dynamic shared memory holds `planes` planes; an item with more sets the batch bit
// of the status word and is skipped.
template <typename Tm>
__global__ void __launch_bounds__(kGradThreads, kGradMinBlocks)
k_grad_batch(const RLBatchHeader* __restrict__ hdr, const RLBatchItem* __restrict__ items, int planes) {
    extern __shared__ float sT[];  // [ceil(planes / kGroup)][kGradThreads]
    const unsigned n = hdr->n, total = hdr->grad_units;
    if (hdr->dtype != (std::is_same<Tm, float>::value ? (unsigned)RL_F32 : (unsigned)RL_BF16)) return;
    const int tid = threadIdx.y * kGradBX + threadIdx.x;
    __shared__ unsigned next_slot;
    for (unsigned u = rl_batch_next(hdr, 1, &next_slot); u < total; u = rl_batch_next(hdr, 1, &next_slot)) {
        const RLBatchItem& it = items[rl_batch_find(items, n, u, &RLBatchItem::grad_begin)];
        if (it.D > planes) {
            if (tid == 0 && hdr->status) atomicOr(hdr->status, RL_DEVFLAG_BATCH);
            continue;
        }
        const unsigned local = u - it.grad_begin;
        const unsigned view = local % (unsigned)it.N, tile = local / (unsigned)it.N;
        const int tx = (int)(tile % it.grad_tiles_x), ty = (int)(tile / it.grad_tiles_x);
        const int h = it.H >> it.level, w = it.W >> it.level;
#define RL_GB(A) grad_tile<Tm, kGroup, true, true, A>(static_cast<const Tm*>(it.Ml), it.D, h, w, it.views, (int)view,    \
                                             tx * kGradBX + threadIdx.x, ty * kGradBY + threadIdx.y, tid, sT,       \
                                             it.level ? it.Il : it.images, 0, nullptr, it.slots, it.G, it.inv_n,    \
                                             it.partials,                                                           \
                                             local, it.grad_units)
        if (it.views.anchored) RL_GB(kAnchored);
        else RL_GB(kPlain);
#undef RL_GB
        __syncthreads();  // sT is reused by the next unit
    }
}

// The loss from the per-block partials (reallife_loss_grad; an HSGD step's update does it).
__global__ void __launch_bounds__(1024) k_loss_reduce(const float* __restrict__ partials, int n, float scale,
                                                     float* __restrict__ out) {
    __shared__ float red[32];
    const float total = rl_partials_sum(partials, (unsigned)n, threadIdx.x, blockDim.x, red);
    if (threadIdx.x == 0) out[0] = total * scale;
}

// Planes a group: one (48 registers, 40 resident warps) while the stored transmittances, 512 bytes a
// plane and block, leave room for the blocks and the L1, else two (64 registers, half the bytes).
// Gradient of 1200x576, 4 anchored views, us, one against two: FP32 D = 32 723 / 757, D = 40 982 / 955,
// D = 64 2204 / 1579; BF16 D = 32 653 / 713, D = 48 985 / 1037, D = 64 1633 / 1349.
int grad_group(int D, bool f32) { return D <= (f32 ? 32 : 48) ? 1 : kGroup; }

template <typename Tm, bool SPARSE, bool LOSS>
void launch_grad_t(const void* M, int D, int H, int W, const RLViews& views, const float* images, int img_level,
                   const float* grad_out, const uint8_t* slots, float* G, float inv_n, float* partials,
                   dim3 grid, cudaStream_t s) {
    const int group = grad_group(D, sizeof(Tm) == 4);
    const size_t smem = (size_t)((D + group - 1) / group) * kGradThreads * sizeof(float);
#define RL_MODE(GR) (views.shifts ? k_grad<Tm, GR, SPARSE, LOSS, kShifts>            \
                     : views.anchored ? k_grad<Tm, GR, SPARSE, LOSS, kAnchored>   \
                                      : k_grad<Tm, GR, SPARSE, LOSS, kPlain>)
    auto kern = group == 1 ? RL_MODE(1) : RL_MODE(kGroup);
#undef RL_MODE
    kern<<<grid, dim3(kGradBX, kGradBY), smem, s>>>((const Tm*)M, D, H, W, views, images, img_level, grad_out, slots, G,
                                                    inv_n, partials);
}

}  // namespace

size_t rl_grad_num_blocks(int H, int W, int N) {
    const size_t own = (size_t)((W + kGradBX - 1) / kGradBX) * ((H + kGradBY - 1) / kGradBY) * N;
    const size_t a = rl_grad_pp_num_blocks(H, W, N);
    return own > a ? own : a;
}

rl_status rl_launch_grad(const void* M, rl_dtype dt, int D, int H, int W, const RLViews& views, bool mode_loss,
                         const float* images, int img_level, const float* grad_out, const uint8_t* slots, float* G,
                         float inv_n, float* partials, int* nblocks, cudaStream_t s) {
    if (rl_grad_path(H, W, views.n, D, views.anchored != 0, views.shifts != 0, slots != nullptr) != 2)
        return rl_launch_grad_pp(M, dt, D, H, W, views, mode_loss, images, img_level, grad_out, slots, G, inv_n,
                                 partials, nblocks, s);
    const int tiles_x = (W + kGradBX - 1) / kGradBX, tiles_y = (H + kGradBY - 1) / kGradBY;
    const dim3 grid((unsigned)views.n, (unsigned)tiles_x, (unsigned)tiles_y);
    if (nblocks) *nblocks = (int)(grid.x * grid.y * grid.z);
    const bool sparse = slots != nullptr;
    const char* name = dt == RL_F32 ? (sparse ? "grad_sparse_f32" : "grad_dense_f32")
                                    : (sparse ? "grad_sparse_bf16" : "grad_dense_bf16");
    RLTraceScope ts(name, s);
#define RL_GRAD_CASE(TM, SP, LS) \
    launch_grad_t<TM, SP, LS>(M, D, H, W, views, images, img_level, grad_out, slots, G, inv_n, partials, grid, s)
    // a slot map comes with the loss mode only
#define RL_KIND(TM)                                                                               \
    do {                                                                                          \
        if (slots) RL_GRAD_CASE(TM, true, true);                                                      \
        else if (mode_loss) RL_GRAD_CASE(TM, false, true);                                            \
        else RL_GRAD_CASE(TM, false, false);                                                          \
    } while (0)
    if (dt == RL_F32) RL_KIND(float);
    else RL_KIND(__nv_bfloat16);
#undef RL_KIND
#undef RL_GRAD_CASE
    return rl_check_launch("grad");
}

unsigned rl_grad_gather_tiles_x(int w) { return (unsigned)((w + kGradBX - 1) / kGradBX); }
unsigned rl_grad_gather_tiles_y(int h) { return (unsigned)((h + kGradBY - 1) / kGradBY); }

rl_status rl_launch_grad_batch(const void* table, rl_dtype dt, int planes, cudaStream_t s) {
    const RLBatchHeader* hdr = static_cast<const RLBatchHeader*>(table);
    const RLBatchItem* items = rl_batch_items(table);
    planes = planes < 1 ? 1 : (planes > RL_DEV_MAX_PLANES ? RL_DEV_MAX_PLANES : planes);
    const size_t smem = (size_t)((planes + kGroup - 1) / kGroup) * kGradThreads * sizeof(float);
    // the resident blocks of the largest shared memory, so that any later capacity fits the grid
    const size_t smem_max = (size_t)((RL_DEV_MAX_PLANES + kGroup - 1) / kGroup) * kGradThreads * sizeof(float);
    const int grid = dt == RL_F32 ? rl_persistent_grid<k_grad_batch<float>>(kGradThreads, smem_max)
                                  : rl_persistent_grid<k_grad_batch<__nv_bfloat16>>(kGradThreads, smem_max);
    if (dt == RL_F32) {
        RLTraceScope ts("grad_batch_f32", s);
        k_grad_batch<float><<<grid, dim3(kGradBX, kGradBY), smem, s>>>(hdr, items, planes);
    } else {
        RLTraceScope ts("grad_batch_bf16", s);
        k_grad_batch<__nv_bfloat16><<<grid, dim3(kGradBX, kGradBY), smem, s>>>(hdr, items, planes);
    }
    return rl_check_launch("grad_batch");
}

rl_status rl_launch_loss_reduce(const float* partials, int n, float scale, float* out, cudaStream_t s) {
    RLTraceScope ts("loss_reduce", s);
    k_loss_reduce<<<1, 1024, 0, s>>>(partials, n, scale, out);
    return rl_check_launch("loss_reduce");
}

RL_DEBUG_READER(grad)
