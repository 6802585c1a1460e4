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
// planes keeps 32 warps an SM instead of 24, and its L1.  1920x1080, D = 64, 8
// views, BF16, anchored: 8.23 ms (one plane at a time 11.56 ms, groups of four 10.8 ms; before,
// with border tests in every sample and a fenced loss reduction at the end of every block, 12.9 ms).
// Views that are pure shifts of the reference take a kernel of their own (k_grad_shift).
#include <type_traits>

#include "rl_internal.h"

namespace {

constexpr int kGradBX = 32, kGradBY = 4, kGradThreads = kGradBX * kGradBY;
constexpr int kGroup = 2;          // planes whose samples are held together (grad_group, the batch)
constexpr int kGradMinBlocks = 8;  // resident blocks the registers must then allow

// One block's tile of 32 x 4 view pixels of one view.  bid / nblocks index the block among
// the launch's (or the batch item's) blocks for the loss partials.
template <typename Tm, int GROUP, bool SPARSE, bool LOSS, bool ANCH>
__device__ __forceinline__ void grad_tile(const Tm* __restrict__ M, int D, int H, int W, const RLViews& views, int view,
                                          int qx, int qy, int tid, float* __restrict__ sT,
                                          const float* __restrict__ images, int img_level,
                                          const float* __restrict__ grad_out, const uint8_t* __restrict__ slots,
                                          float* __restrict__ G, float inv_n, float* __restrict__ partials,
                                          unsigned bid, unsigned nblocks) {
    float lsum = 0.f;
    __shared__ RLAnchor sA;  // the tile's anchor: its centre pixel
    if (ANCH)
        rl_anchor_build(&sA, views, view, (qx & ~(kGradBX - 1)) + kGradBX / 2, qy - qy % kGradBY + kGradBY / 2, D,
                        W, tid, kGradThreads);
    const unsigned act = __ballot_sync(0xffffffffu, qx < W && qy < H);
    if (qx < W && qy < H) {
        const RLPixWarp<ANCH> w = rl_pix_warp<ANCH>(sA, views.v[view], qx, qy);
        const size_t plane = (size_t)H * W * 4;
        const unsigned hw = (unsigned)(H * W), base = rl_fast_base(qx, qy, W);
        // warps whose samples of every plane lie inside it skip the border tests
        const bool fast = __all_sync(act, rl_chunk_inside<ANCH>(w, sA, views, 0, D - 1, qx, qy, H, W));
        const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
        const int groups = (D + GROUP - 1) / GROUP;
        float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
        // the two kinds take separate loops: a branch in every group costs 15%
        const auto pass1 = [&](auto inside) {
#pragma unroll 1
            for (int j = groups - 1; j >= 0; --j) {
                float4 m[GROUP];
#pragma unroll
                for (int i = GROUP - 1; i >= 0; --i) {
                    const int d = j * GROUP + i, dc = GROUP == 1 ? d : min(d, D - 1);
                    if constexpr (decltype(inside)::value) {
                        const RLFastTap t = rl_fast_tap<ANCH>(w, sA, dc, views.rho[dc], base, W);
                        m[i] = RL_IN((long long)t.idx + W + 1, hw)
                                   ? rl_sample_at(M, (unsigned)dc * hw + t.idx, W, t.fx, t.fy) : none;
                    } else {
                        m[i] = rl_sample_fast(M + dc * plane, H, W, w.taps(sA, dc, views.rho[dc], qx, qy));
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
        if (fast) pass1(std::true_type());
        else pass1(std::false_type());
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
        const auto pass2 = [&](auto inside) {
#pragma unroll 1
            for (int j = 0; j < groups; ++j) {
                float4 m[GROUP];
                float Td[GROUP];
                unsigned word[GROUP];
                RLFastTap tap[GROUP];
#pragma unroll
                for (int i = GROUP - 1; i >= 0; --i) {
                    const int d = j * GROUP + i, dc = GROUP == 1 ? d : min(d, D - 1);
                    if constexpr (decltype(inside)::value) {
                        tap[i] = rl_fast_tap<ANCH>(w, sA, dc, views.rho[dc], base, W);
                        const unsigned e = (unsigned)dc * hw + tap[i].idx;
                        m[i] = none;
                        word[i] = 0xFFFFFFFFu;
                        if (RL_IN((long long)tap[i].idx + W + 1, hw)) {
                            if (SPARSE) word[i] = rl_slot_word(slots, e, W);
                            m[i] = rl_sample_at(M, e, W, tap[i].fx, tap[i].fy);
                        }
                    } else {
                        m[i] = rl_sample_fast(M + dc * plane, H, W, w.taps(sA, dc, views.rho[dc], qx, qy));
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
                            const RLFastTap t = GROUP == 1 ? tap[i] : rl_fast_tap<ANCH>(w, sA, d, views.rho[d], base, W);
                            rl_scatter_at<SPARSE>(G, word[i], (unsigned)d, t.idx, (unsigned)d * hw + t.idx, hw, W,
                                                  rl_weights(t.fx, t.fy), g, ng);
                        } else {
                            const RLTaps t = w.taps(sA, d, views.rho[d], qx, qy);
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
        if (fast) pass2(std::true_type());
        else pass2(std::false_type());
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

template <typename Tm, int GROUP, bool SPARSE, bool LOSS, bool ANCH>
__global__ void __launch_bounds__(kGradThreads, GROUP == 1 ? 10 : kGradMinBlocks)
k_grad(const Tm* __restrict__ M, int D, int H, int W, const __grid_constant__ RLViews views,
       const float* __restrict__ images, int img_level, const float* __restrict__ grad_out,
       const uint8_t* __restrict__ slots, float* __restrict__ G, float inv_n, float* __restrict__ partials) {
    extern __shared__ float sT[];  // [ceil(D / GROUP)][kGradThreads]
    // view-fastest block order: the N views of a tile run together and share M through L2
    grad_tile<Tm, GROUP, SPARSE, LOSS, ANCH>(M, D, H, W, views, blockIdx.x, blockIdx.y * kGradBX + threadIdx.x,
                                blockIdx.z * kGradBY + threadIdx.y, threadIdx.y * kGradBX + threadIdx.x, sT, images,
                                img_level, grad_out, slots, G, inv_n, partials,
                                blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z),
                                gridDim.x * gridDim.y * gridDim.z);
}

// Views that are pure shifts of the reference: the offset p - q of plane d, the same for all pixels,
// split in FP64 into an integer and a fraction.
struct ShiftTable {
    float4 w[RL_DEV_MAX_PLANES];  // the taps' weights
    int2 i[RL_DEV_MAX_PLANES];    // the integer offset (a plane not met: far outside)
};

// Fills S for view `view`; every thread of the block calls it.
__device__ __forceinline__ void shift_build(ShiftTable* S, const RLViews& V, int view, int D, int tid) {
    if (tid < D) {
        const RLViewParam64& P = V.v64[view];
        const double rho = V.rho64[tid];
        const double kx = P.dcx + rho * (P.fxr * P.C[0]), ky = P.dcy + rho * (P.fyr * P.C[1]);
        const bool ok = fabs(kx) < 1e9 && fabs(ky) < 1e9;
        const double flx = floor(kx), fly = floor(ky);
        S->i[tid] = ok ? make_int2((int)flx, (int)fly) : make_int2(RL_PLANE_NONE, RL_PLANE_NONE);
        S->w[tid] = ok ? rl_weights((float)(kx - flx), (float)(ky - fly)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
}

// Compact gradient of views that are pure shifts: display and camera grids.  Every pixel of a plane has
// the same offset and weights, so a block forms them once in FP64, reads them from shared memory, and
// two pixels of a column share their middle tap row exactly: six voxels, six slots and at most six
// reductions for two samples instead of eight of each, and no coordinates a pixel.
// What bounds it: instruction issue (67%) and latency at 24 resident warps (80 registers; blocks for 20
// or 28 warps: 6.60 and 6.31 ms).  1920x1080, D = 64, 8 views, BF16: 6.09 ms; one pixel a thread with
// the same table 6.69 ms, with anchored coordinates 8.23 ms.  512x384, D = 32, 4 views, FP32: 170 us;
// one pixel a thread 213 us.
constexpr int kShiftTileY = 2 * kGradBY;

// The tap columns x0, x0 + 1 and rows y0 .. y0 + 2 of a thread's two samples of one plane, and the
// voxel of the first (valid where column and row are inside the plane).
struct ShiftTaps {
    unsigned p;
    bool xl, xr, y[3];
    __device__ __forceinline__ ShiftTaps(const int2& o, int qx, int qy, int H, int W) {
        const int x0 = qx + o.x, y0 = qy + o.y;
        p = (unsigned)y0 * (unsigned)W + (unsigned)x0;
        xl = (unsigned)x0 < (unsigned)W;
        xr = (unsigned)(x0 + 1) < (unsigned)W;
#pragma unroll
        for (int r = 0; r < 3; ++r) y[r] = (unsigned)(y0 + r) < (unsigned)H;
    }
};

// Adds wa ga + wb gb to one voxel of the compact gradient, when it has a slot.
__device__ __forceinline__ void add_kept(float4* __restrict__ G4, unsigned slot, unsigned hw, unsigned p, float wa,
                                         const float4& ga, float wb, const float4& gb, unsigned ng) {
    if (slot == RL_SLOT_NONE || !RL_IN(slot, ng)) return;
    const float2 lo = __ffma2_rn(make_float2(wb, wb), make_float2(gb.x, gb.y),
                                 __fmul2_rn(make_float2(wa, wa), make_float2(ga.x, ga.y)));
    const float2 hi = __ffma2_rn(make_float2(wb, wb), make_float2(gb.z, gb.w),
                                 __fmul2_rn(make_float2(wa, wa), make_float2(ga.z, ga.w)));
    atomicAdd(G4 + (slot * hw + p), make_float4(lo.x, lo.y, hi.x, hi.y));
}

template <typename Tm>
__global__ void __launch_bounds__(kGradThreads, 6)
k_grad_shift(const Tm* __restrict__ M, int D, int H, int W, const __grid_constant__ RLViews views,
             const float* __restrict__ images, int img_level, const uint8_t* __restrict__ slots, float* __restrict__ G,
             float inv_n, float* __restrict__ partials) {
    extern __shared__ float sT[];  // [ceil(D / kGroup)][2][kGradThreads]
    __shared__ ShiftTable sS;
    const int tid = threadIdx.x, view = blockIdx.x;
    shift_build(&sS, views, view, D, tid);
    const int px = blockIdx.y * kGradBX + (tid & 31), qy = blockIdx.z * kShiftTileY + (tid >> 5) * 2;
    const bool act0 = px < W && qy < H, act1 = act0 && qy + 1 < H;
    const int qx = min(px, W - 1);  // lanes without a pixel repeat the last one's and scatter nothing
    const unsigned hw = (unsigned)(H * W);
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    const int groups = (D + kGroup - 1) / kGroup;
    // Zero padding by taps that read as zeros: one path for all samples, whose code fits the
    // instruction cache (with a second, checked path beside it 512x384 takes 223 us).
    const auto samples = [&](const ShiftTaps& t, int d, float4& m0, float4& m1) {
        const float4 w = sS.w[d];
        float4 l[3], r[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const unsigned q = t.p + (unsigned)i * (unsigned)W;
            // as a signed index: the left tap of a valid right one may be voxel -1
            const Tm* v = M + (ptrdiff_t)(int)((unsigned)d * hw + q) * 4;
            l[i] = r[i] = none;
            if (t.y[i] && t.xl && RL_IN(q, hw)) l[i] = RLStore<Tm>::load4(v);
            if (t.y[i] && t.xr && RL_IN(q + 1u, hw)) r[i] = RLStore<Tm>::load4(v + 4);
        }
        m0 = rl_blend(l[0], r[0], l[1], r[1], w);
        m1 = rl_blend(l[1], r[1], l[2], r[2], w);
    };
    float T0 = act0 ? 1.f : 0.f, T1 = act1 ? 1.f : 0.f;
    float3 c0 = make_float3(0.f, 0.f, 0.f), c1 = c0;
    const auto over = [](float& T, float3& c, const float4& m) {
        const float a = T * m.w;
        c.x = fmaf(a, m.x, c.x);
        c.y = fmaf(a, m.y, c.y);
        c.z = fmaf(a, m.z, c.z);
        T = T * (1.f - m.w);
    };
#pragma unroll 1
    for (int j = groups - 1; j >= 0; --j) {
        float4 m0[kGroup], m1[kGroup];
#pragma unroll
        for (int i = kGroup - 1; i >= 0; --i) {
            const int d = j * kGroup + i, dc = min(d, D - 1);
            samples(ShiftTaps(sS.i[dc], qx, qy, H, W), dc, m0[i], m1[i]);
            if (d >= D) m0[i] = m1[i] = none;  // beyond the last plane
        }
        sT[(2 * j) * kGradThreads + tid] = T0;
        sT[(2 * j + 1) * kGradThreads + tid] = T1;
#pragma unroll
        for (int i = kGroup - 1; i >= 0; --i) {
            over(T0, c0, m0[i]);
            over(T1, c1, m1[i]);
        }
    }
    float lsum = 0.f;
    const auto residual = [&](int y, const float3& c, bool act) {
        float3 r = make_float3(0.f, 0.f, 0.f);
        if (!act) return r;
        // source image at this level: mean of the 2^l x 2^l full-resolution block, rounded on its own
        const int s = 1 << img_level, Wf = W << img_level, Hf = H << img_level;
        const float* img = images + (size_t)view * Hf * Wf * 3;
        float i0 = 0.f, i1 = 0.f, i2 = 0.f;
        for (int yy = 0; yy < s; ++yy)
            for (int xx = 0; xx < s; ++xx) {
                const float* q = img + ((size_t)(y * s + yy) * Wf + (qx * s + xx)) * 3;
                i0 += __ldg(q);
                i1 += __ldg(q + 1);
                i2 += __ldg(q + 2);
            }
        const float inv_area = 1.f / (float)(s * s);
        const float e0 = c.x - __fmul_rn(i0, inv_area), e1 = c.y - __fmul_rn(i1, inv_area),
                    e2 = c.z - __fmul_rn(i2, inv_area);
        lsum += fmaf(e0, e0, fmaf(e1, e1, e2 * e2));
        return make_float3(e0 * inv_n, e1 * inv_n, e2 * inv_n);
    };
    const float3 r0 = residual(qy, c0, act0), r1 = residual(qy + 1, c1, act1);
    float3 b0 = make_float3(0.f, 0.f, 0.f), b1 = b0;
    const unsigned ng = views.gplanes ? (unsigned)views.gplanes : (unsigned)D;  // checked in debug builds
    float4* G4 = reinterpret_cast<float4*>(G);
    const auto adjoint = [&](float Td, const float4& m, const float3& b, const float3& r) {
        if (Td == 0.f) return none;
        const float gc = Td * m.w;
        return make_float4(gc * r.x, gc * r.y, gc * r.z,
                           Td * fmaf(m.x - b.x, r.x, fmaf(m.y - b.y, r.y, (m.z - b.z) * r.z)));
    };
    const auto behind = [](float3& b, const float4& m) {
        const float om = 1.f - m.w;
        b.x = fmaf(m.x, m.w, om * b.x);
        b.y = fmaf(m.y, m.w, om * b.y);
        b.z = fmaf(m.z, m.w, om * b.z);
    };
#pragma unroll 1
    for (int j = 0; j < groups; ++j) {
        float4 m0[kGroup], m1[kGroup];
        float Ta[kGroup], Tb[kGroup];
        unsigned word[kGroup], low[kGroup];  // slots of the upper two tap rows, of the lowest
#pragma unroll
        for (int i = kGroup - 1; i >= 0; --i) {
            const int d = j * kGroup + i, dc = min(d, D - 1);
            const ShiftTaps t(sS.i[dc], qx, qy, H, W);
            unsigned s[6];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const unsigned q = t.p + (unsigned)r * (unsigned)W;
                const uint8_t* v = slots + (ptrdiff_t)(int)((unsigned)dc * hw + q);
                s[2 * r] = s[2 * r + 1] = RL_SLOT_NONE;
                if (t.y[r] && t.xl && RL_IN(q, hw)) s[2 * r] = __ldg(v);
                if (t.y[r] && t.xr && RL_IN(q + 1u, hw)) s[2 * r + 1] = __ldg(v + 1);
            }
            samples(t, dc, m0[i], m1[i]);
            word[i] = s[0] | s[1] << 8 | s[2] << 16 | s[3] << 24;
            low[i] = s[4] | s[5] << 8;
            if (d >= D) m0[i] = m1[i] = none;
        }
        float t0 = sT[(2 * j) * kGradThreads + tid], t1 = sT[(2 * j + 1) * kGradThreads + tid];
#pragma unroll
        for (int i = kGroup - 1; i >= 0; --i) {
            Ta[i] = t0;
            Tb[i] = t1;
            t0 = t0 * (1.f - m0[i].w);
            t1 = t1 * (1.f - m1[i].w);
        }
#pragma unroll
        for (int i = 0; i < kGroup; ++i) {
            const int d = j * kGroup + i;
            // a pixel beyond the image scatters nothing, even where a voxel that it alone samples is not finite
            if (d < D && act0 && (Ta[i] != 0.f || Tb[i] != 0.f)) {
                const float4 g0 = adjoint(Ta[i], m0[i], b0, r0), g1 = act1 ? adjoint(Tb[i], m1[i], b1, r1) : none;
                const int2 o = sS.i[d];
                const unsigned p = (unsigned)(qy + o.y) * (unsigned)W + (unsigned)(qx + o.x);
                const float4 w = sS.w[d];
                if (word[i] != 0xFFFFFFFFu) {
                    const unsigned s00 = word[i] & 255u, s10 = (word[i] >> 8) & 255u;
                    if (s00 != RL_SLOT_NONE && RL_IN(s00, ng))
                        rl_add_tap(G4, s00 * hw + p, w.x, make_float2(g0.x, g0.y), make_float2(g0.z, g0.w));
                    if (s10 != RL_SLOT_NONE && RL_IN(s10, ng))
                        rl_add_tap(G4, s10 * hw + p + 1u, w.y, make_float2(g0.x, g0.y), make_float2(g0.z, g0.w));
                    add_kept(G4, (word[i] >> 16) & 255u, hw, p + (unsigned)W, w.z, g0, w.x, g1, ng);
                    add_kept(G4, word[i] >> 24, hw, p + (unsigned)W + 1u, w.w, g0, w.y, g1, ng);
                }
                if (low[i] != 0xFFFFu) {
                    const unsigned s01 = low[i] & 255u, s11 = low[i] >> 8, q = p + 2u * (unsigned)W;
                    if (s01 != RL_SLOT_NONE && RL_IN(s01, ng))
                        rl_add_tap(G4, s01 * hw + q, w.z, make_float2(g1.x, g1.y), make_float2(g1.z, g1.w));
                    if (s11 != RL_SLOT_NONE && RL_IN(s11, ng))
                        rl_add_tap(G4, s11 * hw + q + 1u, w.w, make_float2(g1.x, g1.y), make_float2(g1.z, g1.w));
                }
            }
            behind(b0, m0[i]);
            behind(b1, m1[i]);
        }
    }
    __shared__ float red[kGradThreads / 32];
    lsum = rl_warp_sum(lsum);
    if ((tid & 31) == 0) red[tid >> 5] = lsum;
    __syncthreads();
    if (tid == 0) {
        float blk = 0.f;
        for (int j = 0; j < kGradThreads / 32; ++j) blk += red[j];
        const unsigned bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
        if (RL_IN(bid, gridDim.x * gridDim.y * gridDim.z)) partials[bid] = blk;
    }
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
        if (it.views.anchored) RL_GB(true);
        else RL_GB(false);
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
    auto kern = group == 1
                    ? (views.anchored ? k_grad<Tm, 1, SPARSE, LOSS, true> : k_grad<Tm, 1, SPARSE, LOSS, false>)
                    : (views.anchored ? k_grad<Tm, kGroup, SPARSE, LOSS, true> : k_grad<Tm, kGroup, SPARSE, LOSS, false>);
    kern<<<grid, dim3(kGradBX, kGradBY), smem, s>>>((const Tm*)M, D, H, W, views, images, img_level, grad_out, slots, G,
                                                    inv_n, partials);
}

}  // namespace

size_t rl_grad_num_blocks(int H, int W, int N) {
    const size_t own = (size_t)((W + kGradBX - 1) / kGradBX) * ((H + kGradBY - 1) / kGradBY) * N;
    const size_t a = rl_grad_pp_num_blocks(H, W, N, false), b = rl_grad_pp_num_blocks(H, W, N, true);
    return own > a ? (own > b ? own : b) : (a > b ? a : b);
}

rl_status rl_launch_grad(const void* M, rl_dtype dt, int D, int H, int W, const RLViews& views, bool mode_loss,
                         const float* images, int img_level, const float* grad_out, const uint8_t* slots, float* G,
                         float inv_n, float* partials, int* nblocks, cudaStream_t s) {
    if (rl_grad_path(H, W, views.n, D, views.anchored != 0, views.shifts != 0, slots != nullptr) != 2)
        return rl_launch_grad_pp(M, dt, D, H, W, views, mode_loss, images, img_level, grad_out, slots, G, inv_n,
                                 partials, nblocks, s);
    const int tiles_x = (W + kGradBX - 1) / kGradBX, tiles_y = (H + kGradBY - 1) / kGradBY;
    if (views.shifts && slots && mode_loss) {
        const dim3 sgrid((unsigned)views.n, (unsigned)tiles_x, (unsigned)((H + kShiftTileY - 1) / kShiftTileY));
        const size_t smem = (size_t)((D + kGroup - 1) / kGroup) * 2 * kGradThreads * sizeof(float);
        if (nblocks) *nblocks = (int)(sgrid.x * sgrid.y * sgrid.z);
        if (dt == RL_F32) {
            RLTraceScope ts("grad_sparse_f32", s);
            k_grad_shift<float><<<sgrid, kGradThreads, smem, s>>>((const float*)M, D, H, W, views, images, img_level,
                                                                  slots, G, inv_n, partials);
        } else {
            RLTraceScope ts("grad_sparse_bf16", s);
            k_grad_shift<__nv_bfloat16><<<sgrid, kGradThreads, smem, s>>>((const __nv_bfloat16*)M, D, H, W, views,
                                                                          images, img_level, slots, G, inv_n, partials);
        }
        return rl_check_launch("grad_shift");
    }
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
