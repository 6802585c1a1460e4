// render.cu -- novel-view rendering (Eq. eq_render, Eq. eq_over) and warp diagnostics.
//
// One thread per target pixel: for d = D-1 .. 0 (nearest first) sample plane d at
// p = q + a(q) + rho_d b(q) (bilinear, zero padding per tap; coordinates anchored per block in
// FP64, rl_common.cuh) and accumulate
// C += T alpha c, T *= (1 - alpha).  The loop stops once T is exactly zero, after which
// every further term is exactly zero.
// What bounds it: instruction issue (1920x1080, D = 64, BF16, anchored: 78% of the issue slots at
// 83 instructions a sample before).  A warp whose samples of the nearest and the farthest plane lie
// inside the planes has all of them inside, so it leaves out the border tests and takes the fast
// coordinates of rl_common.cuh, two planes at a time (render_group): 13.2 against 17.0 ms for 45 such views, 82
// against 86 us for 4 rotated 500x375 views, D = 32, FP32 (13.6 ms without the packed arithmetic of
// positions and weights; without it too, one plane at a time 14.7 ms, four 14.5).  Views that are pure
// shifts of the reference (no rotation, no depth offset, same focal lengths) take a kernel that
// computes each plane's shift and weights once per block and renders four pixels of a column per thread, loading
// each tap row once.
#include "rl_internal.h"

namespace {

constexpr int kRenderBX = 32, kRenderBY = 4;
#ifndef RL_RENDER_MIN_BLOCKS
#define RL_RENDER_MIN_BLOCKS 1  // no register cap: measured fastest
#endif

// Blocks are ordered view-fastest (grid x = view) so that the views of a tile, whose plane
// footprints overlap, run together and share the MPI through L2.
// GROUP: planes whose loads are in flight together.
template <typename Tm, bool ANCH, int GROUP>
__global__ void __launch_bounds__(kRenderBX* kRenderBY, RL_RENDER_MIN_BLOCKS)
k_render(const Tm* __restrict__ M, int D, int H, int W, const __grid_constant__ RLViews views, int tiles_x,
         float* __restrict__ out) {
    __shared__ RLAnchor sA;
    const int view = blockIdx.x;  // grid (views, tiles_x, tiles_y): views of a tile run together
    if (ANCH)
        rl_anchor_build(&sA, views, view, blockIdx.y * kRenderBX + kRenderBX / 2,
                        blockIdx.z * kRenderBY + kRenderBY / 2, D, W,
                        threadIdx.y * kRenderBX + threadIdx.x, kRenderBX * kRenderBY);
    const int qx = blockIdx.y * kRenderBX + threadIdx.x;
    const int qy = blockIdx.z * kRenderBY + threadIdx.y;
    const unsigned act = __ballot_sync(0xffffffffu, qx < W && qy < H);
    if (qx >= W || qy >= H) return;
    const RLPixWarp<ANCH> w = rl_pix_warp<ANCH>(sA, views.v[view], qx, qy);
    const size_t plane = (size_t)H * W * 4;
    const unsigned hw = (unsigned)(H * W);
    float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    const auto over = [&](const float4& m) {
        const float a = T * m.w;
        c0 = fmaf(a, m.x, c0);
        c1 = fmaf(a, m.y, c1);
        c2 = fmaf(a, m.z, c2);
        T = T * (1.f - m.w);
    };
    // warps whose samples of every plane lie inside it take GROUP planes at a time, without
    // the border tests (not worth testing for with one or two planes)
    int d = D - 1;
    if (D > 2 && __all_sync(act, rl_chunk_inside<ANCH>(w, sA, views, 0, D - 1, qx, qy, H, W))) {
        const unsigned base = rl_fast_base(qx, qy, W);
#pragma unroll 1
        for (; d >= GROUP - 1 && T != 0.f; d -= GROUP) {
            float4 m[GROUP];
#pragma unroll
            for (int i = 0; i < GROUP; ++i) {
                const RLFastTap t = rl_fast_tap<ANCH>(w, sA, d - i, views.rho[d - i], base, W);
                m[i] = RL_IN((long long)t.idx + W + 1, hw)
                           ? rl_sample_at(M, (unsigned)(d - i) * hw + t.idx, W, rl_weights_packed(t.fx, t.fy))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int i = 0; i < GROUP; ++i)
                if (i == 0 || T != 0.f) over(m[i]);
        }
    }
#pragma unroll 1
    for (; d >= 0 && T != 0.f; --d)
        over(rl_sample_fast(M + d * plane, H, W, w.taps(sA, d, views.rho[d], qx, qy)));
    float* o = out + (((size_t)view * H + qy) * W + qx) * 3;
    o[0] = c0;
    o[1] = c1;
    o[2] = c2;
}

// Views with no rotation relative to the reference, no depth offset and the reference's
// focal lengths: the warp offset p - q = a + rho_d b is the same for every pixel of a plane,
// so the taps' integer shift and the bilinear weights are computed once per plane from the
// block's FP64 anchor table (rl_common.cuh) and read from shared memory.  Same samples, same
// results as k_render.
struct RLPlaneShift {
    int ix, iy, ok;
    float fx, fy;
    float w00, w10, w01, w11;
};

// One thread renders kShiftRows vertically adjacent pixels of a column: for each plane their
// taps span kShiftRows + 1 rows of two columns, loaded once (kShiftRows + 1 rows x 2 loads
// instead of kShiftRows x 4).
constexpr int kShiftRows = 4;

template <typename Tm>
__global__ void __launch_bounds__(kRenderBX* kRenderBY, 8)
k_render_shift(const Tm* __restrict__ M, int D, int H, int W, const __grid_constant__ RLViews views,
               float* __restrict__ out) {
    __shared__ RLPlaneShift sp[RL_DEV_MAX_PLANES];
    const int view = blockIdx.x;  // grid (views, tiles_x, tiles_y of kRenderBY * kShiftRows rows)
    const int tid = threadIdx.y * kRenderBX + threadIdx.x;
    if (tid < D) {
        // a pure shift: p - q = (c_r - c_v) + rho_d f_r C_xy for every pixel, formed in FP64 and
        // split into an integer and an FP32 fraction (the anchors of rl_common.cuh, exactly)
        const RLViewParam64& P = views.v64[view];
        const double rho = views.rho64[tid];
        const double kx = P.dcx + rho * (P.fxr * P.C[0]), ky = P.dcy + rho * (P.fyr * P.C[1]);
        const double flx = floor(kx), fly = floor(ky);
        RLPlaneShift p;
        p.ok = fabs(kx) < 1e9 && fabs(ky) < 1e9;
        p.ix = p.ok ? (int)flx : 0;
        p.iy = p.ok ? (int)fly : 0;
        p.fx = (float)(kx - flx);
        p.fy = (float)(ky - fly);
        p.w00 = (1.f - p.fx) * (1.f - p.fy);
        p.w10 = p.fx * (1.f - p.fy);
        p.w01 = (1.f - p.fx) * p.fy;
        p.w11 = p.fx * p.fy;
        sp[tid] = p;
    }
    __syncthreads();
    const int qx = blockIdx.y * kRenderBX + threadIdx.x;
    const int qy0 = (blockIdx.z * kRenderBY + threadIdx.y) * kShiftRows;
    if (qx >= W || qy0 >= H) return;
    const size_t plane = (size_t)H * W * 4;
    float T[kShiftRows], c0[kShiftRows], c1[kShiftRows], c2[kShiftRows];
#pragma unroll
    for (int r = 0; r < kShiftRows; ++r) { T[r] = 1.f; c0[r] = c1[r] = c2[r] = 0.f; }
    for (int d = D - 1; d >= 0; --d) {
        const RLPlaneShift p = sp[d];
        const int x0 = qx + p.ix, y0 = qy0 + p.iy;
        float4 m[kShiftRows];
        if (p.ok && (unsigned)x0 < (unsigned)(W - 1) && y0 >= 0 && y0 + kShiftRows < H) {
            // all kShiftRows + 1 tap rows inside: load each once
            const Tm* q = M + d * plane + (unsigned)(y0 * W + x0) * 4u;
            float4 a0 = RLStore<Tm>::load4(q), a1 = RLStore<Tm>::load4(q + 4);
#pragma unroll
            for (int r = 0; r < kShiftRows; ++r) {
                const Tm* qr = q + (r + 1) * 4 * W;
                const float4 b0 = RLStore<Tm>::load4(qr), b1 = RLStore<Tm>::load4(qr + 4);
                float2 lo = __fmul2_rn(make_float2(p.w00, p.w00), make_float2(a0.x, a0.y));
                float2 hi = __fmul2_rn(make_float2(p.w00, p.w00), make_float2(a0.z, a0.w));
                lo = __ffma2_rn(make_float2(p.w10, p.w10), make_float2(a1.x, a1.y), lo);
                hi = __ffma2_rn(make_float2(p.w10, p.w10), make_float2(a1.z, a1.w), hi);
                lo = __ffma2_rn(make_float2(p.w01, p.w01), make_float2(b0.x, b0.y), lo);
                hi = __ffma2_rn(make_float2(p.w01, p.w01), make_float2(b0.z, b0.w), hi);
                lo = __ffma2_rn(make_float2(p.w11, p.w11), make_float2(b1.x, b1.y), lo);
                hi = __ffma2_rn(make_float2(p.w11, p.w11), make_float2(b1.z, b1.w), hi);
                m[r] = make_float4(lo.x, lo.y, hi.x, hi.y);
                a0 = b0;
                a1 = b1;
            }
        } else {
#pragma unroll
            for (int r = 0; r < kShiftRows; ++r) {
                RLTaps t;
                t.x0 = x0;
                t.y0 = y0 + r;
                t.fx = p.fx;
                t.fy = p.fy;
                t.ok = p.ok != 0;
                m[r] = rl_sample(M + d * plane, H, W, t);
            }
        }
        bool any = false;
#pragma unroll
        for (int r = 0; r < kShiftRows; ++r) {
            const float a = T[r] * m[r].w;
            c0[r] = fmaf(a, m[r].x, c0[r]);
            c1[r] = fmaf(a, m[r].y, c1[r]);
            c2[r] = fmaf(a, m[r].z, c2[r]);
            T[r] = T[r] * (1.f - m[r].w);
            any |= T[r] != 0.f;
        }
        if (!any) break;  // every further term of every pixel is exactly zero
    }
#pragma unroll
    for (int r = 0; r < kShiftRows; ++r) {
        if (qy0 + r >= H) break;
        float* o = out + (((size_t)view * H + qy0 + r) * W + qx) * 3;
        o[0] = c0[r];
        o[1] = c1[r];
        o[2] = c2[r];
    }
}

__global__ void k_warp_offsets(int D, int H, int W, const __grid_constant__ RLViews views, float* __restrict__ out) {
    const int qx = blockIdx.x * blockDim.x + threadIdx.x;
    const int qy = blockIdx.y;
    if (qx >= W) return;
    const RLWarp w = rl_warp_coeffs(views.v[0], (float)qx, (float)qy);
    for (int d = 0; d < D; ++d) {
        const float rho = views.rho[d];
        const bool ok = w.dir_ok && (fmaf(-rho, w.cz, 1.0f) > 0.0f);
        float* o = out + (((size_t)d * H + qy) * W + qx) * 2;
        o[0] = ok ? fmaf(rho, w.bx, w.ax) : __int_as_float(0x7fc00000);
        o[1] = ok ? fmaf(rho, w.by, w.ay) : __int_as_float(0x7fc00000);
    }
}

// Planes a group: two, but one where the walk is too short to pay for the registers (FP32 70 against 48, BF16 56
// against 48) that keep other blocks from hiding the set-up: FP32 up to 32 planes with anchors, whose FP64
// set-up is long (1920x1080, 3 views: D = 8 269 us with two, 239 with one; D = 32 644 / 614; 9 views:
// D = 32 1987 / 1917, D = 40 2437 / 2466), else up to 4 (960x540, 9 views: D = 4 66.5 / 62.0; 1920x1080,
// D = 8 70.6 / 72.3); BF16 up to 2 (1920x1080, 3 views: D = 1 52.5 / 47.6, D = 4 190.7 / 192.1).
int render_group(int D, bool f32, bool anchored) { return D <= (f32 ? (anchored ? 32 : 4) : 2) ? 1 : 2; }

template <typename Tm>
void launch_render_t(const void* M, int D, int H, int W, const RLViews& views, int tiles_x, dim3 grid, float* out,
                     cudaStream_t s) {
    auto kern = render_group(D, sizeof(Tm) == 4, views.anchored != 0) == 1
                    ? (views.anchored ? k_render<Tm, true, 1> : k_render<Tm, false, 1>)
                    : (views.anchored ? k_render<Tm, true, 2> : k_render<Tm, false, 2>);
    kern<<<grid, dim3(kRenderBX, kRenderBY), 0, s>>>((const Tm*)M, D, H, W, views, tiles_x, out);
}

}  // namespace

rl_status rl_launch_render(const void* M, rl_dtype dt, int D, int H, int W, const RLViews& views, float* out,
                           cudaStream_t s) {
    const int path = rl_kernel_path(H, W, views.n);
    if (path != 2) return rl_launch_render_pp(M, dt, D, H, W, views, out, s);
    dim3 block(kRenderBX, kRenderBY);
    const int tiles_x = (W + kRenderBX - 1) / kRenderBX, tiles_y = (H + kRenderBY - 1) / kRenderBY;
    const dim3 grid((unsigned)views.n, (unsigned)tiles_x, (unsigned)tiles_y);
    if (rl_views_are_shifts(views)) {
        const dim3 sgrid((unsigned)views.n, (unsigned)tiles_x,
                         (unsigned)((H + kRenderBY * kShiftRows - 1) / (kRenderBY * kShiftRows)));
        if (dt == RL_F32) {
            RLTraceScope ts("render_shift_f32", s);
            k_render_shift<float><<<sgrid, block, 0, s>>>((const float*)M, D, H, W, views, out);
        } else {
            RLTraceScope ts("render_shift_bf16", s);
            k_render_shift<__nv_bfloat16><<<sgrid, block, 0, s>>>((const __nv_bfloat16*)M, D, H, W, views, out);
        }
        return rl_check_launch("render");
    }
    if (dt == RL_F32) {
        RLTraceScope ts("render_f32", s);
        launch_render_t<float>(M, D, H, W, views, tiles_x, grid, out, s);
    } else {
        RLTraceScope ts("render_bf16", s);
        launch_render_t<__nv_bfloat16>(M, D, H, W, views, tiles_x, grid, out, s);
    }
    return rl_check_launch("render");
}

rl_status rl_launch_warp_offsets(int D, int H, int W, const RLViews& views, float* out, cudaStream_t s) {
    RLTraceScope ts("warp_offsets", s);
    k_warp_offsets<<<dim3((W + 127) / 128, H), 128, 0, s>>>(D, H, W, views, out);
    return rl_check_launch("warp_offsets");
}

RL_DEBUG_READER(render)
