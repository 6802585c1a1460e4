// pp.cu -- plane-parallel warp kernels: novel-view rendering (Eq. eq_render, eq_over) and
// the fused warp + composite + residual + exact adjoint of one HSGD iteration.
//
// Layout.  Several warps share the same 32 view pixels (grid = (views, tiles_x, tiles_y), so that
// the views of a tile run together); warp g owns a chunk of consecutive planes, so a warp's loads
// of one plane are neighbouring voxels.  Each thread samples its C planes once and keeps them in
// registers, nearest first forming its chunk's composite Cc_g = sum c_d alpha_d T_d^loc
// and transmittance Tc_g = prod (1 - alpha_d).  The over operator is associative, so the
// chunks combine exactly:
//   T before chunk g (everything nearer):  Tb_g = prod_{g' > g} Tc_g'
//   pixel colour:                          C = f_{G-1}(... f_0(0)), f_g(x) = Cc_g + Tc_g x
//   composite of everything farther:       Bb_g = f_{g-1}(... f_0(0))
// (shared-memory exchange of the per-chunk (Cc, Tc)).  The adjoint of plane d then uses
// T_d = Tb_g T_d^loc and the running below-composite B_d (B_{d+1} = c_d alpha_d + (1 -
// alpha_d) B_d, starting from Bb_g) -- no division by (1 - alpha), no second gather.
// Bilinear weights are applied with packed FP32x2 FMAs (same rounding as scalar FMAs).
#include <type_traits>

#include "rl_internal.h"

namespace {

constexpr int kTX = 16, kTY = 2, kPix = 32;  // render: pixels per block, one per lane

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// Bilinear sample; interior samples use packed FMAs, border samples the checked path.
template <typename Tm>
__device__ __forceinline__ float4 sample_pp(const Tm* __restrict__ plane, int H, int W, const RLTaps& t) {
    if (t.ok && (unsigned)t.x0 < (unsigned)(W - 1) && (unsigned)t.y0 < (unsigned)(H - 1) &&
        RL_IN((long long)t.y0 * W + t.x0 + W + 1, (long long)H * W)) {
        const Tm* p = plane + (unsigned)(t.y0 * W + t.x0) * 4u;
        const float4 v00 = RLStore<Tm>::load4(p), v10 = RLStore<Tm>::load4(p + 4);
        const float4 v01 = RLStore<Tm>::load4(p + 4 * W), v11 = RLStore<Tm>::load4(p + 4 * W + 4);
        const float w00 = (1.f - t.fx) * (1.f - t.fy), w10 = t.fx * (1.f - t.fy);
        const float w01 = (1.f - t.fx) * t.fy, w11 = t.fx * t.fy;
        float2 lo = __fmul2_rn(f2(w00, w00), f2(v00.x, v00.y));
        float2 hi = __fmul2_rn(f2(w00, w00), f2(v00.z, v00.w));
        lo = __ffma2_rn(f2(w10, w10), f2(v10.x, v10.y), lo);
        hi = __ffma2_rn(f2(w10, w10), f2(v10.z, v10.w), hi);
        lo = __ffma2_rn(f2(w01, w01), f2(v01.x, v01.y), lo);
        hi = __ffma2_rn(f2(w01, w01), f2(v01.z, v01.w), hi);
        lo = __ffma2_rn(f2(w11, w11), f2(v11.x, v11.y), lo);
        hi = __ffma2_rn(f2(w11, w11), f2(v11.z, v11.w), hi);
        return make_float4(lo.x, lo.y, hi.x, hi.y);
    }
    return rl_sample(plane, H, W, t);
}

struct PixelCoord {
    int qx, qy, view, g, lane;
    bool active;
};

__device__ __forceinline__ PixelCoord pixel_coord_at(int H, int W, int view, int tx, int ty) {
    PixelCoord c;
    c.view = view;
    c.g = threadIdx.x >> 5;
    c.lane = threadIdx.x & 31;
    c.qx = tx * kTX + (c.lane % kTX);
    c.qy = ty * kTY + (c.lane / kTX);
    c.active = c.qx < W && c.qy < H;
    return c;
}

// grid (views, tiles_x, tiles_y): the views of a tile run together and share M in L2
__device__ __forceinline__ PixelCoord pixel_coord(int H, int W) {
    return pixel_coord_at(H, W, blockIdx.x, blockIdx.y, blockIdx.z);
}

template <typename Tm, int C, int kGroups, bool ANCH>
__global__ void __launch_bounds__(kGroups * kPix)
k_render_pp(const Tm* __restrict__ M, int D, int H, int W, const __grid_constant__ RLViews views, int tiles_x,
            float* __restrict__ out) {
    __shared__ float4 xch[kGroups][kPix];  // per chunk: (Cc.rgb, Tc)
    __shared__ RLAnchor sA;
    const PixelCoord pc = pixel_coord(H, W);
    if (ANCH)
        rl_anchor_build(&sA, views, pc.view, blockIdx.y * kTX + kTX / 2, blockIdx.z * kTY + kTY / 2, D, W, threadIdx.x,
                        kGroups * kPix);
    const int qx = min(pc.qx, W - 1), qy = min(pc.qy, H - 1);
    const RLPixWarp<ANCH> w = rl_pix_warp<ANCH>(sA, views.v[pc.view], qx, qy);
    const size_t plane = (size_t)H * W * 4;
    float Tl = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
#pragma unroll
    for (int i = C - 1; i >= 0; --i) {
        const int d = pc.g * C + i;
        if (d < D) {
            const RLTaps t = w.taps(sA, d, views.rho[d], qx, qy);
            const float4 m = sample_pp(M + d * plane, H, W, t);
            const float a = Tl * m.w;
            c0 = fmaf(a, m.x, c0);
            c1 = fmaf(a, m.y, c1);
            c2 = fmaf(a, m.z, c2);
            Tl = Tl * (1.f - m.w);
        }
    }
    xch[pc.g][pc.lane] = make_float4(c0, c1, c2, Tl);
    __syncthreads();
    if (pc.g == 0 && pc.active) {
        float T = 1.f, o0 = 0.f, o1 = 0.f, o2 = 0.f;
#pragma unroll
        for (int g = kGroups - 1; g >= 0; --g) {
            const float4 v = xch[g][pc.lane];
            o0 = fmaf(T, v.x, o0);
            o1 = fmaf(T, v.y, o1);
            o2 = fmaf(T, v.z, o2);
            T = T * v.w;
        }
        float* o = out + (((size_t)pc.view * H + pc.qy) * W + pc.qx) * 3;
        o[0] = o0;
        o[1] = o1;
        o[2] = o2;
    }
}

// ------------------------------------------------------------------ fused gradient
//
// One block: `tiles` tiles of 32 view pixels side by side along x, G warps a tile; warp g of a
// tile holds the kChunk planes from kChunk g on (the last chunk may be short).
//
// What bounds it: at 512x384, D = 32, 4 views, FP32 the level-0 launch issues 179 M warp
// instructions at 67% of the issue slots, with 38 M L1 wavefronts (57%): one gather a sample
// (the per-pixel gather family takes two, 57 M wavefronts) plus the reductions onto the kept
// taps.  Four planes a warp at 64 registers (32 resident warps) is the measured optimum:
// 218 us, against 284 us with eight planes at 128 registers or at 80 (half the warps, and twice
// the unrolled code: instruction fetch stalls), and 455 us with four planes whose taps are kept
// instead of formed again in the adjoint (spills).  The same launch took 274 us per-pixel before.
constexpr int kChunk = 4, kMaxWarps = 16;  // RL_DEV_MAX_PLANES / kChunk

struct PPShape {
    int G, tiles;   // warps a tile, tiles a block
    int tile_x;     // a tile is tile_x x (32 / tile_x) pixels
};

// Tile of the gradient over a W x H image: 32 x 1 pixels (512x384: 218 against 224 us with 16 x 2)
// unless 16 x 2 needs fewer tiles (widths just above a multiple of 32) or the grid is too high.  Tiles
// with an anchor of their own are always 16 x 2: the error of their pixels' positions grows with the
// distance from the anchor (up to 8 pixels instead of 16: 6e-7 instead of 1.2e-6 px, 300x12, f = 300,
// rotated by 45 degrees).
__host__ __device__ inline int grad_pp_tile_x(int H, int W, bool anchored) {
    if (anchored || H > 65535) return 16;
    return (W + 15) / 16 * ((H + 1) / 2) < (W + 31) / 32 * H ? 16 : 32;
}

// Blocks of about `most_warps` warps; a tile of D planes takes ceil(D / 4) of them.
__host__ __device__ inline PPShape grad_pp_shape(int D, int H, int W, int most_warps, bool anchored) {
    PPShape s;
    s.G = (D + kChunk - 1) / kChunk;
    s.tiles = most_warps / s.G > 1 ? most_warps / s.G : 1;
    s.tile_x = grad_pp_tile_x(H, W, anchored);
    return s;
}

// Position of one thread: view pixel (qx, qy), plane chunk g of its tile.
struct PPPos {
    int view, tx, ty, tile, g, G, lane, qx, qy;
    bool active;
};

__device__ __forceinline__ PPPos pp_pos(int H, int W, int view, int bx, int by, PPShape sh) {
    PPPos c;
    const int wi = threadIdx.x >> 5;
    c.view = view;
    c.G = sh.G;
    c.tile = wi / sh.G;
    c.g = wi - c.tile * sh.G;
    c.lane = threadIdx.x & 31;
    c.tx = bx * sh.tiles + c.tile;
    c.ty = by;
    const int log_x = sh.tile_x == 32 ? 5 : 4;
    c.qx = c.tx * sh.tile_x + (c.lane & (sh.tile_x - 1));
    c.qy = (by << (5 - log_x)) + (c.lane >> log_x);
    // warps beyond the last tile of a persistent block hold no pixel
    c.active = c.tile < sh.tiles && c.qx < W && c.qy < H;
    return c;
}

// Dense transpose of a warp's samples inside plane d, one voxel e (top-left tap) a lane: where a lane's
// left taps are its neighbour's right ones, the neighbour's share comes by shuffles and one reduction
// adds both, so most voxels of a row take one reduction instead of two.  4 views of 500x375, D = 32,
// FP32: 224 us, 286 us without the joining, whose reductions were the bound (L1, ten wavefronts each;
// L2).  Now issue is (68%; L1 66%, L2 47%): joining the row below as well costs 237 us.  Lanes outside
// `act` and lanes with live = false pass g = 0.
__device__ __forceinline__ void join_taps(float* __restrict__ G, unsigned act, int lane, bool live, unsigned d,
                                          unsigned e, int W, float fx, float fy, float4 g, unsigned ng) {
    float4* G4 = reinterpret_cast<float4*>(G);
    const float4 w = rl_weights(fx, fy);
    const bool on = (act >> lane) & 1u;
    const unsigned left = __shfl_up_sync(0xffffffffu, e, 1);
    const bool take = on && lane > 0 && ((act >> (lane - 1)) & 1u) && left + 1u == e;
    const unsigned takers = __ballot_sync(0xffffffffu, take);
    const bool given = lane < 31 && ((takers >> (lane + 1)) & 1u);  // the right neighbour adds this lane's right taps
    float wy = __shfl_up_sync(0xffffffffu, w.y, 1), ww = __shfl_up_sync(0xffffffffu, w.w, 1);
    float4 h;
    h.x = __shfl_up_sync(0xffffffffu, g.x, 1);
    h.y = __shfl_up_sync(0xffffffffu, g.y, 1);
    h.z = __shfl_up_sync(0xffffffffu, g.z, 1);
    h.w = __shfl_up_sync(0xffffffffu, g.w, 1);
    if (!take) wy = ww = 0.f, h = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!on || !RL_IN(d, ng)) return;
    const float2 gl = f2(g.x, g.y), gh = f2(g.z, g.w), hl = f2(h.x, h.y), hh = f2(h.z, h.w);
    if (live || take) {
        const float2 a = __ffma2_rn(f2(wy, wy), hl, __fmul2_rn(f2(w.x, w.x), gl));
        const float2 b = __ffma2_rn(f2(wy, wy), hh, __fmul2_rn(f2(w.x, w.x), gh));
        atomicAdd(G4 + e, make_float4(a.x, a.y, b.x, b.y));
        const float2 p = __ffma2_rn(f2(ww, ww), hl, __fmul2_rn(f2(w.z, w.z), gl));
        const float2 q = __ffma2_rn(f2(ww, ww), hh, __fmul2_rn(f2(w.z, w.z), gh));
        atomicAdd(G4 + (e + (unsigned)W), make_float4(p.x, p.y, q.x, q.y));
    }
    if (live && !given) {
        rl_add_tap(G4, e + 1u, w.y, gl, gh);
        rl_add_tap(G4, e + (unsigned)W + 1u, w.w, gl, gh);
    }
}

template <typename Tm, bool FULL, bool SPARSE, bool LOSS, bool ANCH>
__device__ __forceinline__ void grad_pp_tile(const Tm* __restrict__ M, int D, int H, int W, const RLViews& views,
                                             const PPPos pc, PPShape sh, int bx, const float* __restrict__ images,
                                             int img_level, const float* __restrict__ grad_out,
                                             const uint8_t* __restrict__ slots, float* __restrict__ G, float inv_n,
                                             float* __restrict__ partials, unsigned nparts) {
    constexpr int C = kChunk;
    __shared__ float4 xch[kMaxWarps][kPix];  // per chunk: (Cc.rgb, Tc)
    __shared__ float ximg[kMaxWarps][kPix][3];
    // An anchor a tile, at its centre: no farther outside the image than the host's check of the rays
    // reaches.  One anchor for all tiles of a block lies up to 256 pixels from some of its pixels (D <= 4,
    // batched), where the FP32 differences lose what the anchor is for, or outside the image where its
    // ray leaves the reference half-space: positions 0.015 px off at 64x24, f = 64, turned by 33 degrees,
    // 1.5e-6 px with an anchor a tile.  The tiles' tables share one array: a block holds at most
    // kMaxWarps / ceil(D / kChunk) tiles, so tiles x D <= RL_DEV_MAX_PLANES entries.
    // One thread forms a tile's head and one a plane's entry: an FP64 instruction costs the same for one
    // lane as for all.
    __shared__ RLAnchor sA;  // the tables
    __shared__ RLAnchorHead sH[kMaxWarps];
    const int at = pc.tile < sh.tiles ? pc.tile : 0;  // a warp without a tile reads the first one's
    const int first = ANCH ? at * D : 0;
    if (ANCH) {
        // scratch in the exchange buffer, which is written after the last barrier here: the batched kernel
        // holds both kinds, and 512 bytes more a kind would cost it 36 KB of L1 (64 KB for two blocks)
        double(*ab)[4] = reinterpret_cast<double(*)[4]>(xch);
        const RLViewParam64& P = views.v64[pc.view];
        const int last = (W + sh.tile_x - 1) / sh.tile_x - 1, rows = kPix / sh.tile_x;
        if ((int)threadIdx.x < sh.tiles)
            rl_anchor_head(&sH[threadIdx.x], ab[threadIdx.x], P,
                           min(bx * sh.tiles + (int)threadIdx.x, last) * sh.tile_x + sh.tile_x / 2,
                           pc.ty * rows + rows / 2);
        __syncthreads();
        for (int i = threadIdx.x; i < sh.tiles * D; i += blockDim.x)
            rl_anchor_plane(sA.k + i, sA.f + i, ab[i / D], views, P, i % D, W);
        __syncthreads();
    }
    const int qx = min(pc.qx, W - 1), qy = min(pc.qy, H - 1);
    const RLPixWarp<ANCH> w = rl_pix_warp<ANCH>(sH[at], views.v[pc.view], qx, qy);
    const unsigned hw = (unsigned)(H * W);
    const size_t plane = (size_t)H * W * 4;
    const int d0 = pc.g * C;
    const int n = FULL ? C : min(C, D - d0);  // planes of this warp's chunk (>= 1)

    // a level image that is already averaged (img_level 0: one pixel a view) is read by one warp
    // before its gathers and handed to the others through shared memory at the chunk exchange
    const bool img_early = LOSS && img_level == 0 && pc.g == pc.G - 1;
    float li0 = 0.f, li1 = 0.f, li2 = 0.f;
    if (img_early && pc.active) {
        const float* px = images + (((size_t)pc.view * H + pc.qy) * W + pc.qx) * 3;
        li0 = __ldg(px);
        li1 = __ldg(px + 1);
        li2 = __ldg(px + 2);
    }

    // forward over this thread's chunk; the samples and their taps' slots stay in registers
    float4 m[C];
    float Tloc[C];
    unsigned word[C];
    const unsigned base = rl_fast_base(qx, qy, W);
    const bool fast = __all_sync(0xffffffffu, rl_chunk_inside<ANCH>(w, sA, views, d0, d0 + n - 1, qx, qy, H, W, first));
    if (fast) {
#pragma unroll
        for (int i = C - 1; i >= 0; --i) {
            const int d = FULL ? d0 + i : d0 + min(i, n - 1);
            const RLFastTap t = rl_fast_tap<ANCH>(w, sA, first + d, views.rho[d], base, W);
            m[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            word[i] = 0xFFFFFFFFu;
            if (RL_IN((long long)t.idx + W + 1, hw)) {
                m[i] = rl_sample_at(M, (unsigned)d * hw + t.idx, W, t.fx, t.fy);
                if (SPARSE) word[i] = rl_slot_word(slots, (unsigned)d * hw + t.idx, W);
            }
            if (!FULL && i >= n) m[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    } else {
#pragma unroll
        for (int i = C - 1; i >= 0; --i) {
            word[i] = 0u;
            m[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (FULL || i < n) {
                const int d = d0 + i;
                m[i] = rl_sample(M + d * plane, H, W, w.taps(sA, first + d, views.rho[d], qx, qy));
            }
        }
    }
    float Tl = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
#pragma unroll
    for (int i = C - 1; i >= 0; --i) {
        Tloc[i] = Tl;
        const float a = Tl * m[i].w;
        c0 = fmaf(a, m[i].x, c0);
        c1 = fmaf(a, m[i].y, c1);
        c2 = fmaf(a, m[i].z, c2);
        Tl = Tl * (1.f - m[i].w);
    }
    const int wi = threadIdx.x >> 5, w0 = wi - pc.g;  // this tile's warps are w0 .. w0 + G - 1
    xch[wi][pc.lane] = make_float4(c0, c1, c2, Tl);
    if (img_early) {
        ximg[pc.tile][pc.lane][0] = li0;
        ximg[pc.tile][pc.lane][1] = li1;
        ximg[pc.tile][pc.lane][2] = li2;
    }
    __syncthreads();
    // combine the chunks, farthest first: the composite of everything behind this chunk, the
    // transmittance in front of it and the pixel colour
    float b0 = 0.f, b1 = 0.f, b2 = 0.f, Tb = 1.f;
#pragma unroll 4
    for (int g = w0; g < wi; ++g) {
        const float4 v = xch[g][pc.lane];
        b0 = fmaf(v.w, b0, v.x);
        b1 = fmaf(v.w, b1, v.y);
        b2 = fmaf(v.w, b2, v.z);
    }
    float C0 = fmaf(Tl, b0, c0), C1 = fmaf(Tl, b1, c1), C2 = fmaf(Tl, b2, c2);
#pragma unroll 4
    for (int g = wi + 1; g < w0 + pc.G; ++g) {
        const float4 v = xch[g][pc.lane];
        C0 = fmaf(v.w, C0, v.x);
        C1 = fmaf(v.w, C1, v.y);
        C2 = fmaf(v.w, C2, v.z);
        Tb = Tb * v.w;
    }
    float lsum = 0.f;
    float r0 = 0.f, r1 = 0.f, r2 = 0.f;
    if (pc.active) {
        if (LOSS) {
            const int s = 1 << img_level;
            float i0 = 0.f, i1 = 0.f, i2 = 0.f;
            if (img_level == 0) {
                i0 = ximg[pc.tile][pc.lane][0];
                i1 = ximg[pc.tile][pc.lane][1];
                i2 = ximg[pc.tile][pc.lane][2];
            } else {
                const int Wf = W << img_level, Hf = H << img_level;
                const float* img = images + (size_t)pc.view * Hf * Wf * 3;
                for (int yy = 0; yy < s; ++yy)
                    for (int xx = 0; xx < s; ++xx) {
                        const float* px = img + ((size_t)(pc.qy * s + yy) * Wf + (pc.qx * s + xx)) * 3;
                        i0 += __ldg(px);
                        i1 += __ldg(px + 1);
                        i2 += __ldg(px + 2);
                    }
            }
            const float inv_area = 1.f / (float)(s * s);
            // the image mean is rounded on its own (as the level images of the pyramid pass are)
            const float e0 = C0 - __fmul_rn(i0, inv_area), e1 = C1 - __fmul_rn(i1, inv_area),
                        e2 = C2 - __fmul_rn(i2, inv_area);
            lsum = fmaf(e0, e0, fmaf(e1, e1, e2 * e2));
            r0 = e0 * inv_n;
            r1 = e1 * inv_n;
            r2 = e2 * inv_n;
        } else {
            const float* go = grad_out + (((size_t)pc.view * H + pc.qy) * W + pc.qx) * 3;
            r0 = __ldg(go);
            r1 = __ldg(go + 1);
            r2 = __ldg(go + 2);
        }
    }
    // adjoint over the chunk, farthest plane first
    const unsigned ng = views.gplanes ? (unsigned)views.gplanes : (unsigned)D;  // checked in debug builds
    const unsigned act = __ballot_sync(0xffffffffu, pc.active);
    const bool join = !SPARSE && fast;  // a warp that lies inside joins its lanes' shared taps
    if (pc.active || join) {
#pragma unroll
        for (int i = 0; i < C; ++i) {
            if (FULL || i < n) {
                const int d = d0 + i;
                const float Td = Tb * Tloc[i];
                const float4 mi = m[i];
                const float gc = Td * mi.w;
                float4 g;
                g.x = gc * r0;
                g.y = gc * r1;
                g.z = gc * r2;
                g.w = Td * fmaf(mi.x - b0, r0, fmaf(mi.y - b1, r1, (mi.z - b2) * r2));
                if (join) {
                    const RLFastTap t = rl_fast_tap<ANCH>(w, sA, first + d, views.rho[d], base, W);
                    if (!pc.active || Td == 0.f) g = make_float4(0.f, 0.f, 0.f, 0.f);
                    join_taps(G, act, pc.lane, Td != 0.f, (unsigned)d, (unsigned)d * hw + t.idx, W, t.fx, t.fy, g, ng);
                } else if (Td != 0.f) {
                    if (fast) {  // the taps are formed again: keeping them costs registers, and warps
                        const RLFastTap t = rl_fast_tap<ANCH>(w, sA, first + d, views.rho[d], base, W);
                        rl_scatter_at<SPARSE>(G, word[i], (unsigned)d, t.idx, (unsigned)d * hw + t.idx, hw, W,
                                              rl_weights(t.fx, t.fy), g, ng);
                    } else {
                        const RLTaps t = w.taps(sA, first + d, views.rho[d], qx, qy);
                        if (t.ok) rl_scatter<SPARSE>(G, slots, (unsigned)d, hw, H, W, t, g, ng);
                    }
                }
                const float om = 1.f - mi.w;
                b0 = fmaf(mi.x, mi.w, om * b0);
                b1 = fmaf(mi.y, mi.w, om * b1);
                b2 = fmaf(mi.z, mi.w, om * b2);
            }
        }
    }
    // loss: one partial a tile, from the tile's first warp
    const int tiles_x = (W + sh.tile_x - 1) / sh.tile_x;
    if (LOSS && pc.g == 0 && pc.tile < sh.tiles && pc.tx < tiles_x) {
        lsum = rl_warp_sum(lsum);
        const unsigned part = ((unsigned)pc.ty * (unsigned)tiles_x + (unsigned)pc.tx) * (unsigned)views.n +
                              (unsigned)pc.view;
        if (pc.lane == 0 && RL_IN(part, nparts)) partials[part] = lsum;
    }
}

template <typename Tm, bool FULL, bool SPARSE, bool LOSS, bool ANCH>
__global__ void __launch_bounds__(kMaxWarps * kPix, 2)
k_grad_pp(const Tm* __restrict__ M, int D, int H, int W, const __grid_constant__ RLViews views, PPShape sh,
          const float* __restrict__ images, int img_level, const float* __restrict__ grad_out,
          const uint8_t* __restrict__ slots, float* __restrict__ G, float inv_n, float* __restrict__ partials,
          unsigned nparts) {
    // grid (views, blocks_x, tiles_y): the views of a tile run together and share M in L2
    grad_pp_tile<Tm, FULL, SPARSE, LOSS, ANCH>(M, D, H, W, views,
                                               pp_pos(H, W, blockIdx.x, blockIdx.y, blockIdx.z, sh), sh, blockIdx.y,
                                               images, img_level, grad_out, slots, G, inv_n, partials, nparts);
}

// One unit of the batch below: a block's tiles of one view of one item.  A function of its own, so that the
// loop's registers and the other kind of coordinates do not press on it (inlined, 32 to 48 bytes of spills
// a thread): two anchored requests of 2000x58, D = 32, 2 views, FP32: 298 against 308 us; six requests
// of 128x96, D = 32, 3 views: 118 against 127 us.
template <typename Tm, bool ANCH>
__device__ __noinline__ void grad_pp_unit(const RLBatchItem& it, unsigned local) {
    const unsigned view = local % (unsigned)it.N, block = local / (unsigned)it.N;
    const int h = it.H >> it.level, w = it.W >> it.level;
    const int bx = (int)(block % it.pp_tiles_x), by = (int)(block / it.pp_tiles_x);
    const PPShape sh = grad_pp_shape(it.D, h, w, kMaxWarps, ANCH);
    PPPos pc = pp_pos(h, w, (int)view, bx, by, sh);
    if (pc.tile >= sh.tiles) {  // a warp without a tile: a chunk of the first one, used by none
        pc.tx = bx * sh.tiles;
        pc.g = 0;
        pc.G = 1;
    }
    grad_pp_tile<Tm, false, true, true, ANCH>(static_cast<const Tm*>(it.Ml), it.D, h, w, it.views, pc, sh, bx,
                                              it.level ? it.Il : it.images, 0, nullptr, it.slots, it.G, it.inv_n,
                                              it.partials, it.parts);
}

// Batched gradient, plane-parallel family: one persistent launch of 16-warp blocks walks the
// gradient units of the batch table's items that take this family (a unit is one block's tiles of
// one view of one item).
template <typename Tm>
__global__ void __launch_bounds__(kMaxWarps * kPix, 2)
k_grad_pp_batch(const RLBatchHeader* __restrict__ hdr, const RLBatchItem* __restrict__ items) {
    const unsigned n = hdr->n, total = hdr->pp_units;
    if (hdr->dtype != (std::is_same<Tm, float>::value ? (unsigned)RL_F32 : (unsigned)RL_BF16)) return;
    __shared__ unsigned next_slot;
    for (unsigned u = rl_batch_next(hdr, 2, &next_slot); u < total; u = rl_batch_next(hdr, 2, &next_slot)) {
        const RLBatchItem& it = items[rl_batch_find(items, n, u, &RLBatchItem::pp_begin)];
        if (it.views.anchored) grad_pp_unit<Tm, true>(it, u - it.pp_begin);
        else grad_pp_unit<Tm, false>(it, u - it.pp_begin);
        __syncthreads();  // the exchange buffers are reused by the next unit
    }
}

// planes per thread for D planes over G warps: the next of 1, 2, 4, 8 >= ceil(D / G)
int chunk_for(int D, int G) {
    const int c = (D + G - 1) / G;
    return c <= 1 ? 1 : c <= 2 ? 2 : c <= 4 ? 4 : 8;
}

// Warps per block of the render: 8 (measured faster than 4 at D = 32 despite the chunk combination
// being amortised over fewer planes); kernel path 4 forces 4 where D <= 32 (at most 8 planes per
// thread).
int groups_for(int D, int path) {
    return (path == 4 && D <= 32) ? 4 : 8;
}

template <typename Tm, bool SPARSE, bool LOSS>
void launch_grad_pp_t(const PPShape sh, const void* M, int D, int H, int W, const RLViews& views, const float* images,
                      int img_level, const float* grad_out, const uint8_t* slots, float* G, float inv_n,
                      float* partials, unsigned nparts, cudaStream_t s) {
    const int per = sh.tile_x * sh.tiles, rows = kPix / sh.tile_x;
    const dim3 grid((unsigned)views.n, (unsigned)((W + per - 1) / per), (unsigned)((H + rows - 1) / rows));
    const unsigned threads = (unsigned)(sh.G * sh.tiles * kPix);
#define RL_PP_LAUNCH(FULL, A)                                                                                       \
    k_grad_pp<Tm, FULL, SPARSE, LOSS, A><<<grid, threads, 0, s>>>((const Tm*)M, D, H, W, views, sh, images,        \
                                                                  img_level, grad_out, slots, G, inv_n, partials, nparts)
    if (D % kChunk == 0) { if (views.anchored) RL_PP_LAUNCH(true, true); else RL_PP_LAUNCH(true, false); }
    else { if (views.anchored) RL_PP_LAUNCH(false, true); else RL_PP_LAUNCH(false, false); }
#undef RL_PP_LAUNCH
}

template <typename Tm>
void launch_render_pp_t(int G, int C, const void* M, int D, int H, int W, const RLViews& views, int tiles_x,
                        dim3 grid, float* out, cudaStream_t s) {
#define RL_PP_LAUNCH(CC, GG) \
    k_render_pp<Tm, CC, GG, false><<<grid, GG * kPix, 0, s>>>((const Tm*)M, D, H, W, views, tiles_x, out)
#define RL_PP_LAUNCH_A(CC) \
    k_render_pp<Tm, CC, 8, true><<<grid, 8 * kPix, 0, s>>>((const Tm*)M, D, H, W, views, tiles_x, out)
    if (views.anchored) {
        switch (C) {
            case 1: RL_PP_LAUNCH_A(1); break;
            case 2: RL_PP_LAUNCH_A(2); break;
            case 4: RL_PP_LAUNCH_A(4); break;
            default: RL_PP_LAUNCH_A(8); break;
        }
    } else if (G == 4) {
        switch (C) {
            case 1: RL_PP_LAUNCH(1, 4); break;
            case 2: RL_PP_LAUNCH(2, 4); break;
            case 4: RL_PP_LAUNCH(4, 4); break;
            default: RL_PP_LAUNCH(8, 4); break;
        }
    } else {
        switch (C) {
            case 1: RL_PP_LAUNCH(1, 8); break;
            case 2: RL_PP_LAUNCH(2, 8); break;
            case 4: RL_PP_LAUNCH(4, 8); break;
            default: RL_PP_LAUNCH(8, 8); break;
        }
    }
#undef RL_PP_LAUNCH
}

}  // namespace

// Share of an SM's 32 warps (64 registers) that hold planes in a launch of D planes: blocks of G x tiles warps
// fill the SM only in part, and the last chunk of a tile may be short.
double rl_grad_pp_fill(int D) {
    const PPShape s = grad_pp_shape(D, 1, 1, 8, false);
    const int warps = s.G * s.tiles;
    return (double)(32 / warps * warps) / 32.0 * D / (s.G * kChunk);
}

// Tiles of a gradient launch over all views: the loss partials it writes.
size_t rl_grad_pp_num_blocks(int H, int W, int N, bool anchored) {
    const int tx = grad_pp_tile_x(H, W, anchored), ty = kPix / tx;
    return (size_t)((W + tx - 1) / tx) * ((H + ty - 1) / ty) * N;
}

rl_status rl_launch_grad_pp(const void* M, rl_dtype dt, int D, int H, int W, const RLViews& views, bool mode_loss,
                            const float* images, int img_level, const float* grad_out, const uint8_t* slots,
                            float* G_out, float inv_n, float* partials, int* nblocks, cudaStream_t s) {
    // kernel path 4 asks for narrower blocks
    const bool anchored = views.anchored != 0;
    const PPShape sh = grad_pp_shape(D, H, W, rl_kernel_path_setting() == 4 ? 4 : 8, anchored);
    const unsigned nparts = (unsigned)rl_grad_pp_num_blocks(H, W, views.n, anchored);
    if (nblocks) *nblocks = (int)nparts;
    const bool sparse = slots != nullptr;
    const char* name = dt == RL_F32 ? (sparse ? "grad_sparse_f32" : "grad_dense_f32")
                                    : (sparse ? "grad_sparse_bf16" : "grad_dense_bf16");
    RLTraceScope ts(name, s);
#define RL_CASE(TM, SP, LS) \
    launch_grad_pp_t<TM, SP, LS>(sh, M, D, H, W, views, images, img_level, grad_out, slots, G_out, inv_n, partials, \
                                 nparts, s)
    // a slot map comes with the loss mode only
#define RL_KIND(TM)                                                                               \
    do {                                                                                          \
        if (slots) RL_CASE(TM, true, true);                                                      \
        else if (mode_loss) RL_CASE(TM, false, true);                                            \
        else RL_CASE(TM, false, false);                                                          \
    } while (0)
    if (dt == RL_F32) RL_KIND(float);
    else RL_KIND(__nv_bfloat16);
#undef RL_KIND
#undef RL_CASE
    return rl_check_launch("grad_pp");
}

rl_status rl_launch_render_pp(const void* M, rl_dtype dt, int D, int H, int W, const RLViews& views, float* out,
                              cudaStream_t s) {
    const int tiles_x = (W + kTX - 1) / kTX;
    const dim3 grid((unsigned)views.n, (unsigned)tiles_x, (unsigned)((H + kTY - 1) / kTY));
    const int G = views.anchored ? 8 : groups_for(D, rl_kernel_path_setting());
    const int C = chunk_for(D, G);
    if (dt == RL_F32) {
        RLTraceScope ts("render_f32", s);
        launch_render_pp_t<float>(G, C, M, D, H, W, views, tiles_x, grid, out, s);
    } else {
        RLTraceScope ts("render_bf16", s);
        launch_render_pp_t<__nv_bfloat16>(G, C, M, D, H, W, views, tiles_x, grid, out, s);
    }
    return rl_check_launch("render_pp");
}

unsigned rl_grad_pp_tiles_x(int h, int w, int D, bool anchored) {
    const PPShape sh = grad_pp_shape(D, h, w, kMaxWarps, anchored);
    const int per = sh.tile_x * sh.tiles;
    return (unsigned)((w + per - 1) / per);
}
unsigned rl_grad_pp_tiles_y(int h, int w, bool anchored) {
    const int rows = kPix / grad_pp_tile_x(h, w, anchored);
    return (unsigned)((h + rows - 1) / rows);
}

rl_status rl_launch_grad_pp_batch(const void* table, rl_dtype dt, cudaStream_t s) {
    const RLBatchHeader* hdr = static_cast<const RLBatchHeader*>(table);
    const RLBatchItem* items = rl_batch_items(table);
    const int grid = dt == RL_F32 ? rl_persistent_grid<k_grad_pp_batch<float>>(kMaxWarps * kPix, 0)
                                  : rl_persistent_grid<k_grad_pp_batch<__nv_bfloat16>>(kMaxWarps * kPix, 0);
    if (dt == RL_F32) {
        RLTraceScope ts("grad_pp_batch_f32", s);
        k_grad_pp_batch<float><<<grid, kMaxWarps * kPix, 0, s>>>(hdr, items);
    } else {
        RLTraceScope ts("grad_pp_batch_bf16", s);
        k_grad_pp_batch<__nv_bfloat16><<<grid, kMaxWarps * kPix, 0, s>>>(hdr, items);
    }
    return rl_check_launch("grad_pp_batch");
}

RL_DEBUG_READER(pp)
