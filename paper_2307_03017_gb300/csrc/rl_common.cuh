// rl_common.cuh -- device-side building blocks shared by the RealLiFe kernels (sm_103a).
//
// Warp geometry.  For a view camera v and the reference camera r, let R_rel = R_v R_r^T and
// C the view's centre in the reference frame.  The ray of view pixel q = (u, v) has
// reference-frame direction dir = R_rel^T K_v^{-1} (u, v, 1); it meets the fronto-parallel
// plane z = 1/rho at the reference pixel
//     p = q + a(q) + rho * b(q),
//     a_x = (cx_r - cx_v) + (fx_r - fx_v) m_x + fx_r (dir_x/dir_z - m_x),
//     b_x = fx_r (C_x - C_z dir_x/dir_z),         (same for y)
// with m = K_v^{-1} q.  This is the inverse of the plane-induced homography of Eq. (eq_homo)
// written per pixel: exact, linear in inverse depth, and evaluated as small offsets from q
// so that FP32 keeps ~1e-6 px of accuracy at 2k-pixel coordinates.  The plane is met in
// front of the view iff dir_z > 0 and 1 - rho C_z > 0.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#define RL_DEV_MAX_PLANES 64
#define RL_DEV_MAX_VIEWS 16

// Bounds checks of the debug build (-DRL_DEBUG, built by build.py as libreallife_debug.so):
// the hot kernels check the computed index of each global access against its buffer before
// the access; a failed check sets RL_DEVFLAG_BOUNDS in the translation unit's debug word and
// skips the access, never a trap.  reallife_device_status reports the words of every
// translation unit.  In the release build RL_IN is `true` and costs nothing.
#define RL_DEVFLAG_BOUNDS 4u
#ifdef RL_DEBUG
static __device__ unsigned int rl_dbg_word;  // one per translation unit
__device__ __forceinline__ bool rl_dbg_in(long long i, long long n) {
    if (i >= 0 && i < n) return true;
    atomicOr(&rl_dbg_word, RL_DEVFLAG_BOUNDS);
    return false;
}
#define RL_IN(i, n) rl_dbg_in((long long)(i), (long long)(n))
// Host reader of this translation unit's debug word (defined once per .cu by the macro).
#define RL_DEBUG_READER(name)                                                       \
    unsigned int rl_dbg_read_##name(int clear) {                                    \
        unsigned int v = 0;                                                         \
        if (cudaMemcpyFromSymbol(&v, rl_dbg_word, sizeof(v)) != cudaSuccess) {      \
            cudaGetLastError();                                                     \
            return 0;                                                               \
        }                                                                           \
        if (clear) {                                                                \
            const unsigned int z = 0;                                               \
            if (cudaMemcpyToSymbol(rl_dbg_word, &z, sizeof(z)) != cudaSuccess) cudaGetLastError(); \
        }                                                                           \
        return v;                                                                   \
    }
#else
#define RL_IN(i, n) true
#define RL_DEBUG_READER(name) \
    unsigned int rl_dbg_read_##name(int) { return 0; }
#endif

struct RLViewParam {
    float E[9];          // R_rel^T - I (row-major)
    float C[3];          // view centre in the reference frame
    float inv_fxv, inv_fyv, cxv, cyv;
    float fxr, fyr;      // reference focal lengths
    float dcx, dcy;      // cx_r - cx_v, cy_r - cy_v
    float dfx, dfy;      // fx_r - fx_v, fy_r - fy_v
};

// The same parameters in FP64, for the per-block anchors below.
struct RLViewParam64 {
    double E[9], C[3];
    double inv_fxv, inv_fyv, cxv, cyv, fxr, fyr, dcx, dcy, dfx, dfy;
};

// Views and plane inverse depths of one launch, passed by value as a kernel parameter.
struct RLViews {
    int n;
    int anchored;  // 1: the kernels take the anchored coordinates below (offsets beyond ~128 px)
    float rho[RL_DEV_MAX_PLANES];
    RLViewParam v[RL_DEV_MAX_VIEWS];
    double rho64[RL_DEV_MAX_PLANES];
    RLViewParam64 v64[RL_DEV_MAX_VIEWS];
    int gplanes;  // planes of the gradient buffer a launch scatters into (0: D); debug-build bounds checks
    int shifts;   // 1: every view is a pure shift of the reference (rl_views_are_shifts)
};

// ------------------------------------------------------------------ batch work tables
//
// A batch table serves one HSGD iteration of many requests in one launch per stage
// (selection, gradient, update).  It is a header followed by one item per request, in device
// memory; the persistent batched kernels take fixed grids and walk the work units of all items
// (a unit is one block's worth of work of one item), so one captured launch serves any table.

#define RL_DEVFLAG_BATCH 2u  // a batched kernel was given a table of another storage type

struct RLBatchHeader {
    unsigned n;                                // items
    unsigned dtype;                            // rl_dtype of every item's MPI
    unsigned sel_units, grad_units, upd_units;  // work units of the stages (gradient: gather family)
    unsigned pp_units;                         // gradient units of the plane-parallel family
    unsigned int* status;                      // device status word
    unsigned max_gather_D;                     // largest D among the gather family's items
    unsigned next[4];                          // next unit of each launch (0 in the copied table)
    unsigned pad1[3];
};

// The next work unit of a persistent batched launch for the calling block: taken from the
// launch's counter in the table header, so that blocks finishing early take more units.
// Every thread of the block calls it; `slot` is block-shared scratch.
__device__ __forceinline__ unsigned rl_batch_next(const RLBatchHeader* hdr, int which, unsigned* slot) {
    __syncthreads();  // the previous unit's readers of *slot are done
    if (threadIdx.x == 0 && threadIdx.y == 0)
        *slot = atomicAdd(const_cast<unsigned*>(&hdr->next[which]), 1u);
    __syncthreads();
    return *slot;
}

struct RLBatchItem {
    void* M;                 // full-resolution MPI [D][H][W][4], refined in place
    void* Ml;                // level-l MPI (M itself at level 0)
    const float* images;     // full-resolution source images [N][H][W][3]
    uint8_t* S;              // selection [k][h][w]
    uint8_t* slots;          // slot map [D][h][w]
    float* G;                // compact gradient [k][h][w][4]
    float* partials;         // loss partials, one per gradient unit
    float* loss_out;         // device [1] or NULL
    float* Il;               // level-l source images [N][h][w][3] (levels >= 1; written by the selection)
    int D, H, W, level, k, mode, clamp01, N;
    float lambda, prior_scale, inv_n, loss_scale;
    unsigned sel_begin, sel_units;    // first unit and unit count of each stage
    unsigned grad_begin, grad_units, grad_tiles_x;   // gather family (units 0 for the other items)
    unsigned pp_begin, pp_units, pp_tiles_x;         // plane-parallel family (units 0 for the others)
    unsigned upd_begin, upd_units, upd_tiles_x;
    unsigned parts;          // loss partials of the item's gradient
    RLViews views;           // level-l warp parameters of the N views and the plane inverse depths
};

__host__ __device__ inline const RLBatchItem* rl_batch_items(const void* table) {
    return reinterpret_cast<const RLBatchItem*>(static_cast<const char*>(table) + sizeof(RLBatchHeader));
}

// Item owning work unit u of a stage whose first units are items[i].*begin (ascending).
__device__ __forceinline__ unsigned rl_batch_find(const RLBatchItem* __restrict__ items, unsigned n, unsigned u,
                                                  unsigned RLBatchItem::*begin) {
    unsigned lo = 0, hi = n - 1;
    while (lo < hi) {
        const unsigned mid = (lo + hi + 1) >> 1;
        if (items[mid].*begin <= u) lo = mid;
        else hi = mid - 1;
    }
    return RL_IN(lo, n) ? lo : 0;
}

// Per-pixel warp coefficients of one view.
struct RLWarp {
    float ax, ay, bx, by, cz;
    bool dir_ok;
};

__device__ __forceinline__ RLWarp rl_warp_coeffs(const RLViewParam& P, float u, float v) {
    RLWarp w;
    float mx = (u - P.cxv) * P.inv_fxv;
    float my = (v - P.cyv) * P.inv_fyv;
    float ex = fmaf(P.E[0], mx, fmaf(P.E[1], my, P.E[2]));
    float ey = fmaf(P.E[3], mx, fmaf(P.E[4], my, P.E[5]));
    float ez = fmaf(P.E[6], mx, fmaf(P.E[7], my, P.E[8]));
    float dz = 1.0f + ez;
    float inv_dz = 1.0f / dz;
    // r - m = (e - m e_z) / dir_z : small, computed without cancellation
    float rmx = fmaf(-mx, ez, ex) * inv_dz;
    float rmy = fmaf(-my, ez, ey) * inv_dz;
    float rx = mx + rmx, ry = my + rmy;
    w.ax = P.dcx + fmaf(P.dfx, mx, P.fxr * rmx);
    w.ay = P.dcy + fmaf(P.dfy, my, P.fyr * rmy);
    w.bx = P.fxr * fmaf(-P.C[2], rx, P.C[0]);
    w.by = P.fyr * fmaf(-P.C[2], ry, P.C[1]);
    w.cz = P.C[2];
    w.dir_ok = dz > 0.0f;
    return w;
}

// Bilinear footprint of one sample: top-left tap (x0, y0) and fractional offsets.
struct RLTaps {
    int x0, y0;
    float fx, fy;
    bool ok;  // plane met in front of the view
};

__device__ __forceinline__ RLTaps rl_taps(const RLWarp& w, float rho, int qx, int qy) {
    RLTaps t;
    float dx = fmaf(rho, w.bx, w.ax);
    float dy = fmaf(rho, w.by, w.ay);
    float flx = floorf(dx), fly = floorf(dy);
    t.fx = dx - flx;  // exact
    t.fy = dy - fly;
    t.x0 = qx + (int)flx;
    t.y0 = qy + (int)fly;
    t.ok = w.dir_ok && (fmaf(-rho, w.cz, 1.0f) > 0.0f) && fabsf(dx) < 1.0e7f && fabsf(dy) < 1.0e7f;
    return t;
}

// ------------------------------------------------------------------ anchored warp coordinates
//
// The offset p - q = a(q) + rho_d b(q) reaches hundreds of pixels for wide baselines and
// rotated views (|a|, |b| up to ~400 px at 1920 x 1080), where FP32 spacing is ~3e-5 px.  So
// each block evaluates the warp once at an anchor pixel q_c in FP64 and keeps, for every
// plane, the offset at the anchor split into an integer and an FP32 fraction; a pixel of the
// block adds the small FP32 differences a(q) - a(q_c) and b(q) - b(q_c), formed without
// cancellation (exact algebra, small terms only):
//   dm = K_v^{-1} (q - q_c),  de = (R_rel^T - I) dm,
//   dN = de_xy - m_c de_z - dm (e_zc + de_z),   N = e_xy - m e_z,  Dn = 1 + e_z,
//   r_m(q) - r_m(q_c) = (dN Dc - N_c de_z) / (Dn Dc),
//   a(q) - a(q_c) = (f_r - f_v) dm + f_r (r_m(q) - r_m(q_c)),
//   b(q) - b(q_c) = -f_r C_z (dm + r_m(q) - r_m(q_c)).
// The sample position's error stays near 1e-7 px at any image size.  The plane is met in
// front of the view iff 1 - rho_d C_z > 0 (per plane) and the pixel's ray points into the
// reference frame's half-space, 1 + e_z > 0; the host rejects views whose rays at the image
// corners run nearly parallel to the planes, so the anchors are always valid.
//
// The per-pixel FP32 coefficients of rl_warp_coeffs carry an error near 1.2e-7 times the
// offset (measured against the FP64 ray/plane intersection): ~1e-5 px at 100 px.  The host
// therefore takes the anchored path only for launches whose offsets exceed 128 px anywhere
// (RLViews::anchored), where the per-block FP64 set-up pays for itself in accuracy; the
// kernels are compiled for both paths.

struct RLPlaneK {
    float fx, fy;  // fraction of the anchor's offset on plane d
    int ix, iy;    // integer part (plane not met in front of the view: ix = RL_PLANE_NONE)
};
#define RL_PLANE_NONE (-0x40000000)

// What a sample known to lie inside the plane needs of plane d, in one 16-byte load: the fraction,
// the integer part as a voxel offset iy W + ix, and the plane's inverse depth.
struct RLPlaneF {
    float fx, fy;
    int off;
    float rho;
};

struct RLAnchorHead {
    float mx, my, ez, Nx, Ny, Dc;  // anchor quantities (FP32) for the per-pixel differences
    int u, v;                      // anchor pixel
};

struct RLAnchor : RLAnchorHead {
    RLPlaneK k[RL_DEV_MAX_PLANES];
    RLPlaneF f[RL_DEV_MAX_PLANES];
};

// The head of the anchor at pixel (u, v) of view P; ab: the offset's coefficients there, a(q_c) and
// b(q_c), for rl_anchor_plane.
__device__ __forceinline__ void rl_anchor_head(RLAnchorHead* A, double* ab, const RLViewParam64& P, int u, int v) {
    const double mx = ((double)u - P.cxv) * P.inv_fxv, my = ((double)v - P.cyv) * P.inv_fyv;
    const double ex = P.E[0] * mx + P.E[1] * my + P.E[2];
    const double ey = P.E[3] * mx + P.E[4] * my + P.E[5];
    const double ez = P.E[6] * mx + P.E[7] * my + P.E[8];
    const double dz = 1.0 + ez;
    const double Nx = ex - mx * ez, Ny = ey - my * ez;
    // 1 / dz: the FP32 reciprocal refined by two Newton steps in FP64 (relative error far
    // below FP64's 1e-16 after the second), cheaper than an FP64 division on this GPU
    double inv = (double)__frcp_rn((float)dz);
    inv = inv * (2.0 - dz * inv);
    inv = inv * (2.0 - dz * inv);
    const double rmx = Nx * inv, rmy = Ny * inv;
    ab[0] = P.dcx + P.dfx * mx + P.fxr * rmx;
    ab[1] = P.dcy + P.dfy * my + P.fyr * rmy;
    ab[2] = P.fxr * (P.C[0] - P.C[2] * (mx + rmx));
    ab[3] = P.fyr * (P.C[1] - P.C[2] * (my + rmy));
    A->mx = (float)mx;
    A->my = (float)my;
    A->ez = (float)ez;
    A->Nx = (float)Nx;
    A->Ny = (float)Ny;
    A->Dc = (float)dz;
    A->u = u;
    A->v = v;
}

// The entries k, f of plane d (inverse depth V.rho64[d]) of the anchor with coefficients ab; W the plane's width.
__device__ __forceinline__ void rl_anchor_plane(RLPlaneK* kd, RLPlaneF* fd, const double* ab, const RLViews& V,
                                                const RLViewParam64& P, int d, int W) {
    const double rho = V.rho64[d];
    const double kx = ab[0] + rho * ab[2], ky = ab[1] + rho * ab[3];
    RLPlaneK k;
    if (1.0 - rho * P.C[2] > 0.0 && fabs(kx) < 1e9 && fabs(ky) < 1e9) {
        const double fx = floor(kx), fy = floor(ky);
        k.ix = (int)fx;
        k.iy = (int)fy;
        k.fx = (float)(kx - fx);
        k.fy = (float)(ky - fy);
    } else {
        k.ix = k.iy = RL_PLANE_NONE;
        k.fx = k.fy = 0.f;
    }
    *kd = k;
    *fd = RLPlaneF{k.fx, k.fy, (int)((unsigned)k.iy * (unsigned)W + (unsigned)k.ix), V.rho[d]};
}

// Fills A (shared memory) for view `view` of V at anchor pixel (u, v).  Every thread of the
// block calls it (it synchronises the block twice); nthreads threads, index tid; W the plane's width.
__device__ __forceinline__ void rl_anchor_build(RLAnchor* A, const RLViews& V, int view, int u, int v, int D, int W,
                                                int tid, int nthreads) {
    __shared__ double s_ab[4];
    const RLViewParam64& P = V.v64[view];
    if (tid == 0) rl_anchor_head(A, s_ab, P, u, v);
    __syncthreads();
    for (int d = tid; d < D; d += nthreads) rl_anchor_plane(A->k + d, A->f + d, s_ab, V, P, d, W);
    __syncthreads();
}

// Per-pixel differences from the anchor.
struct RLAnchorPix {
    float dax, day, dbx, dby;
    bool ok;  // the pixel's ray points into the reference half-space and its offsets are bounded
};

__device__ __forceinline__ RLAnchorPix rl_anchor_pixel(const RLAnchorHead& A, const RLViewParam& P, int qx, int qy) {
    RLAnchorPix w;
    const float dmx = (float)(qx - A.u) * P.inv_fxv, dmy = (float)(qy - A.v) * P.inv_fyv;
    const float dex = fmaf(P.E[0], dmx, P.E[1] * dmy);
    const float dey = fmaf(P.E[3], dmx, P.E[4] * dmy);
    const float dez = fmaf(P.E[6], dmx, P.E[7] * dmy);
    const float ez = A.ez + dez;
    const float dNx = dex - fmaf(A.mx, dez, dmx * ez);
    const float dNy = dey - fmaf(A.my, dez, dmy * ez);
    const float Dn = A.Dc + dez;
    const float inv = 1.0f / (Dn * A.Dc);
    const float drx = fmaf(dNx, A.Dc, -A.Nx * dez) * inv;
    const float dry = fmaf(dNy, A.Dc, -A.Ny * dez) * inv;
    w.dax = fmaf(P.dfx, dmx, P.fxr * drx);
    w.day = fmaf(P.dfy, dmy, P.fyr * dry);
    w.dbx = -P.fxr * P.C[2] * (dmx + drx);
    w.dby = -P.fyr * P.C[2] * (dmy + dry);
    w.ok = Dn > 0.f && fabsf(w.dax) + fabsf(w.dbx) < 1.0e6f && fabsf(w.day) + fabsf(w.dby) < 1.0e6f;
    return w;
}

// Taps of plane d (inverse depth rho, its FP32 value) at view pixel (qx, qy).
__device__ __forceinline__ RLTaps rl_anchor_taps(const RLAnchor& A, const RLAnchorPix& w, int d, float rho, int qx,
                                                 int qy) {
    const RLPlaneK k = A.k[d];
    RLTaps t;
    const float sx = k.fx + fmaf(rho, w.dbx, w.dax), sy = k.fy + fmaf(rho, w.dby, w.day);
    const float flx = floorf(sx), fly = floorf(sy);
    t.fx = sx - flx;
    t.fy = sy - fly;
    t.x0 = qx + k.ix + (int)flx;
    t.y0 = qy + k.iy + (int)fly;
    t.ok = w.ok && k.ix != RL_PLANE_NONE;
    return t;
}

// Warp state of one view pixel for either coordinate path (ANCH: the block's anchor A).
template <bool ANCH>
struct RLPixWarp;

template <>
struct RLPixWarp<false> {
    RLWarp w;
    __device__ __forceinline__ RLTaps taps(const RLAnchor&, int, float rho, int qx, int qy) const {
        return rl_taps(w, rho, qx, qy);
    }
};

template <>
struct RLPixWarp<true> {
    RLAnchorPix w;
    __device__ __forceinline__ RLTaps taps(const RLAnchor& A, int d, float rho, int qx, int qy) const {
        return rl_anchor_taps(A, w, d, rho, qx, qy);
    }
};

template <bool ANCH>
__device__ __forceinline__ RLPixWarp<ANCH> rl_pix_warp(const RLAnchorHead& A, const RLViewParam& P, int qx, int qy) {
    RLPixWarp<ANCH> r;
    if constexpr (ANCH)
        r.w = rl_anchor_pixel(A, P, qx, qy);
    else
        r.w = rl_warp_coeffs(P, (float)qx, (float)qy);
    return r;
}

// Inverse warp (reference -> view, the direction of Eq. eq_homo's H^{-1}).  The reference
// pixel (u, v) on the plane of inverse depth rho has reference-frame direction
// m = K_r^{-1}(u, v, 1); in the view camera it lies along R_rel m + rho t_rel, with
// R_rel = R_v R_r^T and t_rel = t_v - R_rel t_r.  Writing R_rel = I + F and e = F m:
//     x = u + (cx_v - cx_r) + (fx_v - fx_r) m_x + fx_v (e_x - m_x e_z + rho (t_x - m_x t_z)) / Z,
//     Z = 1 + e_z + rho t_z,                                            (same for y)
// and the point is in front of the view iff Z > 0.  As for the forward warp, the offset
// from u is formed from small terms only.
struct RLInvParam {
    float F[9];          // R_rel - I (row-major)
    float t[3];          // t_rel
    float inv_fxr, inv_fyr, cxr, cyr;
    float fxv, fyv;
    float dcx, dcy;      // cx_v - cx_r, cy_v - cy_r
    float dfx, dfy;      // fx_v - fx_r, fy_v - fy_r
};

// Inverse-warp parameters of one launch (level-l and full-resolution cameras of each view).
struct RLInvViews {
    int n;
    float rho[RL_DEV_MAX_PLANES];
    RLInvParam lv[RL_DEV_MAX_VIEWS];
    RLInvParam full[RL_DEV_MAX_VIEWS];
};

// Per-pixel inverse-warp coefficients: offset = a + f_v (g + rho h) / (z0 + rho tz).
struct RLInvWarp {
    float gx, gy, hx, hy, z0, tz, ax, ay;
};

__device__ __forceinline__ RLInvWarp rl_inv_coeffs(const RLInvParam& P, float u, float v) {
    RLInvWarp c;
    const float mx = (u - P.cxr) * P.inv_fxr;
    const float my = (v - P.cyr) * P.inv_fyr;
    const float ex = fmaf(P.F[0], mx, fmaf(P.F[1], my, P.F[2]));
    const float ey = fmaf(P.F[3], mx, fmaf(P.F[4], my, P.F[5]));
    const float ez = fmaf(P.F[6], mx, fmaf(P.F[7], my, P.F[8]));
    c.gx = fmaf(-mx, ez, ex);
    c.gy = fmaf(-my, ez, ey);
    c.hx = fmaf(-mx, P.t[2], P.t[0]);
    c.hy = fmaf(-my, P.t[2], P.t[1]);
    c.z0 = 1.0f + ez;
    c.tz = P.t[2];
    c.ax = fmaf(P.dfx, mx, P.dcx);
    c.ay = fmaf(P.dfy, my, P.dcy);
    return c;
}

__device__ __forceinline__ RLTaps rl_inv_taps(const RLInvWarp& c, const RLInvParam& P, float rho, int u, int v) {
    RLTaps t;
    const float Z = fmaf(rho, c.tz, c.z0);
    const float inv = 1.0f / Z;
    const float dx = fmaf(P.fxv, fmaf(rho, c.hx, c.gx) * inv, c.ax);
    const float dy = fmaf(P.fyv, fmaf(rho, c.hy, c.gy) * inv, c.ay);
    const float flx = floorf(dx), fly = floorf(dy);
    t.fx = dx - flx;
    t.fy = dy - fly;
    t.x0 = u + (int)flx;
    t.y0 = v + (int)fly;
    t.ok = Z > 0.0f && fabsf(dx) < 1.0e7f && fabsf(dy) < 1.0e7f;
    return t;
}

// ---------------------------------------------------------------- storage types

template <typename T> struct RLStore;

template <> struct RLStore<float> {
    static __device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
    static __device__ __forceinline__ float4 load4_nc(const float* p) { return *reinterpret_cast<const float4*>(p); }
    static __device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
    static __device__ __forceinline__ float load1(const float* p) { return __ldg(p); }
    static __device__ __forceinline__ void store1(float* p, float v) { *p = v; }
    static __device__ __forceinline__ float round1(float v) { return v; }
};

template <> struct RLStore<__nv_bfloat16> {
    static __device__ __forceinline__ float4 cvt(uint2 r) {
        float4 o;
        o.x = __uint_as_float(r.x << 16);
        o.y = __uint_as_float(r.x & 0xffff0000u);
        o.z = __uint_as_float(r.y << 16);
        o.w = __uint_as_float(r.y & 0xffff0000u);
        return o;
    }
    static __device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
        return cvt(__ldg(reinterpret_cast<const uint2*>(p)));
    }
    static __device__ __forceinline__ float4 load4_nc(const __nv_bfloat16* p) {
        return cvt(*reinterpret_cast<const uint2*>(p));
    }
    static __device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v) {
        __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y);  // round to nearest even
        __nv_bfloat162 hi = __floats2bfloat162_rn(v.z, v.w);
        uint2 r;
        r.x = *reinterpret_cast<uint32_t*>(&lo);
        r.y = *reinterpret_cast<uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(p) = r;
    }
    static __device__ __forceinline__ float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void store1(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
    // the value a store of v would hold
    static __device__ __forceinline__ float round1(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
};

// Bilinear sample (zero padding per tap) of plane `plane` (base pointer of [H][W][4]).
template <typename Tm>
__device__ __forceinline__ float4 rl_sample(const Tm* __restrict__ plane, int H, int W, const RLTaps& t) {
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!t.ok) return acc;
    const float w00 = (1.f - t.fx) * (1.f - t.fy), w10 = t.fx * (1.f - t.fy);
    const float w01 = (1.f - t.fx) * t.fy, w11 = t.fx * t.fy;
    const bool x0in = (unsigned)t.x0 < (unsigned)W, x1in = (unsigned)(t.x0 + 1) < (unsigned)W;
    const bool y0in = (unsigned)t.y0 < (unsigned)H, y1in = (unsigned)(t.y0 + 1) < (unsigned)H;
    const size_t r0 = (size_t)t.y0 * W, r1 = r0 + W, hw = (size_t)H * W;
    if (y0in) {
        if (x0in && RL_IN(r0 + t.x0, hw)) { float4 v = RLStore<Tm>::load4(plane + (r0 + t.x0) * 4); acc.x = fmaf(w00, v.x, acc.x); acc.y = fmaf(w00, v.y, acc.y); acc.z = fmaf(w00, v.z, acc.z); acc.w = fmaf(w00, v.w, acc.w); }
        if (x1in && RL_IN(r0 + t.x0 + 1, hw)) { float4 v = RLStore<Tm>::load4(plane + (r0 + t.x0 + 1) * 4); acc.x = fmaf(w10, v.x, acc.x); acc.y = fmaf(w10, v.y, acc.y); acc.z = fmaf(w10, v.z, acc.z); acc.w = fmaf(w10, v.w, acc.w); }
    }
    if (y1in) {
        if (x0in && RL_IN(r1 + t.x0, hw)) { float4 v = RLStore<Tm>::load4(plane + (r1 + t.x0) * 4); acc.x = fmaf(w01, v.x, acc.x); acc.y = fmaf(w01, v.y, acc.y); acc.z = fmaf(w01, v.z, acc.z); acc.w = fmaf(w01, v.w, acc.w); }
        if (x1in && RL_IN(r1 + t.x0 + 1, hw)) { float4 v = RLStore<Tm>::load4(plane + (r1 + t.x0 + 1) * 4); acc.x = fmaf(w11, v.x, acc.x); acc.y = fmaf(w11, v.y, acc.y); acc.z = fmaf(w11, v.z, acc.z); acc.w = fmaf(w11, v.w, acc.w); }
    }
    return acc;
}

// Same sample as rl_sample; when all four taps are inside the plane (the common case) it
// skips the per-tap checks and addresses the taps with 32-bit offsets (D*H*W*4 < 2^31).
template <typename Tm>
__device__ __forceinline__ float4 rl_sample_fast(const Tm* __restrict__ plane, int H, int W, const RLTaps& t) {
    if (t.ok && (unsigned)t.x0 < (unsigned)(W - 1) && (unsigned)t.y0 < (unsigned)(H - 1) &&
        RL_IN((long long)t.y0 * W + t.x0 + W + 1, (long long)H * W)) {
        const Tm* p = plane + (unsigned)(t.y0 * W + t.x0) * 4u;
        const float4 v00 = RLStore<Tm>::load4(p), v10 = RLStore<Tm>::load4(p + 4);
        const float4 v01 = RLStore<Tm>::load4(p + 4 * W), v11 = RLStore<Tm>::load4(p + 4 * W + 4);
        const float w00 = (1.f - t.fx) * (1.f - t.fy), w10 = t.fx * (1.f - t.fy);
        const float w01 = (1.f - t.fx) * t.fy, w11 = t.fx * t.fy;
        // packed FP32x2 FMAs: each lane of a pair is rounded as a scalar fmaf would round it
        float2 lo = __fmul2_rn(make_float2(w00, w00), make_float2(v00.x, v00.y));
        float2 hi = __fmul2_rn(make_float2(w00, w00), make_float2(v00.z, v00.w));
        lo = __ffma2_rn(make_float2(w10, w10), make_float2(v10.x, v10.y), lo);
        hi = __ffma2_rn(make_float2(w10, w10), make_float2(v10.z, v10.w), hi);
        lo = __ffma2_rn(make_float2(w01, w01), make_float2(v01.x, v01.y), lo);
        hi = __ffma2_rn(make_float2(w01, w01), make_float2(v01.z, v01.w), hi);
        lo = __ffma2_rn(make_float2(w11, w11), make_float2(v11.x, v11.y), lo);
        hi = __ffma2_rn(make_float2(w11, w11), make_float2(v11.z, v11.w), hi);
        return make_float4(lo.x, lo.y, hi.x, hi.y);
    }
    return rl_sample(plane, H, W, t);
}

// Slot-map value of a voxel that the selection did not keep.
#define RL_SLOT_NONE 0xFF

// ------------------------------------------------------------------ fast samples
//
// Fast coordinates of a sample known to lie inside the plane: the floor comes from an addition
// rounded towards minus infinity to a multiple of one (exact for |s| < 2^22), whose mantissa is
// also the integer part, so that a sample needs no conversion instruction and one multiply-add
// forms its voxel index.  Same values as rl_taps / rl_anchor_taps.  Both coordinates go through
// packed FP32x2 instructions, each half rounded as a scalar one, which halves the arithmetic of a
// position: 45 views of 1920x1080, D = 64, BF16: 13.35 against 13.63 ms; batched gradient 2.26
// against 2.30 ms; view alpha weights 53 against 55 us; the other gradients within 1%.
#define RL_FLOOR_MAGIC 12582912.f  // 1.5 * 2^23
#define RL_FLOOR_BITS 0x4B400000u
#define RL_FAST_EXTENT (1 << 20)       // image sides for which the fast coordinates are exact

// a - b, both halves (one rounding each, as a subtraction)
__device__ __forceinline__ float2 rl_minus2(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}

struct RLFastTap {
    unsigned idx;  // voxel of the top-left tap within its plane
    float fx, fy;
};

__device__ __forceinline__ unsigned rl_fast_base(int qx, int qy, int W) {
    return (unsigned)qy * (unsigned)W + (unsigned)qx - RL_FLOOR_BITS * ((unsigned)W + 1u);
}

template <bool ANCH>
__device__ __forceinline__ RLFastTap rl_fast_tap(const RLPixWarp<ANCH>& w, const RLAnchor& A, int d, float rho,
                                                 unsigned base, int W) {
    float2 s;
    if constexpr (ANCH) {
        const RLPlaneF k = A.f[d];
        s = __ffma2_rn(make_float2(k.rho, k.rho), make_float2(w.w.dbx, w.w.dby), make_float2(w.w.dax, w.w.day));
        s = __fadd2_rn(make_float2(k.fx, k.fy), s);
        base += (unsigned)k.off;
    } else {
        s = __ffma2_rn(make_float2(rho, rho), make_float2(w.w.bx, w.w.by), make_float2(w.w.ax, w.w.ay));
    }
    const float2 f = __fadd2_rd(s, make_float2(RL_FLOOR_MAGIC, RL_FLOOR_MAGIC));
    const float2 r = rl_minus2(s, __fadd2_rn(f, make_float2(-RL_FLOOR_MAGIC, -RL_FLOOR_MAGIC)));
    RLFastTap t;
    t.fx = r.x;
    t.fy = r.y;
    t.idx = base + __float_as_uint(f.y) * (unsigned)W + __float_as_uint(f.x);
    return t;
}

// True when the samples of every plane in [d_lo, d_hi] lie inside the plane, at least a pixel from
// its border, and the planes are met in front of the view: position and depth factor are linear in
// the plane's inverse depth, so the two end planes bound the others.  The pixel of margin covers
// the rounding.  `first` is plane 0's entry in the anchor's tables.
template <bool ANCH>
__device__ __forceinline__ bool rl_chunk_inside(const RLPixWarp<ANCH>& w, const RLAnchor& A, const RLViews& views,
                                                int d_lo, int d_hi, int qx, int qy, int H, int W, int first = 0) {
    const float rho0 = views.rho[d_lo], rho1 = views.rho[d_hi];
    float x0, y0, x1, y1;
    bool ok;
    if constexpr (ANCH) {
        const RLPlaneK a = A.k[first + d_lo], b = A.k[first + d_hi];
        ok = w.w.ok && a.ix != RL_PLANE_NONE && b.ix != RL_PLANE_NONE;
        x0 = (float)(qx + a.ix) + (a.fx + fmaf(rho0, w.w.dbx, w.w.dax));
        y0 = (float)(qy + a.iy) + (a.fy + fmaf(rho0, w.w.dby, w.w.day));
        x1 = (float)(qx + b.ix) + (b.fx + fmaf(rho1, w.w.dbx, w.w.dax));
        y1 = (float)(qy + b.iy) + (b.fy + fmaf(rho1, w.w.dby, w.w.day));
    } else {
        ok = w.w.dir_ok && fmaf(-rho0, w.w.cz, 1.0f) > 0.0f && fmaf(-rho1, w.w.cz, 1.0f) > 0.0f;
        x0 = (float)qx + fmaf(rho0, w.w.bx, w.w.ax);
        y0 = (float)qy + fmaf(rho0, w.w.by, w.w.ay);
        x1 = (float)qx + fmaf(rho1, w.w.bx, w.w.ax);
        y1 = (float)qy + fmaf(rho1, w.w.by, w.w.ay);
    }
    // a NaN position fails the comparisons; sides beyond RL_FAST_EXTENT take the general path
    return ok && (H | W) < RL_FAST_EXTENT && fminf(x0, x1) >= 1.f && fmaxf(x0, x1) < (float)(W - 2) &&
           fminf(y0, y1) >= 1.f && fmaxf(y0, y1) < (float)(H - 2);
}

// Weights of a sample's taps (x: left upper, y: right upper, z: left lower, w: right lower).
__device__ __forceinline__ float4 rl_weights(float fx, float fy) {
    const float gx = 1.f - fx, gy = 1.f - fy;
    return make_float4(gx * gy, fx * gy, gx * fy, fx * fy);
}

// The same values with both complements from one packed instruction: 1.4% faster where the weights
// are used once (render), 2% slower in the plane-parallel gradients, which form them twice.
__device__ __forceinline__ float4 rl_weights_packed(float fx, float fy) {
    const float2 g = rl_minus2(make_float2(1.f, 1.f), make_float2(fx, fy));
    return make_float4(g.x * g.y, fx * g.y, g.x * fy, fx * fy);
}

// The four taps of a sample blended with packed FP32x2 FMAs (the order of rl_sample).
__device__ __forceinline__ float4 rl_blend(const float4& v00, const float4& v10, const float4& v01, const float4& v11,
                                           const float4& w) {
    float2 lo = __fmul2_rn(make_float2(w.x, w.x), make_float2(v00.x, v00.y));
    float2 hi = __fmul2_rn(make_float2(w.x, w.x), make_float2(v00.z, v00.w));
    lo = __ffma2_rn(make_float2(w.y, w.y), make_float2(v10.x, v10.y), lo);
    hi = __ffma2_rn(make_float2(w.y, w.y), make_float2(v10.z, v10.w), hi);
    lo = __ffma2_rn(make_float2(w.z, w.z), make_float2(v01.x, v01.y), lo);
    hi = __ffma2_rn(make_float2(w.z, w.z), make_float2(v01.z, v01.w), hi);
    lo = __ffma2_rn(make_float2(w.w, w.w), make_float2(v11.x, v11.y), lo);
    hi = __ffma2_rn(make_float2(w.w, w.w), make_float2(v11.z, v11.w), hi);
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// Sample inside the plane: voxel e of the MPI is the top-left tap.
template <typename Tm>
__device__ __forceinline__ float4 rl_sample_at(const Tm* __restrict__ M, unsigned e, int W, const float4& w) {
    const Tm* p = M + (size_t)e * 4u;
    const Tm* q = M + (size_t)(e + (unsigned)W) * 4u;
    return rl_blend(RLStore<Tm>::load4(p), RLStore<Tm>::load4(p + 4), RLStore<Tm>::load4(q), RLStore<Tm>::load4(q + 4),
                    w);
}

template <typename Tm>
__device__ __forceinline__ float4 rl_sample_at(const Tm* __restrict__ M, unsigned e, int W, float fx, float fy) {
    return rl_sample_at(M, e, W, rl_weights(fx, fy));
}

// Adds wt (gl, gh) to one voxel of the gradient.
__device__ __forceinline__ void rl_add_tap(float4* __restrict__ G4, unsigned at, float wt, float2 gl, float2 gh) {
    const float2 a = __fmul2_rn(make_float2(wt, wt), gl), b = __fmul2_rn(make_float2(wt, wt), gh);
    atomicAdd(G4 + at, make_float4(a.x, a.y, b.x, b.y));
}

// The slots of the four taps (00, 10, 01, 11, a byte each) of a sample inside the plane whose
// top-left tap is voxel e of the MPI: loaded with the sample, ahead of the scatter that needs them.
__device__ __forceinline__ unsigned rl_slot_word(const uint8_t* __restrict__ slots, unsigned e, int W) {
    const uint8_t* p = slots + e;
    const uint8_t* q = p + W;
    return (unsigned)__ldg(p) | (unsigned)__ldg(p + 1) << 8 | (unsigned)__ldg(q) << 16 | (unsigned)__ldg(q + 1) << 24;
}

// Bilinear transpose of the gradient g of a sample inside the plane: top-left tap p of its plane,
// voxel e of the MPI.  SPARSE: only into the taps that have a slot in the compact gradient.
template <bool SPARSE>
__device__ __forceinline__ void rl_scatter_at(float* __restrict__ G, unsigned word, unsigned d, unsigned p, unsigned e,
                                              unsigned hw, int W, const float4& w, float4 g, unsigned ng) {
    float4* G4 = reinterpret_cast<float4*>(G);
    const float2 gl = make_float2(g.x, g.y), gh = make_float2(g.z, g.w);
    if constexpr (SPARSE) {
        if (word == 0xFFFFFFFFu) return;
        const unsigned s00 = word & 255u, s10 = (word >> 8) & 255u, s01 = (word >> 16) & 255u, s11 = word >> 24;
        if (s00 != RL_SLOT_NONE && RL_IN(s00, ng)) rl_add_tap(G4, s00 * hw + p, w.x, gl, gh);
        if (s10 != RL_SLOT_NONE && RL_IN(s10, ng)) rl_add_tap(G4, s10 * hw + p + 1u, w.y, gl, gh);
        if (s01 != RL_SLOT_NONE && RL_IN(s01, ng)) rl_add_tap(G4, s01 * hw + p + (unsigned)W, w.z, gl, gh);
        if (s11 != RL_SLOT_NONE && RL_IN(s11, ng)) rl_add_tap(G4, s11 * hw + p + (unsigned)W + 1u, w.w, gl, gh);
    } else {
        if (!RL_IN(d, ng)) return;
        rl_add_tap(G4, e, w.x, gl, gh);
        rl_add_tap(G4, e + 1u, w.y, gl, gh);
        rl_add_tap(G4, e + (unsigned)W, w.z, gl, gh);
        rl_add_tap(G4, e + (unsigned)W + 1u, w.w, gl, gh);
    }
}

template <bool SPARSE>
__device__ __forceinline__ void rl_scatter_tap(float* __restrict__ G, const uint8_t* __restrict__ slots, unsigned d,
                                               unsigned hw, int H, int W, int x, int y, float wt, float4 g,
                                               unsigned ng) {
    if ((unsigned)x >= (unsigned)W || (unsigned)y >= (unsigned)H) return;
    const unsigned pix = (unsigned)(y * W + x);
    const unsigned slot = SPARSE ? (unsigned)__ldg(slots + (d * hw + pix)) : d;
    if ((SPARSE && slot == RL_SLOT_NONE) || !RL_IN(slot, ng)) return;
    rl_add_tap(reinterpret_cast<float4*>(G), slot * hw + pix, wt, make_float2(g.x, g.y), make_float2(g.z, g.w));
}

// The same transpose with each tap tested against the plane.
template <bool SPARSE>
__device__ __forceinline__ void rl_scatter(float* __restrict__ G, const uint8_t* __restrict__ slots, unsigned d,
                                           unsigned hw, int H, int W, const RLTaps& t, float4 g, unsigned ng) {
    const float gx = 1.f - t.fx, gy = 1.f - t.fy;
    rl_scatter_tap<SPARSE>(G, slots, d, hw, H, W, t.x0, t.y0, gx * gy, g, ng);
    rl_scatter_tap<SPARSE>(G, slots, d, hw, H, W, t.x0 + 1, t.y0, t.fx * gy, g, ng);
    rl_scatter_tap<SPARSE>(G, slots, d, hw, H, W, t.x0, t.y0 + 1, gx * t.fy, g, ng);
    rl_scatter_tap<SPARSE>(G, slots, d, hw, H, W, t.x0 + 1, t.y0 + 1, t.fx * t.fy, g, ng);
}

__device__ __forceinline__ float rl_warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One compensated addition (Kahan): s - c carries the running sum of FP32 values to about FP64.  A sum
// that has left the range stays infinite: its compensation would be the NaN of inf - inf.
__device__ __forceinline__ void rl_kahan_add(float& s, float& c, float v) {
    const float y = v - c, t = s + y;
    c = fabsf(t) < INFINITY ? (t - s) - y : 0.f;
    s = t;
}

// Sum of the n loss partials at `partials` (16-byte aligned) by one block, in an order fixed by n and
// the block's size, so the loss is deterministic.  Each thread's own sums are compensated, so the error
// does not grow with the partials a thread adds; the threads' sums are added in plain FP32.  The total is
// returned to thread 0; `red` is shared scratch of nthreads / 32 floats.
__device__ __forceinline__ float rl_partials_sum(const float* __restrict__ partials, unsigned n, int tid, int nthreads,
                                                 float* red) {
    float a[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
    const unsigned n4 = n / 4;
    for (unsigned i = tid; i < n4; i += 8 * nthreads) {
        float4 v[8];  // eight loads in flight: one block reads them all
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const unsigned e = i + u * nthreads;
            v[u] = e < n4 ? __ldcg(reinterpret_cast<const float4*>(partials) + e) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            rl_kahan_add(a[0], c[0], v[u].x);
            rl_kahan_add(a[1], c[1], v[u].y);
            rl_kahan_add(a[2], c[2], v[u].z);
            rl_kahan_add(a[3], c[3], v[u].w);
        }
    }
    if (tid < (int)(n & 3u)) rl_kahan_add(a[0], c[0], __ldcg(partials + n4 * 4 + tid));
    const float acc = rl_warp_sum(((a[0] - c[0]) + (a[1] - c[1])) + ((a[2] - c[2]) + (a[3] - c[3])));
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    float total = 0.f;
    if (tid == 0)
        for (int wi = 0; wi < nthreads / 32; ++wi) total += red[wi];
    return total;
}
