// rl_internal.h -- host-side declarations shared by the translation units of libreallife.
#pragma once
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/reallife.h"
#include "rl_common.cuh"

// Kernel launch tracing (implemented in reallife_api.cu).  rl_trace_begin returns a
// token (-1 when tracing is off) that rl_trace_end closes on the same stream.
int rl_trace_begin(const char* name, cudaStream_t s);
void rl_trace_end(int token, cudaStream_t s);
// Records a failure message for reallife_last_error() and returns `st`.
rl_status rl_fail(rl_status st, const char* fmt, ...);
// Checks the last launch; RL_ECUDA with the CUDA message on failure.
rl_status rl_check_launch(const char* what);

struct RLTraceScope {
    int tok;
    cudaStream_t s;
    RLTraceScope(const char* name, cudaStream_t st) : tok(rl_trace_begin(name, st)), s(st) {}
    ~RLTraceScope() { rl_trace_end(tok, s); }
};

// Device status word (bit RL_DEVFLAG_TIMEOUT: a bounded wait gave up); address on the
// current device, or NULL if it cannot be resolved.
unsigned int* rl_device_status_ptr();
// Warp-kernel family of a render over H x W pixels of n views: 2 per-pixel gather, 3
// plane-parallel.  The automatic setting picks plane-parallel for launches of fewer than
// 2^19 pixel-views (small views), where per-pixel threads are too few to hide gather latency,
// and per-pixel gather otherwise.
int rl_kernel_path(int H, int W, int nviews);
// The same for the gradient of D planes (sparse: compact).  Automatic, in this order, by measured times:
//  - images beyond the plane-parallel grid (H > 131070 or W > 1048560): per-pixel;
//  - pure shifts with a compact gradient, from 2^17 pixel-views on: per-pixel, whose kernel for them
//    shares taps between two pixels and forms no coordinates (256x192, 4 views, D = 32, FP32: 51
//    against 64 us; 512x384, 4 views, BF16: 175 against 206);
//  - fewer than 2^19 pixel-views: plane-parallel, which gathers each sample once (64x48, 2 views,
//    D = 32: 13 against 51 us; 256x192, 8 views, D = 64: 233 against 289 us);
//  - anchored coordinates: per-pixel, since a plane-parallel tile repeats the FP64 set-up of the
//    anchors for every 32 pixels, a per-pixel block for every 128 (1024x768, 4 views, D = 64, BF16:
//    2507 against 1710 us);
//  - compact: plane-parallel where its warps fill the SM (rl_grad_pp_fill >= 0.8) and up to 32 planes
//    (512x384, 4 views, BF16: 206 against 246 us; 700x768: 545 against 593) or 2^20 pixel-views
//    (512x384, 3 views, D = 40, FP32: 225 against 234).  Else per-pixel: with D = 33, 34 and 41 to 50 too
//    few of an SM's warps hold planes (512x384, 5 views, BF16: D = 33 331 against 260 us, D = 42 467 against
//    326), beyond 2^20 the chunk exchange of sixteen warps costs more than the second gather (700x768,
//    D = 64: 1178 against 1112);
//  - dense: plane-parallel, whose warps join their lanes' shared taps (500x375, 4 views, D = 32: 223
//    against 286 us), from a fill on that grows with the pixel-views (from 2^20 on the per-pixel kernel
//    fills the device evenly), for pure shifts (whose per-pixel taps vary least) and beyond 36 planes.
//    960x540, 4 views, FP32, plane-parallel against per-pixel, rotated and shifted: D = 5 137 / 112,
//    136 / 105; D = 13 277 / 287, 285 / 269; D = 25 537 / 547, 555 / 512; D = 36 734 / 796, 732 / 746;
//    D = 42 1120 / 927, 1137 / 869; D = 52 1199 / 1157, 1174 / 1081; D = 57 1378 / 1270, 1348 / 1187;
//    D = 60 1331 / 1341, 1287 / 1249.  500x375, 4 views: D = 5 51 / 47, 50 / 44; D = 13 106 / 117,
//    104 / 110; D = 42 400 / 365, 418 / 349; D = 48 418 / 422, 425 / 401.
int rl_grad_path(int H, int W, int nviews, int D, bool anchored, bool shifts, bool sparse);
// Share of an SM's warps that hold planes in a plane-parallel gradient of D planes.
double rl_grad_pp_fill(int D);
// The gradient family of a batched step of so many pixel-views in all: per-pixel gather, whose long
// units hide the cost of fetching them (three batches of eight requests of mixed sizes and levels, 96x128
// to 1024x768, D = 16 to 64, BF16: 2235, 685 and 1103 us against 3532, 933 and 1822 us plane-parallel),
// unless the whole batch is too small to fill the device with them.
int rl_batch_grad_path(long long pixel_views);
// The raw process-wide setting of reallife_set_kernel_path (0, 2 to 5).
int rl_kernel_path_setting();

// TMA descriptor of a BF16 activation volume [K][H][W][32] (16-byte aligned) with a box of
// {32 channels, halo voxels along W} and 64-byte swizzling; false when it cannot be encoded.
bool rl_encode_act_tmap(CUtensorMap* map, const void* act, int K, int H, int W, int halo);

// True when every view's warp offset p - q is the same for all pixels of a plane: no
// rotation relative to the reference (R_rel - I exactly 0 in FP32), no depth offset of the
// centre and the reference's focal lengths.
inline bool rl_views_are_shifts(const RLViews& v) {
    for (int i = 0; i < v.n; ++i) {
        const RLViewParam& p = v.v[i];
        for (int j = 0; j < 9; ++j)
            if (p.E[j] != 0.f) return false;
        if (p.C[2] != 0.f || p.dfx != 0.f || p.dfy != 0.f) return false;
    }
    return v.n > 0;
}

// ----------------------------------------------------------------- launchers
// All take device pointers and enqueue on `s`; arguments are validated by the caller.

rl_status rl_launch_render(const void* M, rl_dtype dt, int D, int H, int W, const RLViews& views, float* out,
                           cudaStream_t s);
rl_status rl_launch_warp_offsets(int D, int H, int W, const RLViews& views, float* out, cudaStream_t s);

// Fused warp + composite + residual + adjoint.  mode_loss: residual from images (full-res
// images at level img_level, averaged on the fly) else from grad_out.  slots != NULL
// (slot map [D][H][W], RL_SLOT_NONE where not kept; mode_loss only): compact gradient [k][H][W][4]; else
// dense [D][H][W][4].  partials: one float per block
// (loss mode, 16-byte aligned); returns the number of blocks through *nblocks.
rl_status rl_launch_grad(const void* M, rl_dtype dt, int D, int H, int W, const RLViews& views, bool mode_loss,
                         const float* images, int img_level, const float* grad_out, const uint8_t* slots, float* G,
                         float inv_n, float* partials, int* nblocks, cudaStream_t s);
// Largest number of loss partials any gradient kernel family writes.
size_t rl_grad_num_blocks(int H, int W, int N);
rl_status rl_launch_grad_pp(const void* M, rl_dtype dt, int D, int H, int W, const RLViews& views, bool mode_loss,
                            const float* images, int img_level, const float* grad_out, const uint8_t* slots, float* G,
                            float inv_n, float* partials, int* nblocks, cudaStream_t s);
size_t rl_grad_pp_num_blocks(int H, int W, int N, bool anchored);
rl_status rl_launch_render_pp(const void* M, rl_dtype dt, int D, int H, int W, const RLViews& views, float* out,
                              cudaStream_t s);
rl_status rl_launch_loss_reduce(const float* partials, int n, float scale, float* out, cudaStream_t s);

// Top-k selection on the MPI M [D][h][w][4] (or on keys [D][h][w] when keys != NULL).
// Outputs (each optional): S [k][h][w], mask [h][w], slot map [D][h][w], the MPI's alphas alone
// [D][h][w] in its storage type; Gzero [k][h][w][4] is zeroed.
rl_status rl_launch_select(const void* M, rl_dtype dt, const float* keys, int D, int h, int w, int k, uint8_t* S,
                           uint64_t* mask, uint8_t* slots, float* Gzero, cudaStream_t s, int mode = 0,
                           void* alphas = nullptr);
// Level-l MPI Ml [D][H>>l][W>>l][4] = Down^l(M) (level >= 1) and the selection on it in one pass: outputs as
// rl_launch_select without the mask, identical values.  With images and Il != NULL it also writes the
// level-l source images Il [N][H>>l][W>>l][3] (2^l x 2^l means of images [N][H][W][3], formed exactly as
// the gradient kernels form them on the fly), which the gradient then reads at img_level 0.
rl_status rl_launch_pyramid_select(const void* M, rl_dtype dt, int D, int H, int W, int level, void* Ml, int k,
                                   uint8_t* S, uint8_t* slots, float* Gzero, int mode, cudaStream_t s,
                                   const float* images = nullptr, int N = 0, float* Il = nullptr,
                                   void* alphas = nullptr);
// Slot map [D][h][w] from a selection mask [h][w]: the kept planes of a pixel in ascending order
// take slots 0 .. k-1; kept planes beyond the first k get no slot.
rl_status rl_launch_mask_to_slots(const uint64_t* mask, int D, int k, int hw, uint8_t* slots, cudaStream_t s);
rl_status rl_launch_downsample_f32(const float* x, int P, int H, int W, int C, int level, float* y,
                                   cudaStream_t s);
// With Ml (level MPI) and lambda_s != 0 the sparsity prior joins the alpha step.  With loss.out the
// first block also writes loss.out[0] = loss.scale * (sum of the loss.n partials) of the gradient.
struct RLLossSum {
    const float* partials = nullptr;  // 16-byte aligned
    int n = 0;
    float scale = 0.f;
    float* out = nullptr;
};
rl_status rl_launch_update(void* M, rl_dtype dt, int D, int H, int W, int level, const uint8_t* S, const float* G,
                           int k, float lambda, int clamp01, cudaStream_t s, const void* Ml = nullptr,
                           float lambda_s = 0.f, const RLLossSum& loss = RLLossSum());

// Batched stages of one HSGD iteration over a batch table in device memory (header and items
// of rl_common.cuh), each one persistent launch of one wave of resident blocks.  The gradient
// stage has a launch for each family, per-pixel gather (shared memory for `planes` planes) and
// plane-parallel; a batch's items all take the one that rl_batch_grad_path names, and a captured step
// holds both launches.
rl_status rl_launch_select_batch(const void* table, rl_dtype dt, cudaStream_t s);
rl_status rl_launch_grad_batch(const void* table, rl_dtype dt, int planes, cudaStream_t s);
rl_status rl_launch_grad_pp_batch(const void* table, rl_dtype dt, cudaStream_t s);
rl_status rl_launch_update_batch(const void* table, rl_dtype dt, cudaStream_t s);
unsigned rl_grad_gather_tiles_x(int w);
unsigned rl_grad_gather_tiles_y(int h);
unsigned rl_grad_pp_tiles_x(int h, int w, int D, bool anchored);
unsigned rl_grad_pp_tiles_y(int h, int w, bool anchored);

// Blocks of a persistent launch of `kernel`: the resident blocks per SM on the current device
// times its SMs (at least one); computed once per device and kernel instantiation.
template <auto kernel>
inline int rl_persistent_grid(int threads, size_t smem) {
    static int cached[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    const bool cacheable = dev >= 0 && dev < 64;
    if (cacheable && cached[dev]) return cached[dev];
    int sms = 0, per = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess) cudaGetLastError();
    const int grid = (sms > 0 ? sms : 1) * (per > 0 ? per : 1);
    if (cacheable) cached[dev] = grid;
    return grid;
}

// Metrics (metrics.cu): FP64 partial sums of the SSIM windows, squared differences and kept
// mass, and the number of partials the two metric calls need.
size_t rl_ssim_blocks(int N, int H, int W);
size_t rl_metrics_partials(int N, int H, int W);
// out[0] = mean squared difference, out[1] = mean SSIM of x, y [N][H][W][3] (H, W >= 11).
rl_status rl_launch_image_metrics(const float* x, const float* y, int N, int H, int W, double* out, double* partials,
                                  cudaStream_t s);
// out[0] = sum of the kept alpha weights, out[1] = sum of all alpha weights.
rl_status rl_launch_kept_mass(const void* M, rl_dtype dt, int D, int H, int W, const uint64_t* mask, double* out,
                              double* partials, cudaStream_t s);

// Alpha weights of the MPI warped into each view (Eq. eq_gradient): A device [N][D][H][W], from
// the alphas alone [D][H][W] when given, else from the MPI's.
rl_status rl_launch_view_alpha(const void* M, const void* alphas, rl_dtype dt, int D, int H, int W, const RLViews& views, float* A,
                               cudaStream_t s);
// Sparsified gradient volume V [4N+4][k][h][w] from the level MPI Ml [D][h][w][4], the
// selection S [k][h][w], the view alpha weights A [N][D][h][w] and full-resolution images.
// With act != NULL the same channels go to act [k][h][w][32] BF16 channels-last (the learned
// network's input, channels >= 4N+4 zero) instead, and V is not written.
rl_status rl_launch_volume(const void* Ml, rl_dtype dt, int D, int h, int w, int level, const uint8_t* S, int k,
                           const float* A, const float* images, const RLInvViews& iv, float* V, cudaStream_t s,
                           void* act = nullptr);

// Gradient volume of Sec. 3.3 at `level`: selection S, view alpha weights and V_s, with the
// checks of reallife_gradient_volume; with act != NULL it writes the network's packed input
// instead of V (V may then be NULL).
rl_status rl_gradient_volume(const rl_mpi* m, const float* images, const rl_camera* src, int N, int k, int level,
                             int selection, uint8_t* S_out, float* V, void* act, void* ws, size_t ws_bytes,
                             cudaStream_t stream);

// Learned update network (lgd.cu): packed parameter bytes, parameter packing, activation
// buffer bytes and the forward pass (V [C][K][H][W] FP32 -> residual [K][H][W][4] FP32,
// two activation buffers of rl_lgd_act_bytes each and a 4-byte grid-barrier counter that the
// call resets on the stream).
size_t rl_lgd_net_bytes();
rl_status rl_lgd_prepare(const rl_lgd_params* p, void* net, cudaStream_t s);
size_t rl_lgd_act_bytes(int K, int H, int W);
rl_status rl_lgd_forward(const void* net, const float* V, int C, int K, int H, int W, float* residual, void* act0,
                         void* act1, unsigned* grid_bar, cudaStream_t s);
// The network alone, on an input already packed into act0 (act1 and the counter as above).
rl_status rl_lgd_network(const void* net, int K, int H, int W, float* residual, void* act0, void* act1,
                         unsigned* grid_bar, cudaStream_t s);
