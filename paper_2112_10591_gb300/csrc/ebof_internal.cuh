// ebof_internal.cuh -- internal declarations shared by the CUDA translation
// units of libebof.so.  Nothing here is part of the C ABI (include/ebof.h).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda.h>  // CUtensorMap (type only; the driver is reached through the runtime)
#include <cuda_runtime.h>

#include "ebof.h"

namespace ebof {

constexpr int kMaxLevels = 8;
constexpr int kMaxDim = 16384;
constexpr int kMaxPatch = 16;
constexpr int32_t kInfD = 2147483647;  // squared distance with no edge pixel

// Device error bits, latched in StreamState::d_err.
constexpr int kErrBounds = 1;
constexpr int kErrTimeout = 2;  // a bounded wait on an asynchronous copy ran out

__host__ __device__ inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

// Geometry of one pyramid level.  Internal images are row-major with a row
// pitch rounded up to 32 elements (128-byte rows for 4-byte types).
struct Level {
    int w, h, pitch;
    size_t plane;      // pitch * h elements
    int npx, npy;      // patch grid (reading F2); 0 if no patch fits
};

// Geometry of a whole frame: the level chain plus the level-0 pitches.
struct Geometry {
    int width, height;
    int levels;        // levels used by the flow (capped, reading F1)
    Level lv[kMaxLevels];
    size_t pyr_floats; // floats of one pyramid slot (I, Ix, Iy at every level)
    size_t pyr_off[kMaxLevels];  // offset of level l in a slot (I; Ix, Iy follow)
    int max_patches;   // largest npx * npy over the levels
};

Geometry make_geometry(int width, int height, int levels, int ps, int stride);

// The pyramid of one slot as the fused pyramid kernels see it.
struct PyrDesc {
    int levels;
    int w[kMaxLevels], h[kMaxLevels], pitch[kMaxLevels];
    size_t off[kMaxLevels];    // element offset of level l's I in a slot
    size_t plane[kMaxLevels];  // Ix and Iy follow I at one and two planes
    int blk0[kMaxLevels + 1];  // first block of level l in the gradient launch
    int gb0;                   // first block launched (blk0[1] when the box means
                               // kernel writes level 0's gradients, else 0)
};

// Per-window event counters kept on the device (one per batch slot).
struct DevStats {
    unsigned long long in_window;
    unsigned long long dropped_oob;
    unsigned long long edge_px;
    unsigned long long pad;
};

// Kernel parameter bundles ---------------------------------------------------

// Distance to surface value y(d), d = sqrt(D), and surface to level-0
// intensity: Eq. 1 (mode EBOF_SURFACE_EXP, intensity 255 y) or an ablation
// surface of §IV-D (intensity gain * y, gain = 255 / y(d_sat)).
struct SurfaceMap {
    int mode;
    float alpha;  // Eq. 1
    float d_sat;  // bound of DS_LB
    float gain;   // intensity scale of the ablation surfaces
};

inline SurfaceMap exp_surface(float alpha) { return SurfaceMap{0, alpha, 6.0f, 255.0f}; }

// Default bound, in mbarrier try-wait rounds, of a kernel's wait for a
// tensor copy.
constexpr long long kWaitLimitDefault = 1LL << 22;

struct FlowParams {
    bool half;  // pyramid stored as FP16 (loads widened to FP32)
    int ps, stride, gn_iters;
    float gn_damping;
    int var_outer, var_sor;
    float delta, gamma, alpha_s, omega;
    long long wait_limit;  // rounds of the variational kernels' waits
    long long flow_wait_limit;  // of the copy-ahead kernel's for a region's flow
    // variational layouts (ebof_params): none changes a result
    int sor_tma_min_per_sm, sor_row_waves, var_cluster_max;
    // the one-launch refinement's counters (kLevelCtl words, 0 at first) and
    // two buffers of level_n packets of 16 bytes (0 at first), used by
    // no other launch at the same time; null: one launch per step
    unsigned *level_ctl;
    void *level_xch;
    size_t level_n;
    bool chained;  // the search's launch is behind a kernel of the same chain
};
// most regions of a one-launch refinement: 1.75 an SM of 152 (the launch asks the
// device; this bounds the packets that a stream or group holds)
constexpr int kLevelBlocks = 266;
constexpr int kLevelCtl = 4;
// level_n for a stream or group of up to `frames` frames a call.
size_t level_packets(const Geometry &geo, int var_sor, int cluster_max, int frames);

// Launches a kernel; chained: behind a kernel of the same chain, with nothing
// between the two on the stream, as chain_begin() has it.  A window of 641 x 479
// launched kernel by kernel: 585 us, 647 with full dependencies.  Inside a
// graph full dependencies are the faster ones (two windows of 346 x 260 299 us,
// 308 with early starts; one of 1280 x 720 463 against 480), so captured
// launches keep them.
template <class... P, class... A>
cudaError_t launch_chained(bool chained, void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                           cudaStream_t st, A... args)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (chained && cudaStreamIsCapturing(st, &capture) != cudaSuccess) chained = false;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = chained && capture == cudaStreamCaptureStatusNone ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

// Launchers (each enqueues on `st`; frames = batch size). ---------------------

// A1: clear edge images, scatter events of n_windows consecutive windows.
void launch_scatter(const uint16_t *x, const uint16_t *y, const int64_t *t, int64_t n,
                    int64_t t_begin, int64_t dt, int n_windows, int W, int H, int pitch,
                    uint8_t *E, size_t frame_stride, DevStats *stats,
                    unsigned long long *dropped_time, cudaStream_t st);

// A1 for a group of streams: frame f scatters the events of desc[f] (device).
void launch_scatter_desc(const ebof_window_desc *desc, int frames, int W, int H,
                         int pitch, uint8_t *E, size_t frame_stride, DevStats *stats,
                         unsigned long long *dropped_time, cudaStream_t st);

// A2: Alg. 1 then Alg. 2; writes E_df (pitched) and optional dense export.
void launch_denoise_fill(const uint8_t *E, uint8_t *Ed, uint8_t *Edf, int W, int H, int pitch,
                         size_t frame_stride, int frames, int conn, int n_d, int n_f,
                         uint8_t *export_dense, DevStats *stats, cudaStream_t st,
                         bool chained = false);

// A3: per column and 32 rows, the edge pixels' bits and the nearest edge rows
// above and below; g: at least g_pitch * H int32 a frame.
void launch_edt_columns(const uint8_t *E, int edge_pitch, size_t edge_frame_stride, int W,
                        int H, int32_t *g, int g_pitch, size_t g_frame_stride, int frames,
                        cudaStream_t st, bool chained = false);

// A4: per-row lower envelope -> D, fused surface (Eq. 1 or an ablation
// surface) and level-0 intensity.
void launch_edt_rows_surface(const int32_t *g, int g_pitch, size_t g_frame_stride, int W, int H,
                             const SurfaceMap &sm, int32_t *D_dense, float *S_dense, void *I0,
                             int i_pitch, size_t i_frame_stride, int frames, bool half,
                             cudaStream_t st);
// The same with the Eq. 1 surface.
void launch_edt_rows_surface(const int32_t *g, int g_pitch, size_t g_frame_stride, int W, int H,
                             float alpha, int32_t *D_dense, float *S_dense, void *I0,
                             int i_pitch, size_t i_frame_stride, int frames, bool half,
                             cudaStream_t st);

// A3 and A4 with the Eq. 1 surface of a dense edge image, the column distances
// kept in g [H][W], which may be D_dense or S_dense itself.
void launch_edt_inplace(const uint8_t *edge, int W, int H, float alpha, int32_t *g,
                        int32_t *D_dense, float *S_dense, cudaStream_t st);

int sm_count();  // of the current device; 0: unknown

// Per-device kernel attributes (opt-in shared memory); call with the device current.
void init_front_attributes();
void init_flow_attributes();

// Surface given by the caller -> level-0 intensity (255 d_exp, or gain * y).
void launch_surface_to_intensity(const float *S, int W, int H, void *I0, int pitch, bool half,
                                 const SurfaceMap &sm, cudaStream_t st);

// A5: every box-mean level and every level's gradients of `frames` slots
// starting at `slots` (level 0 must be in place), in two launches.
void launch_pyramid(void *slots, const Geometry &geo, size_t frame_stride, int frames, bool half,
                    cudaStream_t st);
// One plane of a level (row pitch `pitch`) into a dense w x h FP32 array.
void launch_pyramid_export(const void *plane, bool half, int w, int h, int pitch, float *dst,
                           cudaStream_t st);

// A6: patch inverse search at one level.
void launch_patch_search(const void *I0, const void *I0x, const void *I0y, const void *I1,
                         const Level &lv, size_t pyr_frame_stride, const float *Uc,
                         const Level *lvc, size_t uc_frame_stride, float *up,
                         size_t up_frame_stride, int frames, const FlowParams &fp,
                         int *err, cudaStream_t st);

// A7: densification.
void launch_densify(const void *I0, const void *I1, const Level &lv, size_t pyr_frame_stride,
                    const float *up, size_t up_frame_stride, float *U, size_t u_frame_stride,
                    int frames, const FlowParams &fp, cudaStream_t st);

// Tensor maps (TMA descriptors) of the variational coefficient planes of
// each pyramid level in a stream's or group's work buffer: level l holds
// frames x coeff_planes() planes of pitch_l x h_l floats.
struct SorMaps {
    CUtensorMap coef;
    CUtensorMap u[2];       // of the flow buffers
    const float *ubase[2];  // which these are
};
struct CoefMaps {
    bool ok[kMaxLevels];
    SorMaps map[kMaxLevels];
};
// Fills m for `frames` frames of `work` and of the flow buffers Ua, Ub, as a
// level lays them out; levels whose maps cannot be encoded are marked not ok
// (their SOR sweeps then load directly).
void make_coef_maps(float *work, const float *Ua, const float *Ub, size_t u_frame_stride,
                    const Geometry &geo, int var_sor, int frames, CoefMaps *m);

// A8: variational refinement of U.  Returns the buffer holding the result:
// U itself, or Utmp (same shape as U) when the fused kernel ping-pongs.
// maps: the level's tensor maps, or nullptr; err: device
// error word (kErrTimeout if a bounded wait runs out).
float *launch_variational(const void *I0, const void *I0x, const void *I0y, const void *I1,
                          const Level &lv, size_t pyr_frame_stride, float *U, float *Utmp,
                          size_t u_frame_stride, float *work, size_t work_frame_stride,
                          int frames, const FlowParams &fp, const SorMaps *maps,
                          int *err, cudaStream_t st);
bool var_fused_supported(int var_sor);
void init_var_attributes();
float *launch_variational_fused(const void *I0, const void *I0x, const void *I0y,
                                const void *I1, const Level &lv, size_t pyr_frame_stride,
                                float *U, float *Utmp, size_t u_frame_stride, float *coef,
                                int frames, const FlowParams &fp, const SorMaps *maps,
                                int *err, cudaStream_t st);

// A9 for one window, destination pointer read from device memory.
void launch_flow_out_ptr(const float *U, int W, int H, int pitch, size_t u_frame_stride,
                         float *const *dst, int frames, cudaStream_t st);

// A9: level-0 flow to the caller's dense planar layout.
void launch_flow_out(const float *U, int W, int H, int pitch, size_t u_frame_stride,
                     float *flow, int frames, cudaStream_t st);

}  // namespace ebof
