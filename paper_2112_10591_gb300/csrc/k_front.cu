// k_front.cu -- event accumulation, denoising/filling, exact EDT, surface.
//
// §III-A: edge image of a window.  §III-B: Alg. 1 (denoise) then Alg. 2
// (fill).  §III-C: exact Euclidean distance transform as int32 squared
// distances (separable: a per-column pass, then a per-row lower envelope of
// parabolas), fused with Eq. 1, d_exp = 1 - exp(-sqrt(D) / alpha), and the
// 8-bit intensity scale 255 * d_exp the flow block runs on.
#include "ebof.h"
#include "dev_common.cuh"
#include "ebof_internal.cuh"
#include "profiler.cuh"
#include "seg.cuh"

#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>

namespace ebof {

namespace {

// ---------------------------------------------------------------- A1 scatter
// One thread per event.  The window index of an event is
// floor((t - t_begin) / dt) when it lies in [0, n_windows); duplicates collapse
// (a byte store of 1 is idempotent).  A block walks one contiguous chunk of
// the events, 32 per warp and step.  Timestamps are sorted, so a warp's 32
// events nearly always share a window and its counts run in registers until
// the window changes (then one atomic per counter); a step whose events
// straddle a window boundary counts per group of lanes that share a window.
__device__ __forceinline__ void flush_counts(int cur, unsigned long long &c_in,
                                             unsigned long long &c_oob, unsigned long long &c_time,
                                             int lane, DevStats *stats,
                                             unsigned long long *dropped_time)
{
    if (lane == 0) {
        if (cur >= 0) {
            if (c_in) atomicAdd(&stats[cur].in_window, c_in);
            if (c_oob) atomicAdd(&stats[cur].dropped_oob, c_oob);
        } else if (cur == -1 && c_time) {
            atomicAdd(dropped_time, c_time);
        }
    }
    c_in = c_oob = c_time = 0;
}

__global__ void scatter_kernel(const uint16_t *__restrict__ x, const uint16_t *__restrict__ y,
                               const int64_t *__restrict__ t, int64_t n, int64_t t_begin,
                               int64_t dt, int n_windows, int W, int H, int pitch,
                               uint8_t *__restrict__ E, size_t fstride, DevStats *stats,
                               unsigned long long *dropped_time)
{
    chain_begin();
    const int64_t span = dt * (int64_t)n_windows;
    const int lane = threadIdx.x & 31;
    const int64_t per_block =
        ((n + gridDim.x - 1) / gridDim.x + blockDim.x - 1) / blockDim.x * blockDim.x;
    const int64_t beg = (int64_t)blockIdx.x * per_block;
    const int64_t end = min(n, beg + per_block);
    int cur = -3;  // window of the running counts (-1: outside every window, -3: none)
    unsigned long long c_in = 0, c_oob = 0, c_time = 0;
    for (int64_t base = beg; base < end; base += blockDim.x) {
        const int64_t i = base + threadIdx.x;
        int k = -2;  // -2: no event (tail), -1: outside every window
        bool oob = false;
        if (i < end) {
            const int64_t rel = t[i] - t_begin;
            k = -1;
            if (rel >= 0 && rel < span) {
                k = (int)(rel / dt);
                const int xi = x[i], yi = y[i];
                if (xi < W && yi < H)
                    E[(size_t)k * fstride + (size_t)yi * pitch + xi] = 1;
                else
                    oob = true;
            }
        }
        const unsigned valid = __ballot_sync(0xffffffffu, k != -2);
        const unsigned oob_mask = __ballot_sync(0xffffffffu, oob);
        if (valid == 0) continue;  // warp-uniform
        const int kl = __shfl_sync(0xffffffffu, k, __ffs(valid) - 1);
        if (__all_sync(0xffffffffu, k == -2 || k == kl)) {
            if (kl != cur) {
                flush_counts(cur, c_in, c_oob, c_time, lane, stats, dropped_time);
                cur = kl;
            }
            if (kl >= 0) {
                c_in += __popc(valid);
                c_oob += __popc(oob_mask);
            } else {
                c_time += __popc(valid);
            }
            continue;
        }
        flush_counts(cur, c_in, c_oob, c_time, lane, stats, dropped_time);
        cur = -3;
        const unsigned peers = __match_any_sync(0xffffffffu, k);
        if (lane == __ffs(peers) - 1) {
            if (k >= 0) {
                atomicAdd(&stats[k].in_window, (unsigned long long)__popc(peers));
                const int no = __popc(peers & oob_mask);
                if (no) atomicAdd(&stats[k].dropped_oob, (unsigned long long)no);
            } else if (k == -1) {
                atomicAdd(dropped_time, (unsigned long long)__popc(peers));
            }
        }
    }
    flush_counts(cur, c_in, c_oob, c_time, lane, stats, dropped_time);
}

// Scatter for a group of streams: frame f takes the events of descriptor f.
__global__ void scatter_desc_kernel(const ebof_window_desc *__restrict__ desc, int W, int H,
                                    int pitch, uint8_t *__restrict__ E, size_t fstride,
                                    DevStats *stats, unsigned long long *dropped_time)
{
    chain_begin();
    const int f = blockIdx.y;
    const ebof_window_desc d = desc[f];
    const int lane = threadIdx.x & 31;
    uint8_t *e = E + (size_t)f * fstride;
    unsigned long long in_w = 0, oob = 0, out_t = 0;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < d.n_events;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + threadIdx.x;
        if (i < d.n_events) {
            const int64_t tt = d.t[i];
            if (tt >= d.t_begin && tt < d.t_end) {
                ++in_w;
                const int xi = d.x[i], yi = d.y[i];
                if (xi < W && yi < H) e[(size_t)yi * pitch + xi] = 1;
                else ++oob;
            } else {
                ++out_t;
            }
        }
    }
    // block sums, one atomic per block and counter (same-address atomics
    // serialise in L2)
    __shared__ unsigned long long s_sum[3][32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        in_w += __shfl_xor_sync(0xffffffffu, in_w, o);
        oob += __shfl_xor_sync(0xffffffffu, oob, o);
        out_t += __shfl_xor_sync(0xffffffffu, out_t, o);
    }
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (lane == 0) {
        s_sum[0][warp] = in_w;
        s_sum[1][warp] = oob;
        s_sum[2][warp] = out_t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < nwarps; ++k) {
            in_w += s_sum[0][k];
            oob += s_sum[1][k];
            out_t += s_sum[2][k];
        }
        if (in_w) atomicAdd(&stats[f].in_window, in_w);
        if (oob) atomicAdd(&stats[f].dropped_oob, oob);
        if (out_t) atomicAdd(dropped_time, out_t);
    }
}

// Scatter of a fused launch over several groups: a work list of event
// chunks (kScatterChunk events of one window) over all the windows.  Every
// block turns the windows' event counts, read from their device
// descriptors, into chunk offsets in shared memory, then walks the chunks
// blockIdx.x, blockIdx.x + gridDim.x, ...: windows of very different sizes
// spread evenly over the blocks.  The counts of a chunk go out as one atomic
// per counter and block, as in scatter_desc_kernel.
__global__ void __launch_bounds__(256)
scatter_list_kernel(const ScatterWin *__restrict__ wins, int n_wins)
{
    __shared__ int s_off[kScatterListMax + 1];
    __shared__ unsigned long long s_sum[3][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0) {
        int run = 0;
        for (int base = 0; base < n_wins; base += 32) {
            const int i = base + lane;
            int c = 0;
            if (i < n_wins) {
                const int64_t ne = wins[i].desc->n_events;
                c = (int)((ne + kScatterChunk - 1) / kScatterChunk);
            }
            int v = c;  // inclusive scan over the lanes
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            if (i < n_wins) s_off[i] = run + v - c;
            run += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) s_off[n_wins] = run;
    }
    __syncthreads();
    const int total = s_off[n_wins];
    for (int c = blockIdx.x; c < total; c += gridDim.x) {
        // the window of chunk c: the last one whose chunks start at or before c
        int lo = 0, hi = n_wins - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_off[mid] <= c) lo = mid;
            else hi = mid - 1;
        }
        const ScatterWin &w = wins[lo];
        const ebof_window_desc d = *w.desc;
        const int64_t i0 = (int64_t)(c - s_off[lo]) * kScatterChunk;
        const int64_t i1 = min(d.n_events, i0 + (int64_t)kScatterChunk);
        unsigned long long in_w = 0, oob = 0, out_t = 0;
        for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            const int64_t tt = d.t[i];
            if (tt >= d.t_begin && tt < d.t_end) {
                ++in_w;
                const int xi = d.x[i], yi = d.y[i];
                if (xi < w.W && yi < w.H) w.E[(size_t)yi * w.pitch + xi] = 1;
                else ++oob;
            } else {
                ++out_t;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            in_w += __shfl_xor_sync(0xffffffffu, in_w, o);
            oob += __shfl_xor_sync(0xffffffffu, oob, o);
            out_t += __shfl_xor_sync(0xffffffffu, out_t, o);
        }
        if (lane == 0) {
            s_sum[0][warp] = in_w;
            s_sum[1][warp] = oob;
            s_sum[2][warp] = out_t;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
                in_w += s_sum[0][k];
                oob += s_sum[1][k];
                out_t += s_sum[2][k];
            }
            if (in_w) atomicAdd(&w.stats->in_window, in_w);
            if (oob) atomicAdd(&w.stats->dropped_oob, oob);
            if (out_t) atomicAdd(w.dropped_time, out_t);
        }
        __syncthreads();  // s_sum is rewritten by the next chunk
    }
}

// ---------------------------------------------------------------- A2
// Alg. 1 then Alg. 2 in one pass: a block stages E for its 32 x 8 tile plus
// a 2-pixel halo in shared memory, denoises the tile plus 1 pixel there
// (counts in E), then fills the tile (counts in the denoised image).
// Neighbours outside the image count as non-edge in both, as in
// count_neighbours, so the result equals denoise_kernel then fill_kernel.
constexpr int kDfX = 32, kDfY = 8;

__device__ __forceinline__ int count_tile(const uint8_t (*t)[kDfX + 4], int lx, int ly, int conn)
{
    int c = t[ly - 1][lx] + t[ly + 1][lx] + t[ly][lx - 1] + t[ly][lx + 1];
    if (conn == 8) c += t[ly - 1][lx - 1] + t[ly - 1][lx + 1] + t[ly + 1][lx - 1] + t[ly + 1][lx + 1];
    return c;
}

// (bx, by): the tile, f: the frame.
__device__ __forceinline__ void denoise_fill_body(const uint8_t *__restrict__ E,
                                                  uint8_t *__restrict__ Edf, int W, int H,
                                                  int pitch, size_t fstride, int conn, int n_d,
                                                  int n_f, uint8_t *__restrict__ export_dense,
                                                  DevStats *stats, int bx, int by, int f)
{
    __shared__ uint8_t sE[kDfY + 4][kDfX + 4];
    __shared__ uint8_t sD[kDfY + 4][kDfX + 4];  // denoised, 1-pixel ring inside a 2-pixel frame
    const uint8_t *e = E + (size_t)f * fstride;
    const int x0 = bx * kDfX - 2, y0 = by * kDfY - 2;
    const int t = threadIdx.y * kDfX + threadIdx.x;
    for (int i = t; i < (kDfX + 4) * (kDfY + 4); i += kDfX * kDfY) {
        const int lx = i % (kDfX + 4), ly = i / (kDfX + 4);
        const int gx = x0 + lx, gy = y0 + ly;
        uint8_t v = 0;
        if (gx >= 0 && gy >= 0 && gx < W && gy < H) v = e[(size_t)gy * pitch + gx] ? 1 : 0;
        sE[ly][lx] = v;
        sD[ly][lx] = 0;
    }
    __syncthreads();
    for (int i = t; i < (kDfX + 2) * (kDfY + 2); i += kDfX * kDfY) {
        const int lx = 1 + i % (kDfX + 2), ly = 1 + i / (kDfX + 2);
        uint8_t v = sE[ly][lx];
        if (v && count_tile(sE, lx, ly, conn) < n_d) v = 0;
        sD[ly][lx] = v;
    }
    __syncthreads();
    const int x = bx * kDfX + threadIdx.x, y = by * kDfY + threadIdx.y;
    uint8_t v = 0;
    if (x < W && y < H) {
        const int lx = threadIdx.x + 2, ly = threadIdx.y + 2;
        v = sD[ly][lx];
        if (!v && count_tile(sD, lx, ly, conn) >= n_f) v = 1;
        Edf[(size_t)f * fstride + (size_t)y * pitch + x] = v;
        if (export_dense) export_dense[(size_t)f * W * H + (size_t)y * W + x] = v;
    }
    // one atomic per block: same-address atomics serialise in L2
    const int nedge = __syncthreads_count(v != 0);
    if (t == 0 && nedge) atomicAdd(&stats[f].edge_px, (unsigned long long)nedge);
}

__global__ void __launch_bounds__(kDfX * kDfY)
denoise_fill_kernel(const uint8_t *__restrict__ E, uint8_t *__restrict__ Edf, int W, int H,
                    int pitch, size_t fstride, int conn, int n_d, int n_f,
                    uint8_t *__restrict__ export_dense, DevStats *stats)
{
    chain_begin();
    denoise_fill_body(E, Edf, W, H, pitch, fstride, conn, n_d, n_f, export_dense, stats,
                      blockIdx.x, blockIdx.y, blockIdx.z);
}

__global__ void __launch_bounds__(kDfX * kDfY)
seg_denoise_fill_kernel(const __grid_constant__ SegTable<SegDenoise> tab)
{
    int b;
    const SegDenoise &a = seg_of(tab, b);
    const int bx = b % a.gx, r = b / a.gx;
    denoise_fill_body(a.E, a.Edf, a.W, a.H, a.pitch, a.fs, a.conn, a.n_d, a.n_f, nullptr,
                      a.stats, bx, r % a.gy, r / a.gy);
}

// ---------------------------------------------------------------- A3
// Column pass.  A column's edge pixels as 32-row bit words, and for every word
// the nearest edge rows outside it: the last one above (-32768: none) and the
// first one below (32767: none), 16 bits each.  The row pass turns a pixel's
// two words into its column distance with two bit scans.  That is 8 bytes per
// 32 pixels of a column where the distances themselves took 128, and the pass
// is one read of the edge image.  An image of one word a column (H <= 32) has
// no second plane, so the words always fit W * H int32.
// Measured against distances written by this pass (column and row pass in one
// stream): see the row pass.
//
// A block covers 32 columns; a warp packs the words ty, ty + blockDim.y, ...
// of its columns (a word's 32 byte loads in flight together) and publishes
// their first and last edge rows; one warp then runs down and one up the
// column's words.
//
// DIST: the distances themselves, a pixel an int32, for a stand-alone call whose
// scratch is one of its results: a row of distances is read by that row's block
// only, before it writes the row's results there, where a word serves 32 rows.
// The words then stay in shared memory.  It writes the 4 bytes a pixel that the
// words save: 640x480 @@A, 1920x1080 @@B us a call, against @@C and @@D.
constexpr int kColWarps = 32;
constexpr int kNoneAbove = -32768, kNoneBelow = 32767;

__host__ __device__ __forceinline__ int col_words(int H) { return (H + 31) / 32; }
// shared memory of a block: the first and last edge rows of its words (dist:
// and the words, 128 KB in all for 16384 rows)
__host__ __device__ __forceinline__ size_t cols_smem_bytes(int nw, bool dist)
{
    return (size_t)nw * 32 * (2 * sizeof(int16_t) + (dist ? sizeof(uint32_t) : 0));
}
// the nearest edge rows above and below, 16 bits each
__device__ __forceinline__ int pack_rows(int above, int below)
{
    return (int)((uint32_t)(above & 0xffff) | ((uint32_t)below << 16));
}
__device__ __forceinline__ int row_above(int v) { return (int)(int16_t)(v & 0xffff); }
__device__ __forceinline__ int row_below(int v) { return v >> 16; }

// Column distance from a pixel's words; above kMaxDim - 1: no edge pixel.
__device__ __forceinline__ int word_distance(uint32_t m, int ab, int y)
{
    const int b = y & 31;
    const uint32_t us = m << (31 - b), ds = m >> b;
    const int up = us ? __clz(us) : y - row_above(ab);
    const int dn = ds ? __clz(__brev(ds)) : row_below(ab) - y;
    return min(up, dn);
}

// bx: the block of 32 columns, f: the frame.
template <bool DIST>
__device__ __forceinline__ void edt_cols_body(const uint8_t *__restrict__ E, int epitch,
                                              size_t efs, int W, int H, int32_t *__restrict__ g,
                                              int gpitch, size_t gfs, unsigned bx, unsigned f)
{
    extern __shared__ __align__(4) int16_t s_rows[];
    const int nw = col_words(H), c = threadIdx.x, x = bx * 32 + c;
    int16_t *s_last = s_rows + c, *s_first = s_last + nw * 32;
    uint32_t *s_words = reinterpret_cast<uint32_t *>(s_rows + nw * 64) + c;  // DIST
    const bool colok = x < W;
    const uint8_t *e = E + (size_t)f * efs + min(x, W - 1);
    uint32_t *words = reinterpret_cast<uint32_t *>(g + (size_t)f * gfs) + x;
    for (int wi = threadIdx.y; wi < nw; wi += blockDim.y) {
        // all 32 loads in flight before the first test (rows past the image
        // read its last row and are masked out)
        uint8_t ev[32];
#pragma unroll
        for (int b = 0; b < 32; ++b) ev[b] = e[(size_t)min(wi * 32 + b, H - 1) * epitch];
        uint32_t m = 0;
#pragma unroll
        for (int b = 0; b < 32; ++b)
            if (ev[b]) m |= 1u << b;
        if (wi == nw - 1 && (H & 31)) m &= (1u << (H & 31)) - 1;
        if (DIST) s_words[wi * 32] = m;
        else if (colok) words[(size_t)wi * gpitch] = m;
        s_last[wi * 32] = (int16_t)(m ? wi * 32 + 31 - __clz(m) : kNoneAbove);
        s_first[wi * 32] = (int16_t)(m ? wi * 32 + __ffs(m) - 1 : kNoneBelow);
    }
    if (!DIST && nw == 1) return;
    __syncthreads();
    // one warp runs down the column's words and one up, eight at a time (the
    // loads before the chain of maxima)
    constexpr int kRun = 8;
    if (threadIdx.y == 0) {  // last edge row above each word
        int run = kNoneAbove;
        for (int w0 = 0; w0 < nw; w0 += kRun) {
            int l[kRun];
#pragma unroll
            for (int k = 0; k < kRun; ++k) l[k] = s_last[min(w0 + k, nw - 1) * 32];
#pragma unroll
            for (int k = 0; k < kRun; ++k) {
                if (w0 + k < nw) s_last[(w0 + k) * 32] = (int16_t)run;
                run = max(run, l[k]);
            }
        }
    }
    if (threadIdx.y == (blockDim.y > 1 ? 1 : 0)) {  // first edge row below
        int run = kNoneBelow;
        for (int w0 = nw - 1; w0 >= 0; w0 -= kRun) {
            int l[kRun];
#pragma unroll
            for (int k = 0; k < kRun; ++k) l[k] = s_first[max(w0 - k, 0) * 32];
#pragma unroll
            for (int k = 0; k < kRun; ++k) {
                if (w0 - k >= 0) s_first[(w0 - k) * 32] = (int16_t)run;
                run = min(run, l[k]);
            }
        }
    }
    __syncthreads();
    if (!colok) return;
    for (int wi = threadIdx.y; wi < nw; wi += blockDim.y) {
        const int ab = pack_rows(s_last[wi * 32], s_first[wi * 32]);
        if (!DIST) {
            words[(size_t)(nw + wi) * gpitch] = ab;
            continue;
        }
        const uint32_t m = s_words[wi * 32];
        const int y1 = min(wi * 32 + 32, H);
        for (int y = wi * 32; y < y1; ++y) words[(size_t)y * gpitch] = word_distance(m, ab, y);
    }
}

template <bool DIST>
__global__ void __launch_bounds__(32 * kColWarps)
edt_cols_kernel(const uint8_t *__restrict__ E, int epitch, size_t efs, int W, int H,
                int32_t *__restrict__ g, int gpitch, size_t gfs)
{
    chain_begin();
    edt_cols_body<DIST>(E, epitch, efs, W, H, g, gpitch, gfs, blockIdx.x, blockIdx.y);
}

__global__ void __launch_bounds__(32 * kColWarps)
seg_edt_cols_kernel(const __grid_constant__ SegTable<SegEdtCols> tab)
{
    int b;
    const SegEdtCols &a = seg_of(tab, b);
    edt_cols_body<false>(a.E, a.epitch, a.efs, a.W, a.H, a.g, a.gpitch, a.gfs, b % a.gx, b / a.gx);
}

// ---------------------------------------------------------------- A4
// Row pass: D(x) = min over columns s of (x - s)^2 + h(s), h(s) = g(s, y)^2.
// With F(s) = s^2 + h(s) it reads D(x) = x^2 + min_s (F(s) - 2 x s).  The
// column that attains the minimum never moves left as x grows: for s < t,
// (F(t) - 2 x t) - (F(s) - 2 x s) falls with x.  So the columns that attain it
// at x0 and x1 bound the ones between them, whichever of equal ones is taken.
//  1. The row's F is staged in shared memory (a column without edge pixels: a
//     value above every distance).
//  2. The columns that own the pixels 32, 64, ... are found coarse to fine: a
//     pixel half way (or an eighth of the way) between two known ones is
//     searched by a warp's lanes over the columns between their owners only.
//  3. A band of 32 pixels, one per lane, takes the minimum over the columns
//     between the owners of its ends: every lane reads the same columns, four
//     at a time, so the bands of a row together cost W evaluations a lane, each
//     a multiply-add and a minimum.
//  4. Eq. 1 (or an ablation surface) and the 8-bit scale, coalesced stores.
// Every step is an exact integer minimum, so D is bit-identical to any exact
// EDT.  No step depends on the distance to the nearest edge, and the lanes of
// a warp never diverge.  It replaced the lower convex hull of the points
// (s, F(s)), built and merged band by band, whose stack and bridge walks were
// serial chains of 64-bit orientation tests.  Bound by the integer pipes (a
// row issues on 75 % of cycles).  Measured, the hull form's time in brackets:
// 6.5 us at 346x260 (17.7), 29.6 at 1920x1080 (39.7), 10.9 a frame in 1280x720
// batches (17.4).

// (x - s)^2 + h(s) is below 2^29 for images up to 16384 px a side; a column
// without edge pixels gets h = 2^30.
constexpr int kNoColumn = 1 << 30;

constexpr int kRowsPerBlock = 4;                  // rows (warps) per block
constexpr int kWarpsLongRow = 16;                 // warps of a long row
constexpr int kRowLoads = 4;                      // pixels in flight per lane
constexpr size_t kRowsSmemCap = 200 * 1024;       // bytes; 16384-px rows fit

// Shared memory of one row, in bytes: F (int32, padded to a multiple of 4) and
// the owners of the band ends.
__host__ __device__ __forceinline__ size_t rows_smem_bytes(int W)
{
    const size_t nb = ((size_t)W + 31) / 32;
    return 4 * (((size_t)W + 3) & ~(size_t)3) + ((4 * (nb + 1) + 15) & ~(size_t)15);
}

// Owners of the NP pixels x, x + dx, ... (NP * dx columns of pixels) among the
// columns lo .. hi, into own[0], own[stride], ...: a warp's lanes share the
// columns; the minima first, then, for each pixel, the column among the
// minimum lane's that attains it.
template <int NP>
__device__ __forceinline__ void find_owners(const int32_t *F, int lo, int hi, int x, int dx,
                                            int32_t *own, int stride, int lane)
{
    int best[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) best[k] = INT32_MAX;
#pragma unroll 2
    for (int s = lo + lane; s <= hi; s += 32) {
        const int f = F[s];
#pragma unroll
        for (int k = 0; k < NP; ++k) best[k] = min(best[k], f - 2 * (x + k * dx) * s);
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int m = __reduce_min_sync(0xffffffffu, best[k]);
        const int l = __ffs(__ballot_sync(0xffffffffu, best[k] == m)) - 1;
        const int n2x = -2 * (x + k * dx);
        int arg = hi;
        for (int s0 = lo + l; s0 <= hi; s0 += 32 * 32) {
            const int s = s0 + 32 * lane;
            const unsigned hit = __ballot_sync(0xffffffffu, s <= hi && F[s] + n2x * s == m);
            if (hit) {
                arg = s0 + 32 * (__ffs(hit) - 1);
                break;
            }
        }
        if (lane == 0) own[k * stride] = arg;
    }
}

// Level-0 intensity of the flow block.  FP32 storage keeps I = 255 d_exp.
// FP16 storage keeps the complement C = 255 - I = 255 exp(-d / alpha): the
// flow is the same for I and 255 - I (mean-normalised patches, squared
// residuals and products of derivatives), and far from the edges, where I
// saturates towards 255 and its variations are far below FP16's 0.125 step
// there, C is small and keeps them at FP16's relative precision.
__device__ __forceinline__ void st_int(float *p, float s, float c) { (void)c; *p = 255.0f * s; }
__device__ __forceinline__ void st_int(__half *p, float s, float c)
{
    (void)s;
    *p = __float2half_rn(255.0f * c);
}

// The ablation surfaces are stored as gain * y itself (no complement); FP16
// clamps at its largest finite value, so distances beyond 65504 / gain
// (about 1540 px for DS_L) read as one plateau.
__device__ __forceinline__ void st_lin(float *p, float v) { *p = v; }
__device__ __forceinline__ void st_lin(__half *p, float v)
{
    *p = __float2half_rn(fminf(v, 65504.0f));
}

// y(d) of the ablation surfaces of §IV-D (mode 1 DS_L, 2 DS_LB, 3 DS_Log).
__device__ __forceinline__ float ablation_surface(const SurfaceMap &sm, float d)
{
    return sm.mode == 1 ? d : (sm.mode == 2 ? fminf(d, sm.d_sat) : log1pf(d));
}

// WPR warps serve a row.  WPR = 1: rows_per_block rows of one warp each,
// warp-level barriers only.  WPR > 1: one row per block.  D is exact whatever
// WPR, so the layout never changes a result.  bx: the block of rows, f: the
// frame.  A warp past the block's rows_per_block rows (a fused launch sized for
// another segment's) exits (WPR = 1 has warp-level barriers only).  DIST: g holds
// distances instead of words, and D_dense or S_dense may be g itself: a row is
// read before row_sync() and written after it, by its own warps.
template <int WPR, bool DIST, typename T>
__device__ __forceinline__ void edt_rows_surface_body(
    const int32_t *g, int gpitch, size_t gfs, int W, int H, int rows_per_block,
    const SurfaceMap &sm, int32_t *D_dense, float *S_dense, T *__restrict__ I0, int ipitch,
    size_t ifs, int bx, int f)
{
    constexpr int NT = 32 * WPR;
    constexpr int FAC = 4;  // how many times finer each level of step 2 is
    extern __shared__ __align__(16) int32_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rib = warp / WPR, wr = warp % WPR;  // row within the block, warp within the row
    const int tr = wr * 32 + lane;
    const int y = bx * rows_per_block + rib;
    // WPR = 1: the whole warp; WPR > 1: never (one row per block)
    if (rib >= rows_per_block || y >= H) return;
    const int Wp = (W + 3) & ~3, nb = (W + 31) / 32;
    int32_t *F = smem + (size_t)rib * (rows_smem_bytes(W) / 4);
    int32_t *own = F + Wp;  // own[b]: owner of pixel 32 b (bounds at both ends)
    auto row_sync = [] {
        if (WPR == 1) __syncwarp();
        else __syncthreads();
    };
    // 1. loads issued in batches of kRowLoads before their first use
    {
        const int nw = col_words(H);
        const uint32_t *words = reinterpret_cast<const uint32_t *>(g + (size_t)f * gfs) +
                                (size_t)(DIST ? y : y >> 5) * gpitch;
        const size_t ab_off = (size_t)nw * gpitch;
        const int none = pack_rows(kNoneAbove, kNoneBelow);
        for (int x0 = tr; x0 < Wp; x0 += NT * kRowLoads) {
            uint32_t m[kRowLoads];
            int ab[kRowLoads], d[kRowLoads];
#pragma unroll
            for (int u = 0; u < kRowLoads; ++u) {
                const int x = x0 + NT * u;
                m[u] = DIST ? kMaxDim : 0;
                ab[u] = none;
                if (x < W) {
                    m[u] = words[x];
                    if (!DIST && nw > 1) ab[u] = (int)words[ab_off + x];
                }
            }
#pragma unroll
            for (int u = 0; u < kRowLoads; ++u)
                d[u] = DIST ? (int)m[u] : word_distance(m[u], ab[u], y);
#pragma unroll
            for (int u = 0; u < kRowLoads; ++u) {
                const int x = x0 + NT * u;
                if (x < Wp) F[x] = x * x + (d[u] < kMaxDim ? d[u] * d[u] : kNoColumn);
            }
        }
    }
    if (tr == 0) {
        own[0] = 0;
        own[nb] = W - 1;
    }
    // 2. owners of the band ends; the FAC - 1 pixels between two known ones
    // share their columns: one warp takes them all, or, while there are fewer
    // such intervals than warps, one each
    int step = 1;
    while (step * FAC < nb) step *= FAC;
    for (; step >= 1; step /= FAC) {
        row_sync();  // F and the coarser owners
        const int wide = step * FAC, ni = (nb + wide - 1) / wide;
        const bool split = WPR > 1 && ni < WPR;
        for (int u = wr; u < (split ? ni * (FAC - 1) : ni); u += WPR) {
            const int i = split ? u / (FAC - 1) : u;
            const int b0 = i * wide + step * (split ? 1 + u % (FAC - 1) : 1);
            if (b0 >= nb) continue;
            const int lo = own[i * wide], hi = own[min(i * wide + wide, nb)];
            if (!split && b0 + (FAC - 2) * step < nb) {
                find_owners<FAC - 1>(F, lo, hi, 32 * b0, 32 * step, own + b0, step, lane);
            } else {
                for (int b = b0; b < min(split ? b0 + 1 : nb, (i + 1) * wide); b += step)
                    find_owners<1>(F, lo, hi, 32 * b, 0, own + b, 0, lane);
            }
        }
    }
    row_sync();

    // 3. the bands; 4. surface and intensity
    T *irow = I0 ? I0 + (size_t)f * ifs + (size_t)y * ipitch : nullptr;
    const size_t dbase = (size_t)f * W * H + (size_t)y * W;
    const float inv_alpha = 1.0f / sm.alpha;
    for (int b = wr; b < nb; b += WPR) {
        const int x = 32 * b + lane, lo = own[b] & ~3, hi = own[b + 1];
        const int n2x = -2 * x;
        int m = INT32_MAX, o = n2x * lo;
#pragma unroll 2
        for (int s = lo; s <= hi; s += 4) {
            // min(a + b, c) is one instruction
            const int4 q = *reinterpret_cast<const int4 *>(F + s);
            int v = __viaddmin_s32(q.y, n2x, q.x);
            v = __viaddmin_s32(q.z, 2 * n2x, v);
            v = __viaddmin_s32(q.w, 3 * n2x, v);
            m = __viaddmin_s32(v, o, m);
            o += 4 * n2x;
        }
        if (x >= W) continue;
        m += x * x;
        const int32_t D = m < kNoColumn ? m : kInfD;  // kInfD: the image has no edge pixel
        float S = 1.0f, C = 0.0f;  // d_exp of Eq. 1 and its complement 1 - d_exp
        if (sm.mode == 0) {
            if (D != kInfD) {
                C = expf(-sqrtf((float)D) * inv_alpha);
                S = 1.0f - C;
            }
            if (irow) st_int(&irow[x], S, C);
        } else {
            // no edge pixel (kInfD): y at the finite d = sqrt(INT32_MAX)
            S = ablation_surface(sm, sqrtf((float)D));
            if (irow) st_lin(&irow[x], sm.gain * S);
        }
        if (D_dense) D_dense[dbase + x] = D;
        if (S_dense) S_dense[dbase + x] = S;
    }
}

template <int WPR, typename T>
__global__ void __launch_bounds__(32 * (WPR > kRowsPerBlock ? WPR : kRowsPerBlock))
edt_rows_surface_kernel(const int32_t *__restrict__ g, int gpitch, size_t gfs, int W, int H,
                        int rows_per_block, SurfaceMap sm, int32_t *__restrict__ D_dense,
                        float *__restrict__ S_dense, T *__restrict__ I0, int ipitch, size_t ifs)
{
    chain_begin();
    edt_rows_surface_body<WPR, false, T>(g, gpitch, gfs, W, H, rows_per_block, sm, D_dense,
                                         S_dense, I0, ipitch, ifs, blockIdx.x, blockIdx.y);
}

// The row pass from distances that lie in one of its results (no restrict: it
// writes where it has read).
template <int WPR>
__global__ void __launch_bounds__(32 * WPR)
edt_rows_inplace_kernel(const int32_t *g, int W, int H, SurfaceMap sm, int32_t *D_dense,
                        float *S_dense)
{
    edt_rows_surface_body<WPR, true, float>(g, W, 0, W, H, 1, sm, D_dense, S_dense, nullptr, 0, 0,
                                            blockIdx.x, 0);
}

template <typename T>
__global__ void __launch_bounds__(32 * kRowsPerBlock)
seg_edt_rows_kernel(const __grid_constant__ SegTable<SegEdtRows> tab)
{
    int b;
    const SegEdtRows &a = seg_of(tab, b);
    edt_rows_surface_body<1, false, T>(a.g, a.gpitch, a.gfs, a.W, a.H, a.rows, a.sm, nullptr,
                                       nullptr, (T *)a.I0, a.ipitch, a.ifs, b % a.gx, b / a.gx);
}

// Caller-given surface (dense, d_exp in [0, 1]) to the level-0 intensity.
template <typename T>
__global__ void surface_to_intensity_kernel(const float *__restrict__ S, int W, int H,
                                            T *__restrict__ I0, int pitch, SurfaceMap sm)
{
    chain_begin();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= W) return;
    const float sv = S[(size_t)y * W + x];
    if (sm.mode == 0)
        st_int(&I0[(size_t)y * pitch + x], sv, 1.0f - sv);
    else
        st_lin(&I0[(size_t)y * pitch + x], sm.gain * sv);
}

inline unsigned grid1d(int64_t n, int block, int cap)
{
    int64_t b = (n + block - 1) / block;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

}  // namespace

void launch_scatter(const uint16_t *x, const uint16_t *y, const int64_t *t, int64_t n,
                    int64_t t_begin, int64_t dt, int n_windows, int W, int H, int pitch,
                    uint8_t *E, size_t frame_stride, DevStats *stats,
                    unsigned long long *dropped_time, cudaStream_t st)
{
    if (n <= 0) return;
    StageScope sc(kStScatter, 1, st);
    scatter_kernel<<<grid1d(n, 256, 152 * 16), 256, 0, st>>>(x, y, t, n, t_begin, dt, n_windows,
                                                             W, H, pitch, E, frame_stride, stats,
                                                             dropped_time);
}

void launch_scatter_desc(const ebof_window_desc *desc, int frames, int W, int H, int pitch,
                         uint8_t *E, size_t frame_stride, DevStats *stats,
                         unsigned long long *dropped_time, cudaStream_t st)
{
    StageScope sc(kStScatter, 1, st);
    // the event counts are read on the device: size the grid for the largest
    // windows (about 4 blocks per SM in all), blocks past a window's end exit
    dim3 grd(std::max(64, 608 / std::max(frames, 1)), frames);
    scatter_desc_kernel<<<grd, 256, 0, st>>>(desc, W, H, pitch, E, frame_stride, stats,
                                             dropped_time);
}

void launch_denoise_fill(const uint8_t *E, uint8_t *Ed, uint8_t *Edf, int W, int H, int pitch,
                         size_t frame_stride, int frames, int conn, int n_d, int n_f,
                         uint8_t *export_dense, DevStats *stats, cudaStream_t st, bool chained)
{
    (void)Ed;  // the denoised image stays in shared memory
    StageScope sc(kStDenoiseFill, 1, st);
    dim3 blk(kDfX, kDfY), grd((W + kDfX - 1) / kDfX, (H + kDfY - 1) / kDfY, frames);
    launch_chained(chained, denoise_fill_kernel, grd, blk, 0, st, E, Edf, W, H, pitch,
                   frame_stride, conn, n_d, n_f, export_dense, stats);
}

int edt_cols_warps(int H) { return std::min(col_words(H), kColWarps); }
size_t edt_cols_smem(int H, bool dist) { return cols_smem_bytes(col_words(H), dist); }

void launch_edt_columns(const uint8_t *E, int edge_pitch, size_t edge_frame_stride, int W,
                        int H, int32_t *g, int g_pitch, size_t g_frame_stride, int frames,
                        cudaStream_t st, bool chained)
{
    StageScope sc(kStEdtCols, 1, st);
    dim3 blk(32, edt_cols_warps(H)), grd((W + 31) / 32, frames);
    launch_chained(chained, edt_cols_kernel<false>, grd, blk, edt_cols_smem(H, false), st, E,
                   edge_pitch, edge_frame_stride, W, H, g, g_pitch, g_frame_stride);
}

int edt_rows_block_rows(int W)
{
    int rows = kRowsPerBlock;
    while (rows > 1 && (size_t)rows * rows_smem_bytes(W) > kRowsSmemCap) --rows;
    return rows;
}

size_t edt_rows_smem(int W, int rows) { return (size_t)rows * rows_smem_bytes(W); }

// Warps per row: one for batches (fewest instructions per frame), four for
// single windows (one or two frames per launch), one row per block, to shorten
// a row's chain; sixteen for long rows that leave each an SM (stand-alone, against
// four warps: 2048x16 16.5 -> 10.4 us, 4096x150 54.6 -> 20.6, 8192x16 86 -> 29,
// 16384x1 109 -> 53, 16384x150 133 -> 55).
int edt_rows_wpr(int W, int H, int frames)
{
    if (frames > 2) return 1;
    return W >= 2048 && (long long)H * frames <= sm_count() ? kWarpsLongRow : kRowsPerBlock;
}

template <typename T>
void edt_rows_t(const int32_t *g, int g_pitch, size_t g_frame_stride, int W, int H,
                const SurfaceMap &sm, int32_t *D_dense, float *S_dense, T *I0, int i_pitch,
                size_t i_frame_stride, int frames, bool chained, cudaStream_t st)
{
    const int wpr = edt_rows_wpr(W, H, frames);
    // one warp a row: four rows per block, fewer where a row's shared memory
    // is large; the wider layout: one row per block
    const int rows = wpr == 1 ? edt_rows_block_rows(W) : 1;
    const size_t smem = edt_rows_smem(W, rows);
    dim3 grd((H + rows - 1) / rows, frames);
    auto kern = wpr == 1               ? edt_rows_surface_kernel<1, T>
                : wpr == kWarpsLongRow ? edt_rows_surface_kernel<kWarpsLongRow, T>
                                       : edt_rows_surface_kernel<kRowsPerBlock, T>;
    launch_chained(chained, kern, grd, 32 * (wpr == 1 ? rows : wpr), smem, st, g, g_pitch,
                   g_frame_stride, W, H, rows, sm, D_dense, S_dense, I0, i_pitch, i_frame_stride);
}

void launch_edt_inplace(const uint8_t *edge, int W, int H, float alpha, int32_t *g,
                        int32_t *D_dense, float *S_dense, cudaStream_t st)
{
    {
        StageScope sc(kStEdtCols, 1, st);
        edt_cols_kernel<true><<<(W + 31) / 32, dim3(32, edt_cols_warps(H)), edt_cols_smem(H, true),
                                st>>>(edge, W, 0, W, H, g, W, 0);
    }
    StageScope sc(kStEdtRows, 1, st);
    const int wpr = edt_rows_wpr(W, H, 1);
    auto kern = wpr == kWarpsLongRow ? edt_rows_inplace_kernel<kWarpsLongRow>
                                     : edt_rows_inplace_kernel<kRowsPerBlock>;
    kern<<<H, 32 * wpr, edt_rows_smem(W, 1), st>>>(g, W, H, exp_surface(alpha), D_dense, S_dense);
}

static void edt_rows(const int32_t *g, int g_pitch, size_t g_frame_stride, int W, int H,
                     const SurfaceMap &sm, int32_t *D_dense, float *S_dense, void *I0,
                     int i_pitch, size_t i_frame_stride, int frames, bool half, bool chained,
                     cudaStream_t st)
{
    StageScope sc(kStEdtRows, 1, st);
    if (half)
        edt_rows_t(g, g_pitch, g_frame_stride, W, H, sm, D_dense, S_dense, (__half *)I0,
                   i_pitch, i_frame_stride, frames, chained, st);
    else
        edt_rows_t(g, g_pitch, g_frame_stride, W, H, sm, D_dense, S_dense, (float *)I0,
                   i_pitch, i_frame_stride, frames, chained, st);
}

void launch_edt_rows_surface(const int32_t *g, int g_pitch, size_t g_frame_stride, int W, int H,
                             const SurfaceMap &sm, int32_t *D_dense, float *S_dense, void *I0,
                             int i_pitch, size_t i_frame_stride, int frames, bool half,
                             cudaStream_t st)
{
    edt_rows(g, g_pitch, g_frame_stride, W, H, sm, D_dense, S_dense, I0, i_pitch, i_frame_stride,
             frames, half, false, st);
}

// Whether a stand-alone transform's rows start while its columns end: that saves
// a launch's latency (2 us), but rows started early fill the SMs that the column
// blocks leave, and only those.  So they do where those SMs take at most one row
// more each than all of them would (measured, early against late: 346x260 8.3
// and 10.3 us, 640x480 12.4 and 14.4, 1024x640 18.5 and 20.4, 2048x200 20.6 and
// 21.3, 3500x40 30.8 and 32.9, 3500x80 32.8 both; beyond it 1280x720 22.6 both,
// 1920x1080 45.1 and 35.4, 4096x300 82.0 and 37.0, 8192x200 90.2 and 62.6).
// Within a window rows start late (613x397 with exports 386 us, early 388).
static bool rows_start_early(int W, int H)
{
    const int sms = sm_count(), left = sms - (W + 31) / 32;
    return left > 0 && (H + left - 1) / left <= (H + sms - 1) / sms + 1;
}

void launch_edt_rows_surface(const int32_t *g, int g_pitch, size_t g_frame_stride, int W, int H,
                             float alpha, int32_t *D_dense, float *S_dense, void *I0,
                             int i_pitch, size_t i_frame_stride, int frames, bool half,
                             cudaStream_t st)
{
    edt_rows(g, g_pitch, g_frame_stride, W, H, exp_surface(alpha), D_dense, S_dense, I0, i_pitch,
             i_frame_stride, frames, half, frames == 1 && rows_start_early(W, H), st);
}

int sm_count()
{
    static std::atomic<int> known[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int n = known[dev].load(std::memory_order_relaxed);
    if (n == 0 && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
        known[dev].store(n, std::memory_order_relaxed);
    return n;
}

void init_front_attributes()
{
    auto opt_in = [](const void *fn) {
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowsSmemCap);
    };
    opt_in((const void *)edt_rows_surface_kernel<1, float>);
    opt_in((const void *)edt_rows_surface_kernel<kRowsPerBlock, float>);
    opt_in((const void *)edt_rows_surface_kernel<1, __half>);
    opt_in((const void *)edt_rows_surface_kernel<kRowsPerBlock, __half>);
    opt_in((const void *)edt_rows_surface_kernel<kWarpsLongRow, float>);
    opt_in((const void *)edt_rows_surface_kernel<kWarpsLongRow, __half>);
    opt_in((const void *)edt_rows_inplace_kernel<kRowsPerBlock>);
    opt_in((const void *)edt_rows_inplace_kernel<kWarpsLongRow>);
    opt_in((const void *)edt_cols_kernel<false>);
    opt_in((const void *)edt_cols_kernel<true>);
    opt_in((const void *)seg_edt_cols_kernel);
    opt_in((const void *)seg_edt_rows_kernel<float>);
    opt_in((const void *)seg_edt_rows_kernel<__half>);
}

void launch_seg_scatter(const ScatterWin *wins, int n_wins, int blocks, cudaStream_t st)
{
    StageScope sc(kStScatter, 1, st);
    scatter_list_kernel<<<blocks, 256, 0, st>>>(wins, n_wins);
}

void launch_seg_denoise_fill(const SegTable<SegDenoise> &t, int blocks, cudaStream_t st)
{
    StageScope sc(kStDenoiseFill, 1, st);
    seg_denoise_fill_kernel<<<blocks, dim3(kDfX, kDfY), 0, st>>>(t);
}

void launch_seg_edt_cols(const SegTable<SegEdtCols> &t, int blocks, int max_h, cudaStream_t st)
{
    StageScope sc(kStEdtCols, 1, st);
    const dim3 blk(32, edt_cols_warps(max_h));
    seg_edt_cols_kernel<<<blocks, blk, edt_cols_smem(max_h, false), st>>>(t);
}

void launch_seg_edt_rows(const SegTable<SegEdtRows> &t, int blocks, int rows_max, size_t smem,
                         bool half, cudaStream_t st)
{
    StageScope sc(kStEdtRows, 1, st);
    if (half)
        seg_edt_rows_kernel<__half><<<blocks, 32 * rows_max, smem, st>>>(t);
    else
        seg_edt_rows_kernel<float><<<blocks, 32 * rows_max, smem, st>>>(t);
}

void launch_surface_to_intensity(const float *S, int W, int H, void *I0, int pitch, bool half,
                                 const SurfaceMap &sm, cudaStream_t st)
{
    StageScope sc(kStEdtRows, 1, st);
    dim3 grd((W + 255) / 256, H);
    if (half)
        surface_to_intensity_kernel<__half>
            <<<grd, 256, 0, st>>>(S, W, H, (__half *)I0, pitch, sm);
    else
        surface_to_intensity_kernel<float><<<grd, 256, 0, st>>>(S, W, H, (float *)I0, pitch, sm);
}

}  // namespace ebof
