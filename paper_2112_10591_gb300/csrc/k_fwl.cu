// k_fwl.cu -- the Flow Warping Loss of §IV-C (ebof_fwl in include/ebof.h).
//
// Two launches on the caller's stream, after the images are cleared:
//   1. fwl_splat_kernel: one thread per event (grid-stride).  An event of
//      the window votes its polarity at its pixel into I_uncomp and, moved
//      back along the flow to t_begin, with bilinear weights into I_comp
//      (float atomics, the two votes of a row as one where they are an aligned
//      pair; votes outside the image are dropped).
//   2. fwl_sums_kernel: per-block sums of I and I^2 of both images in a fixed
//      order; the last block to finish adds the blocks' in a fixed order and
//      writes FWL = var(I_comp) / var(I_uncomp) with the two variances.
// The sums are kept as unevaluated triples of floats (about 70 bits) inside a
// block and as doubles beyond it: this chip's FP64 rate made the sums in double
// the longest step, and two floats (48 bits) held less than a double does.
// Measured at 1280x720 with 276k events: the sums in double 16.9 + 6.6 us in two
// launches, a call 44.9; pairs 10.2 and 25.3; triples 11.1 and 27.3.  The rest is
// the splat, 15 us of L1 requests for scattered votes (L1 at 76 %).
// Traffic: 16 B per event read (x, y, t, p) plus 8 B of flow at its pixel,
// the two images written by atomics and read once (8 B per pixel each way).
#include "ebof.h"
#include "profiler.cuh"

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace {

constexpr int kFwlThreads = 256;
constexpr int kFwlPartialBlocks = 2 * 152;  // blocks the scratch has room for
constexpr int kFwlBlocks = kFwlPartialBlocks - 2;  // blocks used; then the arrival counter

size_t align256(size_t b) { return (b + 255) / 256 * 256; }

__global__ void fwl_splat_kernel(const uint16_t *__restrict__ x, const uint16_t *__restrict__ y,
                                 const int64_t *__restrict__ t, const int8_t *__restrict__ p,
                                 int64_t n, int64_t t_begin, int64_t t_end,
                                 const float *__restrict__ flow, int W, int H,
                                 float *__restrict__ comp, float *__restrict__ uncomp)
{
    const size_t P = (size_t)W * H;
    const float inv_span = t_end > t_begin ? 1.0f / (float)(t_end - t_begin) : 0.0f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t ti = t[i];
        if (ti < t_begin || ti >= t_end) continue;
        const int xi = x[i], yi = y[i];
        if (xi >= W || yi >= H) continue;
        const float s = p ? (float)p[i] : 1.0f;
        const size_t o = (size_t)yi * W + xi;
        atomicAdd(&uncomp[o], s);
        const float tau = (float)(ti - t_begin) * inv_span;
        const float xw = (float)xi - flow[o] * tau;
        const float yw = (float)yi - flow[P + o] * tau;
        const float fx = floorf(xw), fy = floorf(yw);
        const float ax = xw - fx, ay = yw - fy;
        const int X0 = (int)fx, Y0 = (int)fy;
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const int Y = Y0 + dy;
            if (Y < 0 || Y >= H) continue;
            const float wy = dy ? ay : 1.0f - ay;
            const float v0 = s * ((1.0f - ax) * wy), v1 = s * (ax * wy);
            float *q = comp + ((ptrdiff_t)Y * W + X0);
            const bool in0 = X0 >= 0 && X0 < W, in1 = X0 + 1 >= 0 && X0 + 1 < W;
            if (in0 && in1 && ((uintptr_t)q & 7) == 0) {
                asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(q), "f"(v0), "f"(v1)
                             : "memory");
            } else {
                if (in0) atomicAdd(q, v0);
                if (in1) atomicAdd(q + 1, v1);
            }
        }
    }
}

// The sum s + e of two floats, exactly (Knuth's two-sum).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

// A sum held as three floats h + l + m, each the rounding errors of the one
// before: only m's additions lose anything, 2^-24 of 2^-48 of the sum.  Every
// operation rounds once and is never fused, so the error terms are exact.  FP32's
// range holds the squares: pixels are at most 2^31 (128 times the 2^24 at which a
// float stops counting), and what falls below 2^-149 is that small in the sum.
struct TripleSum {
    float h = 0.0f, l = 0.0f, m = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        float e;
        two_sum(h, x, h, e);
        add_low(e);
    }
    __device__ __forceinline__ void add_low(float x)
    {
        float e;
        two_sum(l, x, l, e);
        m = __fadd_rn(m, e);
    }
    __device__ __forceinline__ void add(const TripleSum &o)
    {
        add(o.h);
        add_low(o.l);
        m = __fadd_rn(m, o.m);
    }
    __device__ __forceinline__ TripleSum of_lane(int mask) const  // lane ^ mask
    {
        TripleSum o;
        o.h = __shfl_xor_sync(0xffffffffu, h, mask);
        o.l = __shfl_xor_sync(0xffffffffu, l, mask);
        o.m = __shfl_xor_sync(0xffffffffu, m, mask);
        return o;
    }
    __device__ __forceinline__ double value() const { return (double)h + ((double)l + (double)m); }
};

// v and v^2 of one pixel into the two sums; the square is p + e exactly.
__device__ __forceinline__ void add_moments(TripleSum &m1, TripleSum &m2, float v)
{
    const float p = __fmul_rn(v, v);
    m1.add(v);
    m2.add(p);
    m2.add_low(__fmaf_rn(v, v, -p));
}

// Four adjacent pixels from i on (VEC: an aligned quad), 0 past the image.
template <bool VEC>
__device__ __forceinline__ float4 load4(const float *a, size_t i, size_t P)
{
    if (VEC && i + 4 <= P) return *reinterpret_cast<const float4 *>(a + i);
    float4 v;
    v.x = i < P ? a[i] : 0.0f;
    v.y = i + 1 < P ? a[i + 1] : 0.0f;
    v.z = i + 2 < P ? a[i + 2] : 0.0f;
    v.w = i + 3 < P ? a[i + 3] : 0.0f;
    return v;
}

template <bool VEC>
__global__ void __launch_bounds__(kFwlThreads)
fwl_sums_kernel(const float *__restrict__ comp, const float *__restrict__ uncomp, size_t P,
                double *__restrict__ partial, unsigned *__restrict__ arrived,
                double *__restrict__ out)
{
    constexpr int kWarps = kFwlThreads / 32;
    static_assert(kWarps == 8, "a warp adds the eight warps' four sums");
    __shared__ TripleSum sh[4][kWarps];
    __shared__ double shd[kWarps];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kQuads = 4;  // quads of a thread between additions in double
    double v = 0.0;            // warp 0, lane 8 k: the block's sum k
    const size_t step = (size_t)gridDim.x * kFwlThreads * 4;
    for (size_t i0 = (size_t)blockIdx.x * kFwlThreads * 4; i0 < P; i0 += step * kQuads) {
        float4 c[kQuads], u[kQuads];
#pragma unroll
        for (int k = 0; k < kQuads; ++k) {
            const size_t i = i0 + threadIdx.x * 4 + step * k;
            c[k] = load4<VEC>(comp, i, P);
            u[k] = load4<VEC>(uncomp, i, P);
        }
        TripleSum m[4];
#pragma unroll
        for (int k = 0; k < kQuads; ++k) {
            add_moments(m[0], m[1], c[k].x);
            add_moments(m[2], m[3], u[k].x);
            add_moments(m[0], m[1], c[k].y);
            add_moments(m[2], m[3], u[k].y);
            add_moments(m[0], m[1], c[k].z);
            add_moments(m[2], m[3], u[k].z);
            add_moments(m[0], m[1], c[k].w);
            add_moments(m[2], m[3], u[k].w);
        }
        // over the warp, then over the warps, still in triples.  The lanes share
        // the four sums: halves keep two each, quarters one each (6 additions of
        // triples, 20 with every lane carrying all four)
        const bool hi = lane & 16, hi8 = lane & 8;
        TripleSum a = hi ? m[2] : m[0], b = hi ? m[3] : m[1];
        a.add((hi ? m[0] : m[2]).of_lane(16));
        b.add((hi ? m[1] : m[3]).of_lane(16));
        TripleSum q = hi8 ? b : a;
        q.add((hi8 ? a : b).of_lane(8));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) q.add(q.of_lane(o));
        __syncthreads();  // the last pass's sums are read
        if (lane % 8 == 0) sh[lane / 8][warp] = q;  // quarter k has sum k
        __syncthreads();
        if (warp == 0) {
            TripleSum t = sh[lane / kWarps][lane % kWarps];
#pragma unroll
            for (int o = kWarps / 2; o > 0; o >>= 1) t.add(t.of_lane(o));
            if (lane % kWarps == 0) v += t.value();
        }
    }
    if (warp == 0) {
        if (lane % kWarps == 0) {
            partial[blockIdx.x * 4 + lane / kWarps] = v;
            __threadfence();
        }
        __syncwarp();
        if (lane == 0) s_last = atomicAdd(arrived, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the blocks' sums: two warps a sum, lane by lane, then down the lanes
    double t = 0.0;
    for (int b = threadIdx.x % 64; b < (int)gridDim.x; b += 64)
        t += __ldcg(&partial[b * 4 + threadIdx.x / 64]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) shd[warp] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        const double n = (double)P;
        const double mc = (shd[0] + shd[1]) / n, mu = (shd[4] + shd[5]) / n;
        const double var_c = (shd[2] + shd[3]) / n - mc * mc;
        const double var_u = (shd[6] + shd[7]) / n - mu * mu;
        out[0] = var_u > 0.0 ? var_c / var_u : 1.0;
        out[1] = var_c;
        out[2] = var_u;
    }
}

}  // namespace

extern "C" {

size_t ebof_fwl_scratch_bytes(int32_t width, int32_t height)
{
    if (width < 1 || height < 1) return 0;
    const size_t P = (size_t)width * height;
    return 2 * align256(sizeof(float) * P) + align256(sizeof(double) * 4 * kFwlPartialBlocks);
}

ebof_status ebof_fwl(const uint16_t *d_x, const uint16_t *d_y, const int64_t *d_t,
                     const int8_t *d_p, int64_t n_events, int64_t t_begin, int64_t t_end,
                     const float *d_flow, int32_t width, int32_t height, void *d_scratch,
                     double *d_out, void *cuda_stream)
{
    if (!d_flow || !d_scratch || !d_out || width < 1 || height < 1 || width > 16384 ||
        height > 16384 || n_events < 0 || t_end < t_begin ||
        (n_events > 0 && (!d_x || !d_y || !d_t)))
        return EBOF_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    cudaGetLastError();
    const size_t P = (size_t)width * height;
    char *base = (char *)d_scratch;
    float *comp = (float *)base;
    float *uncomp = (float *)(base + align256(sizeof(float) * P));
    double *partial = (double *)(base + 2 * align256(sizeof(float) * P));
    unsigned *arrived = (unsigned *)(partial + 4 * kFwlBlocks);
    cudaMemsetAsync(base, 0, ebof_fwl_scratch_bytes(width, height), st);
    if (n_events > 0) {
        const int64_t want = (n_events + kFwlThreads - 1) / kFwlThreads;
        const int blocks = (int)(want < 152 * 16 ? want : 152 * 16);
        fwl_splat_kernel<<<blocks, kFwlThreads, 0, st>>>(d_x, d_y, d_t, d_p, n_events, t_begin,
                                                         t_end, d_flow, width, height, comp,
                                                         uncomp);
        ebof::g_launches.fetch_add(1);
    }
    const size_t want = (P + 4 * kFwlThreads - 1) / (4 * kFwlThreads);
    const bool quads = ((uintptr_t)comp & 15) == 0;  // uncomp lies a multiple of 256 bytes on
    (quads ? fwl_sums_kernel<true> : fwl_sums_kernel<false>)
        <<<(int)std::min<size_t>(want, kFwlBlocks), kFwlThreads, 0, st>>>(comp, uncomp, P, partial,
                                                                        arrived, d_out);
    ebof::g_launches.fetch_add(1);
    return cudaGetLastError() == cudaSuccess ? EBOF_OK : EBOF_ERR_CUDA;
}

}  // extern "C"
