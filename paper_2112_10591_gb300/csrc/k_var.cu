// k_var.cu -- variational refinement (reading F6): two kernels per
// fixed-point iteration.
//
// var_coeff_kernel: a block stages U and the warped image I1(x + U) for a tile
// of 64 columns plus 2 px in shared memory, builds the derivatives of the
// warped image and the smoothness weights, and writes every pixel's 2x2 linear
// system (data and gradient-constancy terms normalised, weights lagged at
// dU = 0): omega/a11, omega/a22 (the SOR relaxation factor folded into the
// inverted diagonal), a12, b1, b2 and the smoothness weight, as six planes.
// Everything is done on pairs of pixels, half a row or 32 columns apart, with
// packed FP32 operations.
// What bounds it: issue slots (a scalar form took 340 instructions a pixel row
// of 32) and, once those are halved, the latency of the flow and the image's
// taps, which is why the rows are staged by a block of independent threads: a
// warp that walks its columns down with the rows in registers needs as few
// instructions but only four warps a scheduler fit.  Measured (the first form:
// scalar, a column walk from 1024 px and 32x12 tiles below): 1280x720 14.3 -> 13.0
// us for one frame, 103 -> 85 for eight; 640x360 34 -> 24 for eight.
//
// SOR: one block owns a 64x64 region and refines the flow of its
// (64 - 2R)^2 interior, R = 2 * sweeps - 1.  It loads the region's linear
// systems into registers and runs the red-black SOR sweeps there: a thread
// owns a 2-column x 4-row strip, so one horizontal neighbour is its own and
// the other is a lane shuffle away, and the pixels at strip ends are exchanged
// through shared memory once per half sweep.  The region border keeps
// du = 0; after h half sweeps only pixels within h - 1 px of that border
// differ from the whole-image red-black iteration, and those lie in the
// discarded halo, so the interior is exactly the whole-image iteration (up to
// floating-point rounding).  It writes U + dU for its interior.
//
// What bounds it: the issue slots and the latency between the barriers of the
// half sweeps (four warps a scheduler; the register file holds no more), and
// the L2 bandwidth of the planes, read 1.93 times for the halo.  So (u, v) are
// updated as packed pairs, only the pixels just updated are exchanged, the
// first half sweep (whose neighbours are 0) runs without an exchange, the edge
// weights are rebuilt from one plane, regions begin on odd columns that every
// buffer aligns to 8 bytes, and the interior's flow is fetched behind the
// sweeps.  Measured per 1280x720 launch, against the scalar form of 7 planes
// and a full exchange: 18.3 -> 16.4 us for one frame, 165 -> 118 us for eight.
//
// var_sor_tma_kernel: the same regions in a persistent grid (one block per
// SM).  One thread loads each region's planes into shared memory with a
// single TMA tensor copy (cp.async.bulk.tensor, completion on an mbarrier);
// once every thread has moved its values into registers, the copy of the
// block's next region is issued and runs during the sweeps.  The box starts at
// the region's first column rounded down to the 16-byte rule of tensor copies
// and is 4 columns wider; elements outside the level are filled with zero, as
// the direct loads do, so both kernels give the same result.  With one region an
// SM there is no copy to hide.  Measured against the direct form: 11.2 us both for
// 168 regions, 11.4 and 12.1 for 224, 14.7 and 16.4 for 448, 25.8 and 30.7 for
// 896, 47.5 and 63.4 for 1792, 89.6 and 117.7 for 3584.
#include "dev_common.cuh"
#include "ebof_internal.cuh"
#include "profiler.cuh"
#include "seg.cuh"

#include <mutex>

namespace ebof {

namespace {

constexpr int kVR = 64;                  // region side
constexpr int kVS = 4;                   // rows per thread strip
constexpr int kVWarps = kVR / kVS;       // warps per block (stacked strips)
constexpr int kVThreads = 32 * kVWarps;  // 512
constexpr int kVSmallRows = 32;          // region rows of the small form
constexpr int kVSmallVS = 2;             // and its rows per strip
static_assert(kVSmallRows / kVSmallVS == kVWarps, "both forms run 16 warps");
// Coefficient planes of a pixel's system: omega/a11, omega/a22, a12, b1, b2
// and the smoothness weight.  An edge's weight is the mean of its two pixels'
// smoothness weights, one sum and one product that the sweeps' kernels do
// themselves: one plane instead of the left and upper edge weights' two, a
// seventh of the bytes they load.
//
// The planes are stored one element to the right of their base, column x at
// x + 1: a region starts on an odd column (its halo is odd, its interior
// even), so a lane's two columns are then one aligned 8-byte pair.  The flow
// buffers are offset the same way by their owner.
enum { kCI11 = 0, kCI22, kCA12, kCB1, kCB2, kCAS, kCPlanes };
constexpr int kCoefShift = 1;

constexpr int kTmaBoxW = kVR + 4;  // region columns + the rounding of the box start
constexpr size_t kTmaCoefFloats = (size_t)kCPlanes * kVR * kTmaBoxW;
// the interior's flow, staged while the sweeps run: (u, v) pairs of a strip's rows
template <int VS, int WARPS>
constexpr size_t flow_stage_bytes()
{
    return (size_t)VS * 2 * WARPS * 32 * sizeof(float2);
}
// A region's interior of the flow: its columns and the rounding of the box
// start, as many rows, two planes.  The largest interior (halo 1) is 62 wide.
__host__ __device__ constexpr int u_box_width(int tile) { return (tile + 3 + 3) & ~3; }
constexpr size_t kTmaSmemBytes =
    (kTmaCoefFloats + (2 * (kVR - 2) + kVS - 1) * u_box_width(kVR - 2)) * sizeof(float);
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float2 ld2(const float *p)
{
    return *reinterpret_cast<const float2 *>(p);
}

// A thread's strip of 2 columns x VS rows: the pixels' systems, the weights of
// their edges (right: of column 1 only, column 0's is column 1's left one;
// down: of the last row only) and (du, dv).
template <int VS>
struct Strip {
    float i11[VS][2], i22[VS][2], a12[VS][2];
    pair_t b[VS][2];
    float wl[VS][2], wr[VS], wu[VS][2], wd[2];
    pair_t d[VS][2];
};

// Shared memory of the strip ends, double-buffered by half sweep.  Of a strip's
// first and last row only the pixels just updated are published: a half sweep
// reads the other colour.  top[.][k] is warp k's first row, bot[.][k + 1] its
// last; the entries past either end stay 0.
template <int WARPS>
struct StripEnds {
    pair_t top[2][WARPS + 1][32], bot[2][WARPS + 1][32];
};
template <int WARPS>
__device__ __forceinline__ void clear_ends(StripEnds<WARPS> &x)
{
    const int t = threadIdx.x, lane = t & 31, k = (t >> 5) & 1;
    if (t < 64) x.bot[k][0][lane] = 0;
    else if (t < 128) x.top[k][WARPS][lane] = 0;
}

// One red-black half sweep: row r's pixel of column (Q + r) & 1.  up, dn: the
// neighbours above the strip's first and below its last row.
template <int VS, int Q>
__device__ __forceinline__ void sor_half(Strip<VS> &s, pair_t up, pair_t dn, pair_t om1)
{
#pragma unroll
    for (int r = 0; r < VS; ++r) {
        const int q = (Q + r) & 1;  // compile-time after unrolling
        // lane 0's left and lane 31's right neighbours lie outside the
        // region: the shuffles return the lane's own (finite) values there,
        // and the weights of those edges are 0
        pair_t l, rt;
        if (q == 0) {
            const float2 n = upk(s.d[r][1]);
            l = pk(__shfl_up_sync(kFull, n.x, 1), __shfl_up_sync(kFull, n.y, 1));
            rt = s.d[r][1];
        } else {
            const float2 n = upk(s.d[r][0]);
            rt = pk(__shfl_down_sync(kFull, n.x, 1), __shfl_down_sync(kFull, n.y, 1));
            l = s.d[r][0];
        }
        const pair_t u = r > 0 ? s.d[r > 0 ? r - 1 : 0][q] : up;
        const pair_t d = r < VS - 1 ? s.d[r < VS - 1 ? r + 1 : r][q] : dn;
        const float wl = s.wl[r][q], wr = q == 0 ? s.wl[r][1] : s.wr[r];
        const float wu = s.wu[r][q], wd = r < VS - 1 ? s.wu[r < VS - 1 ? r + 1 : r][q] : s.wd[q];
        // i11 = omega / a11, i22 = omega / a22; fixed rounding order (every
        // SOR layout gives the same values)
        pair_t t = ffma2(pk(wl, wl), l, s.b[r][q]);
        t = ffma2(pk(wr, wr), rt, t);
        t = ffma2(pk(wu, wu), u, t);
        t = ffma2(pk(wd, wd), d, t);
        const float2 tt = upk(t), own = upk(s.d[r][q]), o = upk(fmul2(om1, s.d[r][q]));
        const float nu = ffma(ffma(-s.a12[r][q], own.y, tt.x), s.i11[r][q], o.x);
        const float nv = ffma(ffma(-s.a12[r][q], nu, tt.y), s.i22[r][q], o.y);
        s.d[r][q] = pk(nu, nv);
    }
}

// Publishes the pixels that the last half sweep updated (row r's of column
// (Q + r) & 1) at the strip's ends, waits for the block, and reads the
// neighbours' of the next half sweep.
template <int VS, int WARPS, int Q>
__device__ __forceinline__ void swap_ends(const Strip<VS> &s, StripEnds<WARPS> &x, int buf,
                                          int lane, int wp, pair_t &up, pair_t &dn)
{
    x.top[buf][wp][lane] = s.d[0][Q];
    x.bot[buf][wp + 1][lane] = s.d[VS - 1][(Q + VS - 1) & 1];
    __syncthreads();
    up = x.bot[buf][wp][lane];
    dn = x.top[buf][wp + 1][lane];
}

// n_half half sweeps from dU = 0; P: the column of the red pixel in the strip's
// first row.  The first one has no neighbour to read, so n_half - 1 barriers.
template <int VS, int WARPS, int P>
__device__ __forceinline__ void sor_sweeps_p(Strip<VS> &s, StripEnds<WARPS> &x, int lane, int wp,
                                             int n_half, pair_t om1)
{
    if (n_half <= 0) return;
    sor_half<VS, P>(s, 0, 0, om1);
    pair_t up, dn;
#pragma unroll 1
    for (int hs = 1; hs < n_half; hs += 2) {
        swap_ends<VS, WARPS, P>(s, x, 0, lane, wp, up, dn);
        sor_half<VS, 1 - P>(s, up, dn, om1);
        if (hs + 1 < n_half) {
            swap_ends<VS, WARPS, 1 - P>(s, x, 1, lane, wp, up, dn);
            sor_half<VS, P>(s, up, dn, om1);
        }
    }
}

// par: parity of (x + y) at the strip's first pixel, the same in every warp
// (VS is even).
template <int VS, int WARPS>
__device__ __forceinline__ void sor_sweeps(Strip<VS> &s, StripEnds<WARPS> &x, int lane, int wp,
                                           int par, int n_half, float omega)
{
    static_assert((VS & 1) == 0, "one parity per block");
    const float o = 1.0f - omega;
    const pair_t om1 = pk(o, o);
#pragma unroll
    for (int r = 0; r < VS; ++r) s.d[r][0] = s.d[r][1] = 0;
    if (par == 0)
        sor_sweeps_p<VS, WARPS, 0>(s, x, lane, wp, n_half, om1);
    else
        sor_sweeps_p<VS, WARPS, 1>(s, x, lane, wp, n_half, om1);
}

// The strip's edge weights from the smoothness weights of its rows and of the
// rows above and below it (as[0], as[VS + 1]); (gx, gy): its first pixel.  An
// edge that leaves the level (not INSIDE) or the region has weight 0; past the
// region's ends lie pixels whose dU stays 0.
template <int VS, bool INSIDE>
__device__ __forceinline__ void edge_weights(Strip<VS> &s, const float (&as)[VS + 2][2], int lane,
                                             bool first, bool last, int gx, int gy, int w, int h)
{
    auto mean = [](float a, float b) { return fmul(0.5f, fadd(a, b)); };
    const bool x0 = lane > 0 && (INSIDE || (gx > 0 && gx < w));
    const bool x1 = INSIDE || (gx >= 0 && gx + 1 < w);
    const bool x2 = lane < 31 && (INSIDE || (gx + 1 >= 0 && gx + 2 < w));
#pragma unroll
    for (int r = 0; r < VS; ++r) {
        const float l = __shfl_up_sync(kFull, as[r + 1][1], 1);
        const float n = __shfl_down_sync(kFull, as[r + 1][0], 1);
        s.wl[r][0] = x0 ? mean(as[r + 1][0], l) : 0.0f;
        s.wl[r][1] = x1 ? mean(as[r + 1][1], as[r + 1][0]) : 0.0f;
        s.wr[r] = x2 ? mean(as[r + 1][1], n) : 0.0f;
        const bool yu = !(r == 0 && first) && (INSIDE || (gy + r > 0 && gy + r < h));
#pragma unroll
        for (int q = 0; q < 2; ++q) s.wu[r][q] = yu ? mean(as[r + 1][q], as[r][q]) : 0.0f;
    }
    const bool yd = !last && (INSIDE || (gy + VS > 0 && gy + VS < h));
#pragma unroll
    for (int q = 0; q < 2; ++q) s.wd[q] = yd ? mean(as[VS + 1][q], as[VS][q]) : 0.0f;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void copy_async8(uint32_t dst, const float *src, int bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}

// Where a thread's strip lies: the region's first pixel, the strip's, and
// which of its pixels the region outputs.
template <int VS, int WARPS>
struct StripPlace {
    int gx, gy;    // the strip's first pixel
    int pitch, w, h;
    bool c0, c1;   // column 0 / 1 is an output column
    int r0, r1;    // rows r0 <= r < r1 of the strip are output rows
    __device__ __forceinline__ StripPlace(int bx, int by, int R, int w_, int h_, int pitch_,
                                          int lane, int wp)
        : pitch(pitch_), w(w_), h(h_)
    {
        const int tx = kVR - 2 * R, ty = VS * WARPS - 2 * R;
        gx = bx * tx - R + 2 * lane;
        gy = by * ty - R + wp * VS;
        c0 = 2 * lane >= R && 2 * lane < R + tx && gx < w;
        c1 = 2 * lane + 1 >= R && 2 * lane + 1 < R + tx && gx + 1 < w;
        r0 = max(R - wp * VS, 0);
        r1 = min(min(R + ty - wp * VS, VS), h - gy);
    }
    // the region lies in the level (block-uniform)
    __device__ __forceinline__ bool inside(int lane, int wp) const
    {
        const int rx = gx - 2 * lane, ry = gy - wp * VS;
        return rx >= 0 && ry >= 0 && rx + kVR <= w && ry + VS * WARPS <= h;
    }
};

// Starts the copy of the output pixels' flow into the thread's own slots of
// su ([VS][2][threads] pairs), read back by store_flow: the loads' latency
// passes behind the sweeps.
template <int VS, int WARPS>
__device__ __forceinline__ void stage_flow(const StripPlace<VS, WARPS> &p, const float *Uin,
                                           size_t plane, uint32_t su)
{
    const int bytes = (p.c0 || p.c1) ? (p.gx + 1 < p.w ? 8 : 4) : 0;
#pragma unroll
    for (int r = 0; r < VS; ++r)
        if (bytes && r >= p.r0 && r < p.r1) {
            const float *c = Uin + (p.gy + r) * p.pitch + p.gx;
            copy_async8(su + (2 * r) * 32 * WARPS * 8, c, bytes);
            copy_async8(su + (2 * r + 1) * 32 * WARPS * 8, c + plane, bytes);
        }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The output pixels of a strip's row, o: its first pixel's offset.  The lanes
// at the interior's ends own one pixel: one store for either, not a branch each.
template <int VS, int WARPS>
__device__ __forceinline__ void store_row(const StripPlace<VS, WARPS> &p, float *Uout,
                                          size_t plane, int o, float2 u, float2 v)
{
    if (p.c0 && p.c1) {
        *reinterpret_cast<float2 *>(Uout + o) = u;
        *reinterpret_cast<float2 *>(Uout + plane + o) = v;
    } else if (p.c0 || p.c1) {
        const int e = p.c0 ? o : o + 1;
        Uout[e] = p.c0 ? u.x : u.y;
        (Uout + plane)[e] = p.c0 ? v.x : v.y;
    }
}

// U + dU of the output pixels.  staged: this thread's slots after stage_flow.
template <int VS, int WARPS>
__device__ __forceinline__ void store_flow(const StripPlace<VS, WARPS> &p, const Strip<VS> &s,
                                           float *Uout, size_t plane, const float2 *staged)
{
    asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
    for (int r = 0; r < VS; ++r) {
        if (r < p.r0 || r >= p.r1) continue;
        const int o = (p.gy + r) * p.pitch + p.gx;
        const float2 d0 = upk(s.d[r][0]), d1 = upk(s.d[r][1]);
        const float2 u = staged[(2 * r) * 32 * WARPS];
        const float2 v = staged[(2 * r + 1) * 32 * WARPS];
        store_row(p, Uout, plane, o, make_float2(u.x + d0.x, u.y + d1.x),
                  make_float2(v.x + d0.y, v.y + d1.y));
    }
}

// A region of 64 columns x VS * WARPS rows, its coefficients loaded straight
// into registers.  su: the block's flow stage.
template <int VS, int WARPS>
__device__ __forceinline__ void sor_region(int bx, int by, int f, int w, int h, int pitch,
                                           const float *__restrict__ Uinb,
                                           float *__restrict__ Uoutb, size_t ufs, size_t plane,
                                           const float *__restrict__ coefb, size_t cfs, int R,
                                           int n_half, float omega, StripEnds<WARPS> &ends,
                                           float2 *su)
{
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const StripPlace<VS, WARPS> p(bx, by, R, w, h, pitch, lane, wp);
    const float *Uin = Uinb + (size_t)f * ufs;
    const float *cf = coefb + (size_t)f * cfs;
    const int pl = (int)plane;  // offsets within a frame fit in 32 bits
    const bool inside = p.inside(lane, wp);
    const bool first = wp == 0, last = wp == WARPS - 1;
    Strip<VS> s;
    float as[VS + 2][2];
    if (inside) {
        // the whole region lies in the level: loads without bounds tests
        const float *c0 = cf + p.gy * pitch + p.gx;
#pragma unroll
        for (int r = 0; r < VS; ++r) {
            const float *c = c0 + r * pitch;
            const float2 i1 = ld2(c + kCI11 * pl), i2 = ld2(c + kCI22 * pl);
            const float2 a = ld2(c + kCA12 * pl), g = ld2(c + kCAS * pl);
            const float2 b1 = ld2(c + kCB1 * pl), b2 = ld2(c + kCB2 * pl);
            s.i11[r][0] = i1.x, s.i11[r][1] = i1.y;
            s.i22[r][0] = i2.x, s.i22[r][1] = i2.y;
            s.a12[r][0] = a.x, s.a12[r][1] = a.y;
            as[r + 1][0] = g.x, as[r + 1][1] = g.y;
            s.b[r][0] = pk(b1.x, b2.x);
            s.b[r][1] = pk(b1.y, b2.y);
        }
        const float *ca = c0 + kCAS * pl;
        const float2 z = make_float2(0.0f, 0.0f);
        const float2 gu = first ? z : ld2(ca - pitch);
        const float2 gd = last ? z : ld2(ca + VS * pitch);
        as[0][0] = gu.x, as[0][1] = gu.y;
        as[VS + 1][0] = gd.x, as[VS + 1][1] = gd.y;
    } else {
#pragma unroll
        for (int r = -1; r <= VS; ++r) {
            const int gy = p.gy + r;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int gx = p.gx + q;
                const bool in = gx >= 0 && gx < w && gy >= 0 && gy < h;
                const float *c = cf + (in ? gy * pitch + gx : 0);
                auto ld = [&](int k) { return in ? c[k * pl] : 0.0f; };
                as[r + 1][q] = ld(kCAS);
                if (r >= 0 && r < VS) {
                    s.i11[r][q] = ld(kCI11);
                    s.i22[r][q] = ld(kCI22);
                    s.a12[r][q] = ld(kCA12);
                    s.b[r][q] = pk(ld(kCB1), ld(kCB2));
                }
            }
        }
    }
    float2 *slot = su + threadIdx.x;
    stage_flow(p, Uin, plane, smem_u32(slot));
    clear_ends(ends);
    if (inside)
        edge_weights<VS, true>(s, as, lane, first, last, p.gx, p.gy, w, h);
    else
        edge_weights<VS, false>(s, as, lane, first, last, p.gx, p.gy, w, h);
    sor_sweeps<VS, WARPS>(s, ends, lane, wp, (p.gx + p.gy) & 1, n_half, omega);
    store_flow(p, s, Uoutb + (size_t)f * ufs, plane, slot);
}

template <int VS>
__global__ void __launch_bounds__(kVThreads, 1)
var_sor_kernel(int w, int h, int pitch, const float *__restrict__ Uinb,
               float *__restrict__ Uoutb, size_t ufs, size_t plane,
               const float *__restrict__ coefb, size_t cfs, int R, int n_half, float omega)
{
    chain_begin();
    extern __shared__ float2 su[];
    __shared__ StripEnds<kVWarps> ends;
    sor_region<VS, kVWarps>(blockIdx.x, blockIdx.y, blockIdx.z, w, h, pitch, Uinb, Uoutb, ufs,
                            plane, coefb, cfs, R, n_half, omega, ends, su);
}

// The 64 x 64 regions of several groups' levels in one launch.
__global__ void __launch_bounds__(kVThreads, 1)
seg_var_sor_kernel(const __grid_constant__ SegTable<SegSor> tab)
{
    extern __shared__ float2 su[];
    __shared__ StripEnds<kVWarps> ends;
    int b;
    const SegSor &a = seg_of(tab, b);
    const int r = b / a.gx;
    sor_region<kVS, kVWarps>(b % a.gx, r % a.gy, r / a.gy, a.w, a.h, a.pitch, a.Uin, a.Uout,
                             a.ufs, a.plane, a.coef + kCoefShift, a.cfs, a.R, a.n_half, a.omega,
                             ends, su);
}

// Bounded wait for the mbarrier phase with the given parity: at most
// `limit` try-wait rounds.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, long long limit)
{
    for (long long it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Regions of large levels and batches, one block an SM over them all: the
// tensor copy of the next region's coefficients runs behind the sweeps of this
// one, and so does that of this one's flow.  Bound by the sweeps, 4700 of a
// region's 7700 cycles (9900 before): between two regions one thread's work, or
// a few warps', is the block's, which waits for them at the next barrier.  So
// the next region's place is found by additions instead of divisions, the flow
// comes by one tensor copy instead of eight 8-byte copies a thread, and the
// output's loads and stores stand without branches between them.  The copies
// write a buffer only after the barrier that follows its last reads.
// 1280 x 720, ten half sweeps, against a region a block: one frame 16.4 -> 14.6
// us, eight 118 -> 90.
__global__ void __launch_bounds__(kVThreads, 1)
var_sor_tma_kernel(const __grid_constant__ CUtensorMap cmap,
                   const __grid_constant__ CUtensorMap umap, int w, int h, int pitch,
                   float *__restrict__ Uoutb, size_t ufs, size_t plane, int R, int nrx, int nry,
                   int total, int n_half, float omega, long long wait_limit,
                   long long flow_wait_limit, int *err)
{
    chain_begin();
    extern __shared__ __align__(1024) float tsm[];
    float *cbuf = tsm;                    // [kCPlanes][kVR][kTmaBoxW]
    const float *ubuf = tsm + kTmaCoefFloats;  // [2][tile][u_box_width(tile)]
    __shared__ StripEnds<kVWarps> ends;
    __shared__ __align__(8) unsigned long long mbar_s[2];
    const uint32_t cbar = smem_u32(&mbar_s[0]), ubar = smem_u32(&mbar_s[1]);
    const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
    const int tile = kVR - 2 * R, uw = u_box_width(tile);
    const unsigned long long cmap_addr = (unsigned long long)&cmap;
    const unsigned long long umap_addr = (unsigned long long)&umap;
    const uint32_t cdst = smem_u32(cbuf), udst = smem_u32(ubuf);

    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(cbar) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(ubar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    clear_ends(ends);
    __syncthreads();
    auto copy = [](uint32_t dst, unsigned long long map, int x, int y, int f, uint32_t bar,
                   int floats) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                     "r"((unsigned)(floats * sizeof(float)))
                     : "memory");
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes "
            "[%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
            "l"(map), "r"(x), "r"(y), "r"(0), "r"(f), "r"(bar)
            : "memory");
    };
    // the tensor maps' column x + 1 is the level's column x
    auto issue = [&](int rx, int ry, int f) {
        copy(cdst, cmap_addr, (rx * tile - R + kCoefShift) & ~3, ry * tile - R, f, cbar,
             (int)kTmaCoefFloats);
    };
    const int per_frame = nrx * nry;
    int f = blockIdx.x / per_frame, ry = (blockIdx.x - f * per_frame) / nrx;
    int rx = blockIdx.x - f * per_frame - ry * nrx;
    const int sf = gridDim.x / per_frame, sy = (gridDim.x - sf * per_frame) / nrx;
    const int sx = gridDim.x - sf * per_frame - sy * nrx;
    if (t == 0 && (int)blockIdx.x < total) issue(rx, ry, f);
    uint32_t parity = 0;
    bool late = false;
#pragma unroll 1
    for (int r = blockIdx.x; r < total; r += gridDim.x) {
        late |= !mbar_wait(cbar, parity, wait_limit);
        const StripPlace<kVS, kVWarps> p(rx, ry, R, w, h, pitch, lane, wp);
        const bool first = wp == 0, last = wp == kVWarps - 1;
        // a left border's column -1 holds the end of the row before: masked
        const bool out = p.gx < 0;
        Strip<kVS> s;
        float as[kVS + 2][2];
        constexpr int P = kVR * kTmaBoxW;
        const float *c0 = cbuf + wp * kVS * kTmaBoxW + ((rx * tile - R + kCoefShift) & 3) + 2 * lane;
        auto ld = [&](const float *c) {
            float2 v = *reinterpret_cast<const float2 *>(c);
            if (out) v.x = 0.0f;
            return v;
        };
#pragma unroll
        for (int k = 0; k < kVS; ++k) {
            const float *c = c0 + k * kTmaBoxW;
            const float2 i1 = ld(c + kCI11 * P), i2 = ld(c + kCI22 * P), a = ld(c + kCA12 * P);
            const float2 b1 = ld(c + kCB1 * P), b2 = ld(c + kCB2 * P), g = ld(c + kCAS * P);
            s.i11[k][0] = i1.x, s.i11[k][1] = i1.y;
            s.i22[k][0] = i2.x, s.i22[k][1] = i2.y;
            s.a12[k][0] = a.x, s.a12[k][1] = a.y;
            as[k + 1][0] = g.x, as[k + 1][1] = g.y;
            s.b[k][0] = pk(b1.x, b2.x);
            s.b[k][1] = pk(b1.y, b2.y);
        }
        const float *ca = c0 + kCAS * P;
        const float2 z = make_float2(0.0f, 0.0f);
        const float2 gu = first ? z : ld(ca - kTmaBoxW), gd = last ? z : ld(ca + kVS * kTmaBoxW);
        as[0][0] = gu.x, as[0][1] = gu.y;
        as[kVS + 1][0] = gd.x, as[kVS + 1][1] = gd.y;
        // the next region
        int nx = rx + sx, ny = ry + sy, nf = f + sf;
        if (nx >= nrx) nx -= nrx, ++ny;
        if (ny >= nry) ny -= nry, ++nf;
        // every thread holds its coefficients and has read the last region's
        // flow: the buffers are free
        if (__syncthreads_or(late)) {
            if (t == 0) {
                atomicOr(err, kErrTimeout);
                // let the copies in flight land before the block exits (bounded
                // by the default limit, whatever the first wait's was); the
                // last flow's, if any, was of the phase before
                mbar_wait(cbar, parity, kWaitLimitDefault);
                if (r != (int)blockIdx.x) mbar_wait(ubar, parity ^ 1u, kWaitLimitDefault);
            }
            return;
        }
        const int ux = (rx * tile + kCoefShift) & ~3;
        if (t == 0) {
            copy(udst, umap_addr, ux, ry * tile, f, ubar, 2 * tile * uw);
            if (r + (int)gridDim.x < total) issue(nx, ny, nf);
        }
        if (p.inside(lane, wp))
            edge_weights<kVS, true>(s, as, lane, first, last, p.gx, p.gy, w, h);
        else
            edge_weights<kVS, false>(s, as, lane, first, last, p.gx, p.gy, w, h);
        sor_sweeps<kVS, kVWarps>(s, ends, lane, wp, (p.gx + p.gy) & 1, n_half, omega);
        late = !mbar_wait(ubar, parity, flow_wait_limit);
        parity ^= 1u;
        if (p.r0 < p.r1) {
            // loads before the tests of what is stored; those of pixels that
            // are not may lie up to three rows past the tile, inside smem
            const bool both = p.c0 && p.c1 && !late, one = p.c0 != p.c1 && !late;
            const float *u0 = ubuf + (p.gy - ry * tile) * uw + (p.gx + kCoefShift - ux);
            if (!p.c0 && !p.c1) u0 = ubuf;
            float2 u[kVS], v[kVS];
#pragma unroll
            for (int k = 0; k < kVS; ++k) {
                const float2 d0 = upk(s.d[k][0]), d1 = upk(s.d[k][1]);
                const float2 a = *reinterpret_cast<const float2 *>(u0 + k * uw);
                const float2 b = *reinterpret_cast<const float2 *>(u0 + (tile + k) * uw);
                u[k] = make_float2(a.x + d0.x, a.y + d1.x);
                v[k] = make_float2(b.x + d0.y, b.y + d1.y);
            }
            float *q = Uoutb + (size_t)f * ufs + p.gy * pitch + p.gx;
#pragma unroll
            for (int k = 0; k < kVS; ++k, q += pitch) {
                const bool row = k >= p.r0 && k < p.r1;
                if (row && both) {
                    *reinterpret_cast<float2 *>(q) = u[k];
                    *reinterpret_cast<float2 *>(q + plane) = v[k];
                }
                // the lanes at the interior's ends own one pixel
                if (row && one) {
                    q[p.c0 ? 0 : 1] = p.c0 ? u[k].x : u[k].y;
                    q[plane + (p.c0 ? 0 : 1)] = p.c0 ? v[k].x : v[k].y;
                }
            }
        }
        rx = nx, ry = ny, f = nf;
    }
    if (__syncthreads_or(late) && t == 0) {  // the last region's flow came late
        atomicOr(err, kErrTimeout);
        mbar_wait(ubar, parity ^ 1u, kWaitLimitDefault);
    }
}

// ---------------------------------------------------------------- resident levels
__device__ __forceinline__ pair_t dup(float a) { return pk(a, a); }
__device__ __forceinline__ pair_t neg2(pair_t a)
{
    const float2 v = upk(a);
    return pk(-v.x, -v.y);
}
// The approximate reciprocal square root and reciprocal, without the scaling
// of subnormal inputs that rsqrtf and __fdividef carry: the arguments here are
// at least 1e-6 and 0.01, and over the normal floats up to 2^126 both give the
// same bits.
__device__ __forceinline__ float rsqrt_normal(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_normal(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ pair_t psi_prime2(pair_t s2)
{
    const float2 v = upk(s2);
    return fmul2(dup(0.5f),
                 pk(rsqrt_normal(fadd(v.x, 1e-6f)), rsqrt_normal(fadd(v.y, 1e-6f))));
}

// The bilinear samples (bilinear_i's, bit for bit) at two clamped positions.
// The floor comes from an addition rounded down to the integers above 2^23,
// whose low bits are the column and row; both are held one short of the last,
// where the weight is 1 instead of a clamped neighbour's index (the level has
// at least two columns and rows).
struct Taps2 {
    float2 a, b, c, d;
    pair_t fx, fy;
};
template <typename T>
__device__ __forceinline__ Taps2 bil_taps2(const T *__restrict__ I, int w, int h, int pitch,
                                           pair_t x, pair_t y)
{
    constexpr float kInt = 8388608.0f;  // 2^23
    const float wm = (float)(w - 1), hm = (float)(h - 1);
    const float tw = kInt + (float)(w - 2), th = kInt + (float)(h - 2);
    const float2 px = upk(x), py = upk(y);
    const float x0 = fminf(fmaxf(px.x, 0.0f), wm), x1 = fminf(fmaxf(px.y, 0.0f), wm);
    const float y0 = fminf(fmaxf(py.x, 0.0f), hm), y1 = fminf(fmaxf(py.y, 0.0f), hm);
    const float tx0 = fminf(__fadd_rd(x0, kInt), tw), tx1 = fminf(__fadd_rd(x1, kInt), tw);
    const float ty0 = fminf(__fadd_rd(y0, kInt), th), ty1 = fminf(__fadd_rd(y1, kInt), th);
    Taps2 t;
    t.fx = fsub2(pk(x0, x1), fsub2(pk(tx0, tx1), dup(kInt)));
    t.fy = fsub2(pk(y0, y1), fsub2(pk(ty0, ty1), dup(kInt)));
    // the bits are 0x4b000000 + the integer: the products wrap alike
    const uint32_t bias = 0x4b000000u * (uint32_t)pitch + 0x4b000000u;
    const T *q0 = I + (__float_as_uint(ty0) * (uint32_t)pitch + __float_as_uint(tx0) - bias);
    const T *q1 = I + (__float_as_uint(ty1) * (uint32_t)pitch + __float_as_uint(tx1) - bias);
    t.a = make_float2(ldp(q0), ldp(q1));
    t.b = make_float2(ldp(q0 + 1), ldp(q1 + 1));
    t.c = make_float2(ldp(q0 + pitch), ldp(q1 + pitch));
    t.d = make_float2(ldp(q0 + pitch + 1), ldp(q1 + pitch + 1));
    return t;
}
__device__ __forceinline__ pair_t bil_lerp2(const Taps2 &t)
{
    const pair_t one = dup(1.0f), gx = fsub2(one, t.fx);
    const pair_t top = ffma2(t.fx, pk(t.b.x, t.b.y), fmul2(gx, pk(t.a.x, t.a.y)));
    const pair_t bot = ffma2(t.fx, pk(t.d.x, t.d.y), fmul2(gx, pk(t.c.x, t.c.y)));
    return ffma2(t.fy, bot, fmul2(fsub2(one, t.fy), top));
}

constexpr int kLvW = kVR + 4;  // staged columns: 64 and 2 around

// The windows of a tile of 64 columns, WH - 4 rows and 2 px around, from pixel
// (ex, ey), ex odd.
template <int WH>
struct Windows {
    float *U, *V, *W, *Ix, *Iy, *As;
    __device__ __forceinline__ explicit Windows(float *m)
        : U(m), V(U + kLvW * WH), W(V + kLvW * WH), Ix(W + kLvW * WH), Iy(Ix + kLvW * WH),
          As(Iy + kLvW * WH)
    {
    }
    static constexpr size_t kBytes = (size_t)6 * kLvW * WH * sizeof(float);
};
__device__ __forceinline__ pair_t ld_pair(const float *a)
{
    return *reinterpret_cast<const pair_t *>(a);
}
__device__ __forceinline__ void st_pair(float *a, pair_t v)
{
    *reinterpret_cast<pair_t *>(a) = v;
}

// The flow of the window and the warped image there.  Positions outside the
// level are those of the nearest pixel inside: the replicated borders of the
// differences.  inside: the window lies in the level (block-uniform).
// load(c0, c1, cy, u, v): the flow of KI pairs of pixels (c0, cy), (c1, cy);
// all of a thread's loads come before their first use.  A pair is half a row
// apart, so that a warp's taps lie side by side (adjacent pixels a pair spread
// them over twice the lines: 640 x 360 in one launch 60.0 us against 57.7).
template <int WH, int NT, int KI, typename T, class L>
__device__ __forceinline__ void stage_window(const Windows<WH> &m, const T *__restrict__ I1,
                                             int w, int h, int pitch, int ex, int ey, bool inside,
                                             L load)
{
    constexpr int NP = kLvW / 2, NI = NP * WH;
#pragma unroll 1
    for (int i0 = threadIdx.x; i0 < NI; i0 += NT * KI) {
        pair_t u[KI], v[KI];
        int c0[KI], c1[KI], cy[KI];
#pragma unroll
        for (int j = 0; j < KI; ++j) {
            const int i = min(i0 + NT * j, NI - 1);
            const int row = i / NP;
            c0[j] = ex + i - row * NP;
            c1[j] = c0[j] + NP;
            cy[j] = ey + row;
            if (!inside) {
                c0[j] = clampi(c0[j], 0, w - 1);
                c1[j] = clampi(c1[j], 0, w - 1);
                cy[j] = clampi(cy[j], 0, h - 1);
            }
        }
        load(c0, c1, cy, u, v);
        Taps2 tp[KI];
#pragma unroll
        for (int j = 0; j < KI; ++j)
            tp[j] = bil_taps2(I1, w, h, pitch, fadd2(pk((float)c0[j], (float)c1[j]), u[j]),
                              fadd2(dup((float)cy[j]), v[j]));
#pragma unroll
        for (int j = 0; j < KI; ++j) {
            const int i = i0 + NT * j;
            if (i < NI) {
                const int e = i + i / NP * NP;
                const float2 uu = upk(u[j]), vv = upk(v[j]), ww = upk(bil_lerp2(tp[j]));
                m.U[e] = uu.x;
                m.U[e + NP] = uu.y;
                m.V[e] = vv.x;
                m.V[e + NP] = vv.y;
                m.W[e] = ww.x;
                m.W[e + NP] = ww.y;
            }
        }
    }
}

// The flow of the pairs from its planes.
template <int KI>
__device__ __forceinline__ void load_planes(const float *__restrict__ a, size_t plane, int pitch,
                                            const int (&c0)[KI], const int (&c1)[KI],
                                            const int (&cy)[KI], pair_t (&u)[KI],
                                            pair_t (&v)[KI])
{
#pragma unroll
    for (int j = 0; j < KI; ++j) {
        const float *q = a + cy[j] * pitch;
        u[j] = pk(q[c0[j]], q[c1[j]]);
        v[j] = pk(q[plane + c0[j]], q[plane + c1[j]]);
    }
}

// The warped image's derivatives and the smoothness weights 1 px around the
// tile, rows 1 .. WH - 2 (the first and last column's left and right
// neighbours are another row's; nothing reads those results).
template <int WH, int NT>
__device__ __forceinline__ void derive_window(const Windows<WH> &m, float alpha_s)
{
    constexpr int NP = kLvW / 2;
#pragma unroll 1
    for (int i = NP + threadIdx.x; i < NP * (WH - 1); i += NT) {
        const int e = 2 * i;
        const pair_t half = dup(0.5f);
        const float2 u = upk(ld_pair(m.U + e)), v = upk(ld_pair(m.V + e));
        const float2 wc = upk(ld_pair(m.W + e));
        const float un = m.U[e + 2], vn = m.V[e + 2];
        const pair_t ix = pk(fsub(wc.y, m.W[e - 1]), fsub(m.W[e + 2], wc.x));
        const pair_t iy = fsub2(ld_pair(m.W + e + kLvW), ld_pair(m.W + e - kLvW));
        const pair_t ux = pk(fsub(u.y, u.x), fsub(un, u.y));
        const pair_t vx = pk(fsub(v.y, v.x), fsub(vn, v.y));
        const pair_t uy = fsub2(ld_pair(m.U + e + kLvW), pk(u.x, u.y));
        const pair_t vy = fsub2(ld_pair(m.V + e + kLvW), pk(v.x, v.y));
        const pair_t q = psi_prime2(ffma2(vy, vy, ffma2(vx, vx, ffma2(uy, uy, fmul2(ux, ux)))));
        st_pair(m.Ix + e, fmul2(half, ix));
        st_pair(m.Iy + e, fmul2(half, iy));
        st_pair(m.As + e, fmul2(dup(alpha_s), q));
    }
}

// The systems of pixels (gx, gy), (gx + D, gy), e the first one's place in the
// windows; i0, i0x, i0y: the template's values.  d1, d2: the diagonal; wl, wr,
// wu, wd: the edge weights, 0 where the edge leaves the level.
struct PairSystem {
    float2 d1, d2, a12, b1, b2, wl, wr, wu, wd;
};
template <int D, int WH>
__device__ __forceinline__ PairSystem pair_system(const Windows<WH> &m, int e, int gx, int gy,
                                                  int w, int h, bool inside, pair_t i0,
                                                  pair_t i0x, pair_t i0y, float delta,
                                                  float gamma)
{
    const float wm1 = (float)(w - 1), hm1 = (float)(h - 1);
    const pair_t half = dup(0.5f);
    // a window's values at the two pixels and beside them; of adjacent pixels
    // either is the other's neighbour
    auto at = [&](const float *q) { return D == 1 ? ld_pair(q + e) : pk(q[e], q[e + D]); };
    auto left = [&](const float *q, float2 c) {
        return make_float2(q[e - 1], D == 1 ? c.x : q[e + D - 1]);
    };
    auto right = [&](const float *q, float2 c) {
        return make_float2(D == 1 ? c.y : q[e + 1], q[e + D + 1]);
    };
    auto cd2 = [&](pair_t hi, pair_t lo) { return fmul2(half, fsub2(hi, lo)); };
    const bool top = !inside && gy <= 0, bottom = !inside && gy + 1 >= h;
    const pair_t ix = at(m.Ix), iy = at(m.Iy);
    const pair_t ixu = top ? ix : at(m.Ix - kLvW);
    const pair_t ixd = bottom ? ix : at(m.Ix + kLvW);
    const pair_t iyu = top ? iy : at(m.Iy - kLvW);
    const pair_t iyd = bottom ? iy : at(m.Iy + kLvW);
    const float2 ixv = upk(ix);
    // clamped neighbours along x
    const bool l0 = inside || gx > 0, r0 = inside || gx + 1 < w;
    const bool l1 = inside || gx + D > 0, r1 = inside || gx + D + 1 < w;
    const float2 ixl = left(m.Ix, ixv), ixr = right(m.Ix, ixv);
    const pair_t Ixx = fmul2(half, pk(fsub(r0 ? ixr.x : ixv.x, l0 ? ixl.x : ixv.x),
                                      fsub(r1 ? ixr.y : ixv.y, l1 ? ixl.y : ixv.y)));
    const pair_t Ixy = cd2(ixd, ixu), Iyy = cd2(iyd, iyu);
    const pair_t Iz = fsub2(at(m.W), i0);
    const pair_t Ixz = fsub2(ix, i0x), Iyz = fsub2(iy, i0y);
    const pair_t z2 = dup(kZeta2);
    const pair_t xx = fmul2(Ixx, Ixx), yy = fmul2(Ixy, Ixy);
    const float2 n1 = upk(fadd2(ffma2(iy, iy, fmul2(ix, ix)), z2));
    const float2 n2 = upk(fadd2(ffma2(Iyy, Iyy, ffma2(fmul2(dup(2.0f), Ixy), Ixy, xx)), z2));
    const pair_t nd = pk(rcp_normal(n1.x), rcp_normal(n1.y));
    const pair_t ng = pk(rcp_normal(n2.x), rcp_normal(n2.y));
    float2 adv = upk(fmul2(fmul2(dup(delta), nd), psi_prime2(fmul2(fmul2(nd, Iz), Iz))));
    float2 agv = upk(fmul2(fmul2(dup(gamma), ng),
                           psi_prime2(fmul2(ng, ffma2(Iyz, Iyz, fmul2(Ixz, Ixz))))));
    const pair_t u = at(m.U), v = at(m.V);
    const float2 wx = upk(fadd2(pk((float)gx, (float)(gx + D)), u));
    const float2 wy = upk(fadd2(dup((float)gy), v));
    if (wx.x < 0.0f || wx.x > wm1 || wy.x < 0.0f || wy.x > hm1) adv.x = agv.x = 0.0f;
    if (wx.y < 0.0f || wx.y > wm1 || wy.y < 0.0f || wy.y > hm1) adv.y = agv.y = 0.0f;
    const pair_t ad = pk(adv.x, adv.y), ag = pk(agv.x, agv.y);
    const pair_t as = at(m.As);
    const float2 av = upk(as);
    const float2 al = left(m.As, av), ar = right(m.As, av);
    auto mean = [](float p, float q) { return fmul(0.5f, fadd(p, q)); };
    PairSystem ps;
    ps.wl = make_float2(l0 ? mean(av.x, al.x) : 0.0f, l1 ? mean(av.y, al.y) : 0.0f);
    ps.wr = make_float2(r0 ? mean(av.x, ar.x) : 0.0f, r1 ? mean(av.y, ar.y) : 0.0f);
    const pair_t cl = pk(ps.wl.x, ps.wl.y), cr = pk(ps.wr.x, ps.wr.y);
    const pair_t cu = top ? 0 : fmul2(half, fadd2(as, at(m.As - kLvW)));
    const pair_t cd = bottom ? 0 : fmul2(half, fadd2(as, at(m.As + kLvW)));
    ps.wu = upk(cu);
    ps.wd = upk(cd);
    const pair_t sw = fadd2(fadd2(fadd2(cl, cr), cu), cd);
    auto smooth = [&](const float *q, pair_t c) {
        const float2 n = upk(c);
        const float2 ql = left(q, n), qr = right(q, n);
        const pair_t dl = pk(fsub(ql.x, n.x), fsub(ql.y, n.y));
        const pair_t dr = pk(fsub(qr.x, n.x), fsub(qr.y, n.y));
        return ffma2(cd, fsub2(at(q + kLvW), c),
                     ffma2(cu, fsub2(at(q - kLvW), c), ffma2(cr, dr, fmul2(cl, dl))));
    };
    const pair_t su = smooth(m.U, u), sv = smooth(m.V, v);
    const pair_t adx = fmul2(ad, ix), ady = fmul2(ad, iy), nag = neg2(ag);
    ps.d1 = upk(fadd2(ffma2(ag, ffma2(Ixy, Ixy, xx), fmul2(adx, ix)), sw));
    ps.d2 = upk(fadd2(ffma2(ag, ffma2(Iyy, Iyy, yy), fmul2(ady, iy)), sw));
    ps.a12 = upk(ffma2(ag, ffma2(Ixy, Iyy, fmul2(Ixx, Ixy)), fmul2(adx, iy)));
    ps.b1 = upk(ffma2(nag, ffma2(Ixy, Iyz, fmul2(Ixx, Ixz)), ffma2(neg2(adx), Iz, su)));
    ps.b2 = upk(ffma2(nag, ffma2(Iyy, Iyz, fmul2(Ixy, Ixz)), ffma2(neg2(ady), Iz, sv)));
    return ps;
}

// The linear systems of a level as planes: a block stages a tile of 64 columns
// x TH rows and writes its pixels' systems, two a thread and step, 32 columns
// apart: every access of a warp is to 32 columns side by side, from any column
// (adjacent pixels a pair want odd ones, one tile more at widths of 64 k).
// Bound by L1 (77 % of its cycles) and issue (69 %): eight frames of 1280 x 720
// 85 us a launch, 354 MB of planes 50.
template <int TH, int NT, typename T>
__device__ __forceinline__ void var_coeff_body(
    float *smem, const T *__restrict__ I0, const T *__restrict__ I0x, const T *__restrict__ I0y,
    const T *__restrict__ I1, int w, int h, int pitch, const float *__restrict__ U, size_t plane,
    float *__restrict__ cf, float delta, float gamma, float alpha_s, float omega, int bx, int by)
{
    constexpr int WH = TH + 4, WARPS = NT / 32;
    const Windows<WH> m(smem);
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int tx = bx * 64, ty = by * TH;
    const bool inside = tx >= 2 && ty >= 2 && tx + 66 <= w && ty + TH + 2 <= h;
    stage_window<WH, NT, 3>(m, I1, w, h, pitch, tx - 2, ty - 2, inside,
                            [&](auto &c0, auto &c1, auto &cy, auto &u, auto &v) {
                                load_planes<3>(U, plane, pitch, c0, c1, cy, u, v);
                            });
    __syncthreads();
    const int gx = tx + lane, pl = (int)plane;
    const bool c0 = inside || gx < w, c1 = inside || gx + 32 < w;
    // the template's values of a row are loaded while the row before, or the
    // derivatives, are computed; no test between the loads (columns outside:
    // any value, nothing is written there)
    const int xa = min(gx, w - 1), xb = min(gx + 32, w - 1);
    T t0[2], tx0[2], ty0[2];
    auto fetch = [&](int r) {
        const int o = min(ty + r, h - 1) * pitch;
        t0[0] = I0[o + xa], t0[1] = I0[o + xb];
        tx0[0] = I0x[o + xa], tx0[1] = I0x[o + xb];
        ty0[0] = I0y[o + xa], ty0[1] = I0y[o + xb];
    };
    fetch(wp);
    derive_window<WH, NT>(m, alpha_s);
    __syncthreads();
#pragma unroll 1
    for (int r = wp; r < TH; r += WARPS) {
        const int gy = ty + r, o = gy * pitch + gx;
        if (gy >= h) break;
        const pair_t i0 = pk((float)t0[0], (float)t0[1]);
        const pair_t i0x = pk((float)tx0[0], (float)tx0[1]);
        const pair_t i0y = pk((float)ty0[0], (float)ty0[1]);
        if (r + WARPS < TH) fetch(r + WARPS);
        const int e = (r + 2) * kLvW + lane + 2;
        const PairSystem ps = pair_system<32>(m, e, gx, gy, w, h, inside, i0, i0x, i0y, delta, gamma);
        float *c = cf + o;
        auto st = [&](int k, float x, float y) {
            if (c0) c[k * pl] = x;
            if (c1) c[k * pl + 32] = y;
        };
        st(kCI11, __fdividef(omega, ps.d1.x), __fdividef(omega, ps.d1.y));
        st(kCI22, __fdividef(omega, ps.d2.x), __fdividef(omega, ps.d2.y));
        st(kCA12, ps.a12.x, ps.a12.y);
        st(kCB1, ps.b1.x, ps.b1.y);
        st(kCB2, ps.b2.x, ps.b2.y);
        st(kCAS, m.As[e], m.As[e + 32]);
    }
}

// Tiles of 16 rows, 256 threads of 64 registers (four blocks an SM), or of 8
// rows for grids of under two blocks an SM, where the chain of the three phases
// counts.
constexpr int kCoefThreads = 256, kCoefRows = 16, kCoefRowsSmall = 8;

template <int TH, typename T>
__global__ void __launch_bounds__(kCoefThreads, TH == kCoefRows ? 4 : 3)
var_coeff_kernel(const T *__restrict__ I0b, const T *__restrict__ I0xb,
                 const T *__restrict__ I0yb, const T *__restrict__ I1b, int w, int h, int pitch,
                 size_t pfs, const float *__restrict__ Ub, size_t ufs, size_t plane,
                 float *__restrict__ coefb, size_t cfs, float delta, float gamma, float alpha_s,
                 float omega)
{
    chain_begin();
    extern __shared__ __align__(16) float csm[];
    const int f = blockIdx.z;
    const size_t po = (size_t)f * pfs;
    var_coeff_body<TH, kCoefThreads>(csm, I0b + po, I0xb + po, I0yb + po, I1b + po, w, h, pitch,
                                     Ub + (size_t)f * ufs, plane, coefb + (size_t)f * cfs, delta,
                                     gamma, alpha_s, omega, blockIdx.x, blockIdx.y);
}

template <typename T>
__global__ void __launch_bounds__(kCoefThreads, 4)
seg_var_coeff_kernel(const __grid_constant__ SegTable<SegCoeff> tab)
{
    extern __shared__ __align__(16) float csm[];
    int b;
    const SegCoeff &a = seg_of(tab, b);
    const int r = b / a.gx;
    const size_t f = r / a.gy, po = f * a.pfs;
    var_coeff_body<kCoefRows, kCoefThreads>(
        csm, (const T *)a.I0 + po, (const T *)a.I0x + po, (const T *)a.I0y + po,
        (const T *)a.I1 + po, a.w, a.h, a.pitch, a.U + f * a.ufs, a.plane,
        a.coef + kCoefShift + f * a.cfs, a.delta, a.gamma, a.alpha_s, a.omega, b % a.gx, r % a.gy);
}

// The whole variational refinement of a level in one launch.  The work is a
// list of items (iteration, region of 64 x 16 VS), iteration by iteration; a
// block claims them in order from a counter, the next one during the sweeps
// of the last (not before: a block that started early must not take an item
// of one that starts a little later, which would then come an item late):
//  A. It stages the flow of the region and 2 px around, which the region and
//     its eight neighbours wrote in the previous iteration (the halo and the
//     2 px are no wider than an interior), and the warped image there.
//  B. The warped image's derivatives and the smoothness weights, 1 px around.
//  C. Each thread builds the systems of its strip in registers, where the
//     sweeps use them: they never leave the SM.
//  D. The sweeps, then U + dU of the interior.
// The arithmetic is that of the per-iteration kernels, pixel by pixel with the
// same rounding, so the flow is the same bit for bit.
//
// Between iterations the flow travels as packets of a pixel's (u, v) and a
// 64-bit tag, written and read as one 128-bit word: a reader polls the packets
// it needs until they carry the iteration's tag.  No flag and no fence stands
// between a write and its use: a release fence alone took about 2000 of an
// item's 12500 cycles (the acknowledgements of the block's stores), the polls
// of a flag 700 more.  Two buffers take turns: a region overwrites one only
// after its neighbours have written the other, so after they read the first.
// Tags never repeat: a launch's follow on the last one's.
//
// Items are claimed by running blocks and in order, so whatever an item waits
// for is already claimed by a block that runs: the kernel ends with any number
// of blocks resident, beside any other kernel, and needs no cooperative launch
// (which, inside a CUDA graph, cost more than the ten launches it replaced).
//
// It pays where an iteration's two launches are latency: the launches
// themselves, and three round trips through L2 (flow, image, coefficients)
// before the sweeps start.  The halo's systems are built again by every region
// that holds them (1.9 times at 64 x 64, 3.2 at 64 x 32).
//
// ctl: [0] the claim counter, [1] blocks gone, [2..3] the tag that the
// launch's follow.  The last block to leave prepares them for the next launch.
// Polls are bounded; a block whose polls run out reports kErrTimeout and leaves.
// The items that it and the others then leave undone are nobody's: the blocks
// that wait for them leave the same way, and the next launch's tags are new.
//
// Measured, two windows of all levels: 346 x 260 425 us with launches, 324 with
// flags, 298 with packets; a window of 641 x 479 and its surface 741 us with
// its finest level in launches, 647 here.
//
// The packets of odd and of even columns lie apart: regions start at odd ones,
// so a warp's accesses, a pair of pixels a lane, are contiguous.
__host__ __device__ __forceinline__ int packet_pitch(int w) { return (w + 1) >> 1; }
__device__ __forceinline__ int packet_at(int x, int y, int w2, int h)
{
    return ((x & 1 ? 0 : h) + y) * w2 + (x >> 1);
}
__device__ __forceinline__ void store_packet(float4 *q, float u, float v, unsigned long long tag)
{
    asm volatile("{ .reg .b64 uv; .reg .b128 p;\n\t"
                 "mov.b64 uv, {%1, %2};\n\t"
                 "mov.b128 p, {uv, %3};\n\t"
                 "st.relaxed.gpu.global.b128 [%0], p; }" ::"l"(q),
                 "f"(u), "f"(v), "l"(tag)
                 : "memory");
}
__device__ __forceinline__ bool load_packet(const float4 *q, unsigned long long tag, float &u,
                                            float &v)
{
    unsigned long long got;
    asm volatile("{ .reg .b64 uv; .reg .b128 p;\n\t"
                 "ld.relaxed.gpu.global.b128 p, [%3];\n\t"
                 "mov.b128 {uv, %2}, p;\n\t"
                 "mov.b64 {%0, %1}, uv; }"
                 : "=f"(u), "=f"(v), "=l"(got)
                 : "l"(q)
                 : "memory");
    return got == tag;
}

template <int VS>
constexpr size_t level_smem_bytes()
{
    return Windows<VS * kVWarps + 4>::kBytes;
}

template <int VS, typename T>
__global__ void __launch_bounds__(kVThreads, 1)
var_level_kernel(const T *__restrict__ I0b, const T *__restrict__ I0xb,
                 const T *__restrict__ I0yb, const T *__restrict__ I1b, int w, int h, int pitch,
                 size_t pfs, float *Ua, float *Ub, size_t ufs, size_t plane, int outer, int n_half,
                 int R, int nrx, int nry, float delta, float gamma, float alpha_s, float omega,
                 int blocks, uint3 mg, unsigned *ctl, float4 *xch, size_t xch_n, long long wait_limit,
                 int *err)
{
    chain_begin();
    constexpr int RH = VS * kVWarps, WH = RH + 4;
    // pairs a thread stages: all of them at once, one wait for the packets
    constexpr int KI = (kLvW / 2 * WH + kVThreads - 1) / kVThreads;
    extern __shared__ __align__(16) float lsm[];
    const Windows<WH> m(lsm);
    __shared__ StripEnds<kVWarps> ends;
    const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
    __shared__ int s_item;
    const int per_frame = nrx * nry, total = outer * blocks;
    const int w2 = packet_pitch(w), pk_fs = 2 * w2 * h;
    clear_ends(ends);
    // written by a launch's last block only
    unsigned long long *ctl_tag = reinterpret_cast<unsigned long long *>(ctl + 2);
    const unsigned long long base = *ctl_tag;
    if (t == 0) s_item = (int)atomicAdd(ctl, 1u);
    __syncthreads();
    for (int item = s_item; item < total; item = s_item) {
        const int k = div_stride(item, mg.x), reg = item - k * blocks;
        const int f = div_stride(reg, mg.y), rem = reg - f * per_frame;
        const int by = div_stride(rem, mg.z), bx = rem - by * nrx;
        const StripPlace<VS, kVWarps> p(bx, by, R, w, h, pitch, lane, wp);
        const int rx0 = p.gx - 2 * lane, ry0 = p.gy - wp * VS;
        const size_t po = (size_t)f * pfs;
        const T *I0 = I0b + po, *I0x = I0xb + po, *I0y = I0yb + po, *I1 = I1b + po;
        // the staged window lies in the level (block-uniform)
        const bool inside = rx0 >= 2 && ry0 >= 2 && rx0 + kVR + 2 <= w && ry0 + RH + 2 <= h;
        bool late = false;
        stage_window<WH, kVThreads, KI>(
            m, I1, w, h, pitch, rx0 - 2, ry0 - 2, inside,
            [&](auto &c0, auto &c1, auto &cy, auto &u, auto &v) {
                if (k == 0) {
                    load_planes<KI>(Ua + (size_t)f * ufs, plane, pitch, c0, c1, cy, u, v);
                    return;
                }
                const float4 *src = xch + ((k - 1) & 1) * xch_n + (size_t)f * pk_fs;
                const unsigned long long tag = base + k;
                float x0[KI], x1[KI], y0[KI], y1[KI];
                for (long long it = 0;; ++it) {
                    bool ok = true;
#pragma unroll
                    for (int j = 0; j < KI; ++j) {
                        ok &= load_packet(src + packet_at(c0[j], cy[j], w2, h), tag, x0[j], y0[j]);
                        ok &= load_packet(src + packet_at(c1[j], cy[j], w2, h), tag, x1[j], y1[j]);
                    }
                    if (it >= wait_limit) {  // a limit of 0: whatever came
                        late = true;
                        break;
                    }
                    if (ok) break;
                }
#pragma unroll
                for (int j = 0; j < KI; ++j) {
                    u[j] = pk(x0[j], x1[j]);
                    v[j] = pk(y0[j], y1[j]);
                }
            });
        if (__syncthreads_or(late)) {
            if (t == 0) atomicOr(err, kErrTimeout);
            break;
        }
        // the strip's template values, in flight during B; no test between the
        // loads, so that none waits for another (pixels outside the level: any
        // value, their systems are 0)
        pair_t i0[VS], i0x[VS], i0y[VS];
        const int xa = clampi(p.gx, 0, w - 1), xb = clampi(p.gx + 1, 0, w - 1);
#pragma unroll
        for (int r = 0; r < VS; ++r) {
            const int o = clampi(p.gy + r, 0, h - 1) * pitch;
            i0[r] = pk(ldp(I0 + o + xa), ldp(I0 + o + xb));
            i0x[r] = pk(ldp(I0x + o + xa), ldp(I0x + o + xb));
            i0y[r] = pk(ldp(I0y + o + xa), ldp(I0y + o + xb));
        }
        derive_window<WH, kVThreads>(m, alpha_s);
        __syncthreads();
        Strip<VS> s;
#pragma unroll
        for (int r = 0; r < VS; ++r) {
            const int e = (wp * VS + r + 2) * kLvW + 2 * lane + 2;
            const int gx = p.gx, gy = p.gy + r;
            const bool row_in = inside || (gy >= 0 && gy < h);
            const bool in0 = row_in && (inside || (gx >= 0 && gx < w));
            const bool in1 = row_in && (inside || (gx + 1 >= 0 && gx + 1 < w));
            const PairSystem ps =
                pair_system<1>(m, e, gx, gy, w, h, inside, i0[r], i0x[r], i0y[r], delta, gamma);
            s.i11[r][0] = in0 ? __fdividef(omega, ps.d1.x) : 0.0f;
            s.i11[r][1] = in1 ? __fdividef(omega, ps.d1.y) : 0.0f;
            s.i22[r][0] = in0 ? __fdividef(omega, ps.d2.x) : 0.0f;
            s.i22[r][1] = in1 ? __fdividef(omega, ps.d2.y) : 0.0f;
            s.a12[r][0] = in0 ? ps.a12.x : 0.0f;
            s.a12[r][1] = in1 ? ps.a12.y : 0.0f;
            s.b[r][0] = in0 ? pk(ps.b1.x, ps.b2.x) : 0;
            s.b[r][1] = in1 ? pk(ps.b1.y, ps.b2.y) : 0;
            // the region's own edges carry no weight, nor do pixels outside
            const bool up_in = !(r == 0 && wp == 0);
            s.wl[r][0] = lane > 0 && in0 ? ps.wl.x : 0.0f;
            s.wl[r][1] = in1 ? ps.wl.y : 0.0f;
            s.wr[r] = lane < 31 && in1 ? ps.wr.y : 0.0f;
            s.wu[r][0] = up_in && in0 ? ps.wu.x : 0.0f;
            s.wu[r][1] = up_in && in1 ? ps.wu.y : 0.0f;
            if (r == VS - 1) {
                s.wd[0] = wp < kVWarps - 1 && in0 ? ps.wd.x : 0.0f;
                s.wd[1] = wp < kVWarps - 1 && in1 ? ps.wd.y : 0.0f;
            }
        }
        // D
        const unsigned next = t == 0 ? atomicAdd(ctl, 1u) : 0u;
        sor_sweeps<VS, kVWarps>(s, ends, lane, wp, (p.gx + p.gy) & 1, n_half, omega);
#pragma unroll
        for (int r = 0; r < VS; ++r) {
            if (r < p.r0 || r >= p.r1) continue;
            const int e = (wp * VS + r + 2) * kLvW + 2 * lane + 2;
            const float2 u = upk(ld_pair(m.U + e)), v = upk(ld_pair(m.V + e));
            const float2 d0 = upk(s.d[r][0]), d1 = upk(s.d[r][1]);
            const float2 nu = make_float2(u.x + d0.x, u.y + d1.x);
            const float2 nv = make_float2(v.x + d0.y, v.y + d1.y);
            if (k + 1 < outer) {
                const unsigned long long tag = base + k + 1;
                float4 *q = xch + (k & 1) * xch_n + (size_t)f * pk_fs;
                if (p.c0) store_packet(q + packet_at(p.gx, p.gy + r, w2, h), nu.x, nv.x, tag);
                if (p.c1) store_packet(q + packet_at(p.gx + 1, p.gy + r, w2, h), nu.y, nv.y, tag);
                continue;
            }
            float *q = ((outer & 1) ? Ub : Ua) + (size_t)f * ufs + (p.gy + r) * pitch + p.gx;
            if (p.c0 && p.c1) {
                *reinterpret_cast<float2 *>(q) = nu;
                *reinterpret_cast<float2 *>(q + plane) = nv;
            } else if (p.c0) {
                q[0] = nu.x;
                q[plane] = nv.x;
            } else if (p.c1) {
                q[1] = nu.y;
                q[plane + 1] = nv.y;
            }
        }
        if (t == 0) s_item = (int)next;
        __syncthreads();  // the block's reads of the stage
    }
    // the last block to leave prepares the counters of the next launch
    if (t == 0) {
        __threadfence();
        if (atomicInc(ctl + 1, gridDim.x - 1) == gridDim.x - 1) {
            ctl[0] = 0;
            *ctl_tag = base + outer;
        }
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
        cudaGetLastError();
    });
    return fn;
}

}  // namespace

void make_coef_maps(float *work, const float *Ua, const float *Ub, size_t u_frame_stride,
                    const Geometry &geo, int var_sor, int frames, CoefMaps *m)
{
    for (int l = 0; l < kMaxLevels; ++l) m->ok[l] = false;
    EncodeTiledFn enc = encode_tiled();
    const int tile = sor_tile(sor_halo(var_sor));
    if (!enc || !work || !Ua || !Ub || tile < 1) return;
    auto encode = [&](CUtensorMap *map, const float *base, const Level &lv, int planes,
                      size_t frame_stride, int bw, int bh) {
        const cuuint64_t dims[4] = {(cuuint64_t)lv.w + kCoefShift, (cuuint64_t)lv.h,
                                    (cuuint64_t)planes, (cuuint64_t)frames};
        const cuuint64_t strides[3] = {(cuuint64_t)lv.pitch * sizeof(float),
                                       (cuuint64_t)lv.plane * sizeof(float),
                                       (cuuint64_t)frame_stride * sizeof(float)};
        const cuuint32_t box[4] = {(cuuint32_t)bw, (cuuint32_t)bh, (cuuint32_t)planes, 1};
        const cuuint32_t estr[4] = {1, 1, 1, 1};
        return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void *)base, dims, strides, box,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    for (int l = 0; l < geo.levels; ++l) {
        const Level &lv = geo.lv[l];
        SorMaps &x = m->map[l];
        bool ok = encode(&x.coef, work, lv, kCPlanes, kCPlanes * lv.plane, kTmaBoxW, kVR);
        for (int k = 0; k < 2; ++k) {
            x.ubase[k] = k ? Ub : Ua;
            ok = ok && encode(&x.u[k], x.ubase[k] - kCoefShift, lv, 2, u_frame_stride,
                              u_box_width(tile), tile);
        }
        m->ok[l] = ok;
    }
}

bool var_fused_supported(int var_sor)
{
    return kVR - 2 * sor_halo(var_sor) >= 16;
}

void init_var_attributes()
{
    cudaFuncSetAttribute(var_sor_tma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)kTmaSmemBytes);
    cudaFuncSetAttribute(var_sor_kernel<kVS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)flow_stage_bytes<kVS, kVWarps>());
    cudaFuncSetAttribute(seg_var_sor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)flow_stage_bytes<kVS, kVWarps>());
    auto level_smem = [](const void *fn, size_t bytes) {
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    level_smem((const void *)var_level_kernel<kVS, float>, level_smem_bytes<kVS>());
    level_smem((const void *)var_level_kernel<kVS, __half>, level_smem_bytes<kVS>());
    level_smem((const void *)var_level_kernel<kVSmallVS, float>, level_smem_bytes<kVSmallVS>());
    level_smem((const void *)var_level_kernel<kVSmallVS, __half>, level_smem_bytes<kVSmallVS>());
    cudaGetLastError();
}

// The packets of a frame of a level.
static size_t frame_packets(const Level &lv) { return 2 * (size_t)packet_pitch(lv.w) * lv.h; }

size_t level_packets(const Geometry &geo, int var_sor, int cluster_max, int frames)
{
    const int R = sor_halo(var_sor), tile = sor_tile(R);
    size_t most = 0;
    if (tile < R + 2) return 0;
    for (int l = 0; l < geo.levels; ++l) {
        const Level &lv = geo.lv[l];
        const int per = ((lv.w + tile - 1) / tile) * ((lv.h + tile - 1) / tile);
        const int f = cluster_max > 0 ? std::min(frames, kLevelBlocks / std::max(per, 1)) : 1;
        if (per <= kLevelBlocks) most = std::max(most, frame_packets(lv) * std::max(f, 1));
    }
    return most;
}

int sor_halo(int var_sor) { return var_sor > 0 ? 2 * var_sor - 1 : 1; }
int sor_tile(int R) { return kVR - 2 * R; }
int coeff_tiles_x(int w) { return (w + 63) / 64; }
int coeff_tiles_y(int h) { return (h + kCoefRows - 1) / kCoefRows; }
int coeff_planes() { return kCPlanes; }

void launch_seg_coeff(const SegTable<SegCoeff> &t, int blocks, bool half, cudaStream_t st)
{
    StageScope sc(kStVarCoeff, 1, st);
    constexpr size_t smem = Windows<kCoefRows + 4>::kBytes;
    if (half) seg_var_coeff_kernel<__half><<<blocks, kCoefThreads, smem, st>>>(t);
    else seg_var_coeff_kernel<float><<<blocks, kCoefThreads, smem, st>>>(t);
}

void launch_seg_sor(const SegTable<SegSor> &t, int blocks, cudaStream_t st)
{
    StageScope sc(kStVarSor, 1, st);
    seg_var_sor_kernel<<<blocks, kVThreads, flow_stage_bytes<kVS, kVWarps>(), st>>>(t);
}

float *launch_variational_fused(const void *I0, const void *I0x, const void *I0y,
                                const void *I1, const Level &lv, size_t pyr_frame_stride,
                                float *U, float *Utmp, size_t u_frame_stride, float *coef,
                                int frames, const FlowParams &fp, const SorMaps *maps,
                                int *err, cudaStream_t st)
{
    // the level's planes are packed: frame stride kCPlanes planes of this level
    const size_t coef_frame_stride = (size_t)kCPlanes * lv.plane;
    const int nsm = sm_count();
    const int n_half = 2 * fp.var_sor;
    const int R = sor_halo(fp.var_sor);
    const int tile = sor_tile(R);           // interior side of a 64 x 64 region
    const int small = kVSmallRows - 2 * R;  // interior rows of a 64 x 32 region
    coef += kCoefShift;
    dim3 cgrd(coeff_tiles_x(lv.w), coeff_tiles_y(lv.h), frames);
    const bool small_tiles = (long long)(cgrd.x * cgrd.y * cgrd.z) < 2LL * nsm;
    if (small_tiles) cgrd.y = (lv.h + kCoefRowsSmall - 1) / kCoefRowsSmall;
    const dim3 sgrd((lv.w + tile - 1) / tile, (lv.h + tile - 1) / tile, frames);
    // small levels of a single frame: every outer iteration in one launch (same
    // flow bit for bit), where a region's staged window reaches no further than
    // its neighbours' interiors: 64 x 32 regions if one wave holds them (more
    // was slower at every size: 640 x 360, 364 of them, 582 us a window against
    // 548 with 112 of 64 x 64), else 64 x 64 up to 1.75 waves.  There the items
    // of all iterations fill the waves that a launch an iteration leaves open;
    // one window (all levels) with the finest level here against per-iteration
    // launches: 640 x 480, 154 regions, 605 against 640 us; 800 x 600, 252, 733
    // against 739; 880 x 640, 280, 775 against 767; 1280 x 720, 448, 960 against
    // 935.  Several frames fill the SMs either way (640 x 480, eight frames:
    // 1.01 ms a call with and without), so only where asked for
    for (int vs : {kVSmallVS, kVS}) {
        const int ty = vs * kVWarps - 2 * R, nrx = (int)sgrd.x;
        const int nry = ty > 0 ? (lv.h + ty - 1) / ty : 0;
        const long long per = (long long)nrx * nry, blocks = per * frames;
        const long long most = std::min(vs == kVS ? 7 * nsm / 4 : nsm, kLevelBlocks);
        if (!fp.level_ctl || fp.var_outer < 1 || ty < R + 2 || tile < R + 2 || lv.w < 2 ||
            lv.h < 2 || nsm < 1 || blocks > most || frame_packets(lv) * frames > fp.level_n ||
            (frames > 1 && per > fp.var_cluster_max))
            continue;
        const bool small_form = vs == kVSmallVS;
        const int lgrid = (int)std::min<long long>(blocks, nsm);
        // items < 1000 x 266, so the products stay below 2^31
        const uint3 mg = make_uint3(stride_magic((int)blocks), stride_magic((int)per),
                                    stride_magic(nrx));
        cudaError_t e;
        {
            StageScope sc(kStVarSor, 1, st);
#define EBOF_LV(VS, T)                                                                          \
    launch_chained(true, var_level_kernel<VS, T>, lgrid, kVThreads, level_smem_bytes<VS>(), st, \
                   (const T *)I0, (const T *)I0x,                                               \
                       (const T *)I0y, (const T *)I1, lv.w, lv.h, lv.pitch, pyr_frame_stride,   \
                       U, Utmp, u_frame_stride, lv.plane, fp.var_outer, n_half, R, nrx, nry,    \
                       fp.delta, fp.gamma, fp.alpha_s, fp.omega, (int)blocks, mg, fp.level_ctl,     \
                       (float4 *)fp.level_xch, fp.level_n, fp.wait_limit, err)
            if (fp.half)
                e = small_form ? EBOF_LV(kVSmallVS, __half) : EBOF_LV(kVS, __half);
            else
                e = small_form ? EBOF_LV(kVSmallVS, float) : EBOF_LV(kVS, float);
#undef EBOF_LV
        }
        if (e == cudaSuccess) return (fp.var_outer & 1) ? Utmp : U;
        cudaGetLastError();  // not launched: the per-iteration kernels below
    }
    float *a = U, *b = Utmp;
    for (int k = 0; k < fp.var_outer; ++k) {
        {
            StageScope sc(kStVarCoeff, 1, st);
#define EBOF_CF(TH, T)                                                                          \
    launch_chained(true, var_coeff_kernel<TH, T>, cgrd, kCoefThreads,                            \
                   Windows<TH + 4>::kBytes, st, (const T *)I0, (const T *)I0x, (const T *)I0y,   \
                   (const T *)I1, lv.w, lv.h, lv.pitch, pyr_frame_stride, a, u_frame_stride,     \
                   lv.plane, coef, coef_frame_stride, fp.delta, fp.gamma, fp.alpha_s, fp.omega)
            if (fp.half) {
                if (small_tiles) EBOF_CF(kCoefRowsSmall, __half);
                else EBOF_CF(kCoefRows, __half);
            } else {
                if (small_tiles) EBOF_CF(kCoefRowsSmall, float);
                else EBOF_CF(kCoefRows, float);
            }
#undef EBOF_CF
        }
        {
            StageScope sc(kStVarSor, 1, st);
            const int total = (int)(sgrd.x * sgrd.y * sgrd.z);
            const int row_waves = fp.sor_row_waves;
            const dim3 g1(sgrd.x, small > 0 ? (lv.h + small - 1) / small : 1, frames);
            const int ub = !maps ? -1 : a == maps->ubase[0] ? 0 : a == maps->ubase[1] ? 1 : -1;
            if (ub >= 0 && nsm > 0 && (long long)total >= (long long)fp.sor_tma_min_per_sm * nsm)
                launch_chained(true, var_sor_tma_kernel, std::min(nsm, total), kVThreads,
                               kTmaSmemBytes, st, maps->coef, maps->u[ub], lv.w, lv.h, lv.pitch, b,
                               u_frame_stride, lv.plane, R, (int)sgrd.x, (int)sgrd.y, total,
                               n_half, fp.omega, fp.wait_limit, fp.flow_wait_limit, err);
            else if (small >= 8 && (long long)(g1.x * g1.y * g1.z) <= (long long)row_waves * nsm)
                launch_chained(true, var_sor_kernel<kVSmallVS>, g1, kVThreads,
                               flow_stage_bytes<kVSmallVS, kVWarps>(), st, lv.w, lv.h, lv.pitch,
                               a, b, u_frame_stride, lv.plane, coef, coef_frame_stride, R, n_half,
                               fp.omega);
            else
                launch_chained(true, var_sor_kernel<kVS>, sgrd, kVThreads,
                               flow_stage_bytes<kVS, kVWarps>(), st, lv.w, lv.h, lv.pitch, a, b,
                               u_frame_stride, lv.plane, coef, coef_frame_stride, R, n_half,
                               fp.omega);
        }
        float *t = a;
        a = b;
        b = t;
    }
    return a;
}

}  // namespace ebof
