// k_var.cu -- variational refinement (reading F6): two kernels per
// fixed-point iteration.
//
// var_coeff_kernel, one thread per pixel: stages U and the warped image
// I1(x + U) for a 32x12 tile plus 2 px in shared memory, builds derivatives
// of the warped image and the smoothness weights, and writes every pixel's
// 2x2 linear system (data and gradient-constancy terms normalised, weights
// lagged at dU = 0): omega/a11, omega/a22 (the SOR relaxation factor folded
// into the inverted diagonal), a12, b1, b2 and the smoothness weight, as six
// planes.  Only the staging halo is shared between tiles.  On levels from
// 1024 px wide the same systems come from var_coeff_cw_kernel, a column walk
// with the rows in registers.
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
// sweeps.  Measured per 1280x720 launch on a GB300, inside a graph, against
// the scalar form of 7 planes and a full exchange: 18.3 -> 15.6 us for one
// frame, 165 -> 126 us for eight.
//
// var_sor_tma_kernel: the same regions in a persistent grid (one block per
// SM).  One thread loads each region's planes into shared memory with a
// single TMA tensor copy (cp.async.bulk.tensor, completion on an mbarrier);
// once every thread has moved its values into registers, the copy of the
// block's next region is issued and runs during the sweeps.  The box starts at
// the region's first column rounded down to the 16-byte rule of tensor copies
// and is 4 columns wider; elements outside the level are filled with zero, as
// the direct loads do, so both kernels give the same result.  It needs at
// least two regions an SM to hide a copy: measured against the direct form (in
// a graph, 7 planes) 6.8 vs 6.1 us for 112 regions, 10.4 vs 9.8 for 154, 14.7
// vs 15.6 for 448, 27.0 vs 30.4 for 896, 101 vs 126 for 3584.
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
constexpr size_t kTmaSmemBytes =
    kTmaCoefFloats * sizeof(float) + flow_stage_bytes<kVS, kVWarps>();
constexpr int kMaxDevs = 64;
int g_num_sms[kMaxDevs];
// coefficient tile: 384 threads at 40 registers, four blocks per SM, so a
// 640 x 360 level (600 tiles) takes one wave where 32 x 16 tiles took two
constexpr int kAX = 32, kAY = 12;
constexpr int kAEX = kAX + 4, kAEY = kAY + 4;  // staging window: tile + 2 px
constexpr int kADX = kAX + 2, kADY = kAY + 2;  // derivative window: tile + 1 px
constexpr unsigned kFull = 0xffffffffu;

// Loads of data that the same launch may have written on another SM earlier
// (COH: through L2 with ld.global.cg, never from a possibly stale L1 or the
// read-only path); plain loads otherwise.  The values are the same.
template <bool COH>
__device__ __forceinline__ float ldf(const float *p)
{
    if constexpr (COH)
        return __ldcg(p);
    else
        return *p;
}
template <bool COH>
__device__ __forceinline__ float2 ldf2(const float *p)
{
    if constexpr (COH)
        return __ldcg(reinterpret_cast<const float2 *>(p));
    else
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

// Smoothness weight alpha_s Psi'(|grad u|^2 + |grad v|^2) with forward
// differences (ur, ud: U to the right and below; hx, hy: those neighbours are
// in the level, else the difference is 0).
__device__ __forceinline__ float smooth_weight(float u, float ur, float ud, float v, float vr,
                                               float vd, bool hx, bool hy, float alpha_s)
{
    const float ux = hx ? fsub(ur, u) : 0.0f;
    const float uy = hy ? fsub(ud, u) : 0.0f;
    const float vx = hx ? fsub(vr, v) : 0.0f;
    const float vy = hy ? fsub(vd, v) : 0.0f;
    return fmul(alpha_s, psi_prime(ffma(vy, vy, ffma(vx, vx, ffma(uy, uy, fmul(ux, ux))))));
}

__device__ __forceinline__ float cdiff(float hi, float lo) { return fmul(0.5f, fsub(hi, lo)); }

// Derivatives of the warped image and the smoothness weight at a pixel of a
// staging window (row stride ES; (e) the pixel, at image position gx, gy).
// IN: the pixel and its neighbours lie inside the level, so the clamps and
// border tests are known to pass and are left out (same values).
template <bool IN>
__device__ __forceinline__ void stage_derivs(const float *sW, const float *sU, const float *sV,
                                             int ES, int e, int ex0, int ey0, int gx, int gy,
                                             int w, int h, float alpha_s, float &ix, float &iy,
                                             float &as)
{
    const int xp = (IN ? gx + 1 : min(gx + 1, w - 1)) - ex0;
    const int xm = (IN ? gx - 1 : max(gx - 1, 0)) - ex0;
    const int yp = (IN ? gy + 1 : min(gy + 1, h - 1)) - ey0;
    const int ym = (IN ? gy - 1 : max(gy - 1, 0)) - ey0;
    const int ex = gx - ex0, ey = gy - ey0;
    ix = cdiff(sW[ey * ES + xp], sW[ey * ES + xm]);
    iy = cdiff(sW[yp * ES + ex], sW[ym * ES + ex]);
    as = smooth_weight(sU[e], sU[e + 1], sU[e + ES], sV[e], sV[e + 1], sV[e + ES],
                       IN || gx + 1 < w, IN || gy + 1 < h, alpha_s);
}

struct PixelSystem {
    float i11, i22, a12, b1, b2;
};

// The 2x2 system of pixel (gx, gy) from its neighbourhood.  ix, iy: the
// warped image's derivatives at the pixel; ixl, ixr: Ix at the clamped left
// and right neighbours, ixu, ixd and iyu, iyd: Ix and Iy at the clamped upper
// and lower ones; iw: the warped sample; as*: smoothness weights at the pixel
// and its four neighbours, used only where that neighbour is in the level
// (bl, br, bu, bd); u*, v*: the flow at the pixel and its four neighbours (0
// outside the level); i0, i0x, i0y: the template image and its gradient.
// The diagonal is stored inverted and scaled by the SOR relaxation factor:
// i11 = omega / a11, i22 = omega / a22.
__device__ __forceinline__ PixelSystem pixel_system_vals(
    float ix, float iy, float ixl, float ixr, float ixu, float ixd, float iyu, float iyd,
    float iw, float asp, float asl, float asr, float asu, float asd, float u, float ul, float ur,
    float uu, float ud, float v, float vl, float vr, float vu, float vd, bool bl, bool br,
    bool bu, bool bd, int gx, int gy, int w, int h, float i0, float i0x, float i0y, float delta,
    float gamma, float omega)
{
    // every operation with a fixed rounding (fmul, fadd, fsub, ffma), so that
    // the two kernel forms that call this function give the same systems
    const float Ix = ix, Iy = iy;
    const float Ixx = cdiff(ixr, ixl);
    const float Ixy = cdiff(ixd, ixu);
    const float Iyy = cdiff(iyd, iyu);
    const float Iz = fsub(iw, i0);
    const float Ixz = fsub(Ix, i0x), Iyz = fsub(Iy, i0y);
    const float nd = __fdividef(1.0f, fadd(ffma(Iy, Iy, fmul(Ix, Ix)), kZeta2));
    const float ng = __fdividef(
        1.0f, fadd(ffma(Iyy, Iyy, ffma(fmul(2.0f, Ixy), Ixy, fmul(Ixx, Ixx))), kZeta2));
    float ad = fmul(fmul(delta, nd), psi_prime(fmul(fmul(nd, Iz), Iz)));
    float ag = fmul(fmul(gamma, ng), psi_prime(fmul(ng, ffma(Iyz, Iyz, fmul(Ixz, Ixz)))));
    const float wx = fadd((float)gx, u), wy = fadd((float)gy, v);
    if (wx < 0.0f || wx > (float)(w - 1) || wy < 0.0f || wy > (float)(h - 1)) {
        ad = 0.0f;
        ag = 0.0f;
    }
    PixelSystem ps;
    const float cl = bl ? fmul(0.5f, fadd(asp, asl)) : 0.0f;
    const float cr = br ? fmul(0.5f, fadd(asp, asr)) : 0.0f;
    const float cu = bu ? fmul(0.5f, fadd(asp, asu)) : 0.0f;
    const float cd = bd ? fmul(0.5f, fadd(asp, asd)) : 0.0f;
    const float sw = fadd(fadd(fadd(cl, cr), cu), cd);
    const float su0 = ffma(cd, fsub(ud, u),
                           ffma(cu, fsub(uu, u), ffma(cr, fsub(ur, u),
                                                         fmul(cl, fsub(ul, u)))));
    const float sv0 = ffma(cd, fsub(vd, v),
                           ffma(cu, fsub(vu, v), ffma(cr, fsub(vr, v),
                                                         fmul(cl, fsub(vl, v)))));
    const float adx = fmul(ad, Ix), ady = fmul(ad, Iy);
    ps.i11 = __fdividef(omega, fadd(ffma(ag, ffma(Ixy, Ixy, fmul(Ixx, Ixx)), fmul(adx, Ix)), sw));
    ps.i22 = __fdividef(omega, fadd(ffma(ag, ffma(Iyy, Iyy, fmul(Ixy, Ixy)), fmul(ady, Iy)), sw));
    ps.a12 = ffma(ag, ffma(Ixy, Iyy, fmul(Ixx, Ixy)), fmul(adx, Iy));
    ps.b1 = ffma(-ag, ffma(Ixy, Iyz, fmul(Ixx, Ixz)), ffma(-adx, Iz, su0));
    ps.b2 = ffma(-ag, ffma(Iyy, Iyz, fmul(Ixy, Ixz)), ffma(-ady, Iz, sv0));
    return ps;
}

// The same system read from the staging and derivative windows: d indexes
// the derivative window (row stride DS, origin dx0, dy0), e the staging
// window (row stride ES).  Every index read lies in the windows (their rings
// hold 0 outside the level).  IN as in stage_derivs.
template <bool IN>
__device__ __forceinline__ PixelSystem pixel_system(const float *sIx, const float *sIy,
                                                    const float *sAs, int DS, int dx0, int dy0,
                                                    const float *sW, const float *sU,
                                                    const float *sV, int ES, int e, int gx,
                                                    int gy, int w, int h, float i0, float i0x,
                                                    float i0y, float delta, float gamma,
                                                    float omega)
{
    const int xp = (IN ? gx + 1 : min(gx + 1, w - 1)) - dx0;
    const int xm = (IN ? gx - 1 : max(gx - 1, 0)) - dx0;
    const int yp = (IN ? gy + 1 : min(gy + 1, h - 1)) - dy0;
    const int ym = (IN ? gy - 1 : max(gy - 1, 0)) - dy0;
    const int dx = gx - dx0, dy = gy - dy0;
    const int d = dy * DS + dx;
    return pixel_system_vals(
        sIx[d], sIy[d], sIx[dy * DS + xm], sIx[dy * DS + xp], sIx[ym * DS + dx],
        sIx[yp * DS + dx], sIy[ym * DS + dx], sIy[yp * DS + dx], sW[e], sAs[d], sAs[d - 1],
        sAs[d + 1], sAs[d - DS], sAs[d + DS], sU[e], sU[e - 1], sU[e + 1], sU[e - ES],
        sU[e + ES], sV[e], sV[e - 1], sV[e + 1], sV[e - ES], sV[e + ES], IN || gx > 0,
        IN || gx + 1 < w, IN || gy > 0, IN || gy + 1 < h, gx, gy, w, h, i0, i0x, i0y, delta,
        gamma, omega);
}

// One coefficient tile.  IN: the tile's staging window (tile + 2 px) lies
// inside the level, so no load or neighbour needs a bounds test.
template <bool IN, typename T>
__device__ __forceinline__ void coeff_tile(
    float (&sU)[kAEY][kAEX], float (&sV)[kAEY][kAEX], float (&sW)[kAEY][kAEX],
    float (&sIx)[kADY][kADX], float (&sIy)[kADY][kADX], float (&sAs)[kADY][kADX],
    const T *__restrict__ I0b, const T *__restrict__ I0xb, const T *__restrict__ I0yb,
    const T *__restrict__ I1b, int w, int h, int pitch, size_t pfs, const float *__restrict__ Ub,
    size_t ufs, size_t plane, float *__restrict__ coefb, size_t cfs, float delta, float gamma,
    float alpha_s, float omega, unsigned bx, unsigned by, unsigned f)
{
    const int tx0 = bx * kAX, ty0 = by * kAY;
    const int ex0 = tx0 - 2, ey0 = ty0 - 2, dx0 = tx0 - 1, dy0 = ty0 - 1;
    // frame base pointers once; offsets within a frame fit in 32 bits
    const size_t po = (size_t)f * pfs;
    const T *I1 = I1b + po;
    const float *U = Ub + (size_t)f * ufs;
    const float *V = U + plane;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 12 threads, one per tile pixel

    const int t = ty * kAX + tx;
    constexpr int kN = kAX * kAY;
    for (int i = t; i < kAEX * kAEY; i += kN) {
        const int lx = i % kAEX, ly = i / kAEX;
        const int gx = ex0 + lx, gy = ey0 + ly;
        float u = 0.0f, v = 0.0f, wv = 0.0f;
        if (IN || (gx >= 0 && gx < w && gy >= 0 && gy < h)) {
            const int p = gy * pitch + gx;
            u = U[p];
            v = V[p];
            wv = bilinear_i(I1, w, h, pitch, (float)gx + u, (float)gy + v);
        }
        sU[ly][lx] = u;
        sV[ly][lx] = v;
        sW[ly][lx] = wv;
    }
    __syncthreads();
    for (int i = t; i < kADX * kADY; i += kN) {
        const int lx = i % kADX, ly = i / kADX;
        const int gx = dx0 + lx, gy = dy0 + ly;
        float ix = 0.0f, iy = 0.0f, as = 0.0f;
        if (IN || (gx >= 0 && gx < w && gy >= 0 && gy < h))
            stage_derivs<IN>(&sW[0][0], &sU[0][0], &sV[0][0], kAEX,
                             (gy - ey0) * kAEX + (gx - ex0), ex0, ey0, gx, gy, w, h, alpha_s,
                             ix, iy, as);
        sIx[ly][lx] = ix;
        sIy[ly][lx] = iy;
        sAs[ly][lx] = as;
    }
    __syncthreads();

    const int gx = tx0 + threadIdx.x, gy = ty0 + threadIdx.y;
    if (!IN && (gx >= w || gy >= h)) return;
    const int p = gy * pitch + gx;
    const PixelSystem ps = pixel_system<IN>(
        &sIx[0][0], &sIy[0][0], &sAs[0][0], kADX, dx0, dy0, &sW[0][0], &sU[0][0], &sV[0][0], kAEX,
        (gy - ey0) * kAEX + (gx - ex0), gx, gy, w, h, ldp(&(I0b + po)[p]), ldp(&(I0xb + po)[p]),
        ldp(&(I0yb + po)[p]), delta, gamma, omega);
    const int pl = (int)plane;
    float *cf = coefb + (size_t)f * cfs + p;
    cf[kCI11 * pl] = ps.i11;
    cf[kCI22 * pl] = ps.i22;
    cf[kCA12 * pl] = ps.a12;
    cf[kCB1 * pl] = ps.b1;
    cf[kCB2 * pl] = ps.b2;
    cf[kCAS * pl] = sAs[ty + 1][tx + 1];
}

// (bx, by): the tile, f: the frame.
template <typename T>
__device__ __forceinline__ void var_coeff_body(
    const T *__restrict__ I0b, const T *__restrict__ I0xb, const T *__restrict__ I0yb,
    const T *__restrict__ I1b, int w, int h, int pitch, size_t pfs, const float *__restrict__ Ub,
    size_t ufs, size_t plane, float *__restrict__ coefb, size_t cfs, float delta, float gamma,
    float alpha_s, float omega, unsigned bx, unsigned by, unsigned f)
{
    __shared__ float sU[kAEY][kAEX], sV[kAEY][kAEX], sW[kAEY][kAEX];
    __shared__ float sIx[kADY][kADX], sIy[kADY][kADX], sAs[kADY][kADX];
    const int tx0 = bx * kAX, ty0 = by * kAY;
    if (tx0 >= 2 && ty0 >= 2 && tx0 + kAX + 2 <= w && ty0 + kAY + 2 <= h)
        coeff_tile<true>(sU, sV, sW, sIx, sIy, sAs, I0b, I0xb, I0yb, I1b, w, h, pitch, pfs, Ub,
                         ufs, plane, coefb, cfs, delta, gamma, alpha_s, omega, bx, by, f);
    else
        coeff_tile<false>(sU, sV, sW, sIx, sIy, sAs, I0b, I0xb, I0yb, I1b, w, h, pitch, pfs, Ub,
                          ufs, plane, coefb, cfs, delta, gamma, alpha_s, omega, bx, by, f);
}

template <typename T>
__global__ void __launch_bounds__(kAX * kAY)
var_coeff_kernel(const T *__restrict__ I0b, const T *__restrict__ I0xb,
                 const T *__restrict__ I0yb, const T *__restrict__ I1b, int w, int h,
                 int pitch, size_t pfs, const float *__restrict__ Ub, size_t ufs, size_t plane,
                 float *__restrict__ coefb, size_t cfs, float delta, float gamma, float alpha_s,
                 float omega)
{
    var_coeff_body(I0b, I0xb, I0yb, I1b, w, h, pitch, pfs, Ub, ufs, plane, coefb, cfs, delta,
                   gamma, alpha_s, omega, blockIdx.x, blockIdx.y, blockIdx.z);
}

template <typename T>
__global__ void __launch_bounds__(kAX * kAY)
seg_var_coeff_kernel(const __grid_constant__ SegTable<SegCoeff> tab)
{
    int b;
    const SegCoeff &a = seg_of(tab, b);
    const int r = b / a.gx;
    var_coeff_body((const T *)a.I0, (const T *)a.I0x, (const T *)a.I0y, (const T *)a.I1, a.w, a.h,
                   a.pitch, a.pfs, a.U, a.ufs, a.plane, a.coef + kCoefShift, a.cfs, a.delta, a.gamma,
                   a.alpha_s, a.omega, b % a.gx, r % a.gy, r / a.gy);
}

// Column-walk form of the same kernel.  A warp owns 28 output columns: lane
// l holds column x = x0 - 2 + l, lanes 2..29 are outputs and lanes 0, 1, 30,
// 31 the halo that the central differences and the forward differences of
// the smoothness term need.  The warp walks R output rows down and keeps
// the rows it needs in registers: W (the warped sample I1(x + U)) of rows
// y .. y + 2, Ix, Iy and the smoothness weight of rows y - 1 .. y + 1, U and
// V of rows y - 1 .. y + 2; horizontal neighbours come from lane shuffles.
// Each row's U, V loads are issued two iterations and its bilinear taps one
// iteration before their use.  Values of positions outside the level are 0,
// as in the staging windows of coeff_tile, and every clamp and border test
// is the tile form's; the arithmetic has a fixed rounding sequence (fmul,
// fadd, ffma), so both forms write the same coefficients bit for bit.  Seven
// blocks of 72 registers per SM: a 1280 x 720 level's 1058 blocks take one
// wave (at eight blocks, 64 registers, the kernel spilled).
constexpr int kCWOut = 28;   // output columns per warp
constexpr int kCWWarps = 4;  // warps per block, row strips stacked
constexpr int kCWRows = 8;   // output rows per warp (default; ebof_params.coeff_cw_rows)

template <int R, bool IN, typename T, bool COH = false>
__device__ __forceinline__ void coeff_strip(const T *__restrict__ I0, const T *__restrict__ I0x,
                                            const T *__restrict__ I0y, const T *__restrict__ I1,
                                            int w, int h, int pitch, const float *__restrict__ U,
                                            const float *__restrict__ V, float *__restrict__ cf,
                                            int pl, int x, int y0, bool out_lane, float delta,
                                            float gamma, float alpha_s, float omega)
{
    const bool xin = IN || (x >= 0 && x < w);
    const bool hx = IN || x + 1 < w;
    const bool bl = IN || x > 0;
    const int ylast = y0 + R + 1;  // last row whose W, U and V are read
    auto row_in = [&](int r) { return IN || (r >= 0 && r < h); };
    auto load_uv = [&](int r, float &u, float &v) {
        u = 0.0f;
        v = 0.0f;
        if (row_in(r) && xin) {
            const int p = r * pitch + x;
            u = ldf<COH>(U + p);
            v = ldf<COH>(V + p);
        }
    };
    auto taps = [&](int r, float u, float v) {
        BilTaps t = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (row_in(r) && xin) t = bil_taps_i(I1, w, h, pitch, (float)x + u, (float)r + v);
        return t;
    };
    // neighbour in x with the clamp of the central differences
    auto right = [&](float c) {
        const float n = __shfl_down_sync(kFull, c, 1);
        return (IN || x + 1 < w) ? n : c;
    };
    auto left = [&](float c) {
        const float n = __shfl_up_sync(kFull, c, 1);
        return (IN || x > 0) ? n : c;
    };
    // Ix, Iy and the smoothness weight of row r from W of rows r - 1 .. r + 1
    // and U, V of rows r, r + 1
    auto derive = [&](int r, float wm, float w0, float wp, float u0, float u1, float v0,
                      float v1, float &ix, float &iy, float &as) {
        ix = cdiff(right(w0), left(w0));
        iy = cdiff((IN || r + 1 < h) ? wp : w0, (IN || r > 0) ? wm : w0);
        as = smooth_weight(u0, __shfl_down_sync(kFull, u0, 1), u1, v0,
                           __shfl_down_sync(kFull, v0, 1), v1, hx, IN || r + 1 < h, alpha_s);
    };

    // prologue: U, V of rows y0 - 2 .. y0 + 3, W of rows y0 - 2 .. y0 + 1,
    // the derivatives of rows y0 - 1 and y0, the taps of row y0 + 2
    float ua, va, ub, vb, uc, vc, ud, vd, u2, v2, u3, v3;
    load_uv(y0 - 2, ua, va);
    load_uv(y0 - 1, ub, vb);
    load_uv(y0, uc, vc);
    load_uv(y0 + 1, ud, vd);
    load_uv(y0 + 2, u2, v2);
    load_uv(y0 + 3, u3, v3);
    const float wa = bil_lerp(taps(y0 - 2, ua, va));
    const float wb = bil_lerp(taps(y0 - 1, ub, vb));
    float wc = bil_lerp(taps(y0, uc, vc));
    float wd = bil_lerp(taps(y0 + 1, ud, vd));
    BilTaps t2 = taps(y0 + 2, u2, v2);
    float ixm, iym, asm_, ix0, iy0, as0;
    derive(y0 - 1, wa, wb, wc, ub, uc, vb, vc, ixm, iym, asm_);
    derive(y0, wb, wc, wd, uc, ud, vc, vd, ix0, iy0, as0);
    auto ld_t = [&](const T *a, int p) { return ldp(&a[p]); };
    int p = y0 * pitch + x;
    const bool pin = row_in(y0) && xin;
    float i0 = pin ? ld_t(I0, p) : 0.0f, i0x = pin ? ld_t(I0x, p) : 0.0f;
    float i0y = pin ? ld_t(I0y, p) : 0.0f;

#pragma unroll 1
    for (int y = y0; y < y0 + R; ++y) {
        if (!IN && y >= h) break;
        // W, derivatives of row y + 1
        const float we = bil_lerp(t2);
        float ixp, iyp, asp_;
        derive(y + 1, wc, wd, we, ud, u2, vd, v2, ixp, iyp, asp_);
        // loads for the next iterations
        BilTaps t3 = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (y + 3 <= ylast) t3 = taps(y + 3, u3, v3);
        float u4 = 0.0f, v4 = 0.0f;
        if (y + 4 <= ylast) load_uv(y + 4, u4, v4);
        const int pn = p + pitch;
        const bool nin = y + 1 < y0 + R && row_in(y + 1) && xin;
        const float n_i0 = nin ? ld_t(I0, pn) : 0.0f, n_i0x = nin ? ld_t(I0x, pn) : 0.0f;
        const float n_i0y = nin ? ld_t(I0y, pn) : 0.0f;
        // the system of row y
        const PixelSystem ps = pixel_system_vals(
            ix0, iy0, left(ix0), right(ix0), (IN || y > 0) ? ixm : ix0,
            (IN || y + 1 < h) ? ixp : ix0, (IN || y > 0) ? iym : iy0,
            (IN || y + 1 < h) ? iyp : iy0, wc, as0, __shfl_up_sync(kFull, as0, 1),
            __shfl_down_sync(kFull, as0, 1), asm_, asp_, uc, __shfl_up_sync(kFull, uc, 1),
            __shfl_down_sync(kFull, uc, 1), ub, ud, vc, __shfl_up_sync(kFull, vc, 1),
            __shfl_down_sync(kFull, vc, 1), vb, vd, bl, hx, IN || y > 0, IN || y + 1 < h, x, y,
            w, h, i0, i0x, i0y, delta, gamma, omega);
        if (out_lane && xin) {
            float *c = cf + p;
            c[kCI11 * pl] = ps.i11;
            c[kCI22 * pl] = ps.i22;
            c[kCA12 * pl] = ps.a12;
            c[kCB1 * pl] = ps.b1;
            c[kCB2 * pl] = ps.b2;
            c[kCAS * pl] = as0;
        }
        // move the windows down one row
        ixm = ix0; iym = iy0; asm_ = as0;
        ix0 = ixp; iy0 = iyp; as0 = asp_;
        wc = wd; wd = we;
        ub = uc; vb = vc; uc = ud; vc = vd; ud = u2; vd = v2; u2 = u3; v2 = v3; u3 = u4; v3 = v4;
        t2 = t3;
        p = pn;
        i0 = n_i0; i0x = n_i0x; i0y = n_i0y;
    }
}

template <int R, typename T>
__global__ void __launch_bounds__(32 * kCWWarps, 7)
var_coeff_cw_kernel(const T *__restrict__ I0b, const T *__restrict__ I0xb,
                    const T *__restrict__ I0yb, const T *__restrict__ I1b, int w, int h,
                    int pitch, size_t pfs, const float *__restrict__ Ub, size_t ufs,
                    size_t plane, float *__restrict__ coefb, size_t cfs, float delta,
                    float gamma, float alpha_s, float omega)
{
    const int lane = threadIdx.x;
    const int y0 = (blockIdx.y * kCWWarps + threadIdx.y) * R;
    if (y0 >= h) return;  // the whole warp
    const int f = blockIdx.z;
    const int cx0 = blockIdx.x * kCWOut - 2;  // column of lane 0
    const size_t po = (size_t)f * pfs;
    const float *U = Ub + (size_t)f * ufs;
    const bool out_lane = lane >= 2 && lane < 2 + kCWOut;
    if (cx0 >= 0 && cx0 + 31 < w && y0 >= 2 && y0 + R + 1 < h)
        coeff_strip<R, true>(I0b + po, I0xb + po, I0yb + po, I1b + po, w, h, pitch, U, U + plane,
                             coefb + (size_t)f * cfs, (int)plane, cx0 + lane, y0, out_lane,
                             delta, gamma, alpha_s, omega);
    else
        coeff_strip<R, false>(I0b + po, I0xb + po, I0yb + po, I1b + po, w, h, pitch, U,
                              U + plane, coefb + (size_t)f * cfs, (int)plane, cx0 + lane, y0,
                              out_lane, delta, gamma, alpha_s, omega);
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

// U + dU of the output pixels.  staged: this thread's slots after stage_flow,
// or null: the flow is read here, through L2 (another SM may have written it
// earlier in the launch).
template <int VS, int WARPS>
__device__ __forceinline__ void store_flow(const StripPlace<VS, WARPS> &p, const Strip<VS> &s,
                                           const float *Uin, float *Uout, size_t plane,
                                           const float2 *staged)
{
    if (staged) asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
    for (int r = 0; r < VS; ++r) {
        if (r < p.r0 || r >= p.r1) continue;
        const int o = (p.gy + r) * p.pitch + p.gx;
        const float2 d0 = upk(s.d[r][0]), d1 = upk(s.d[r][1]);
        float2 u = make_float2(0.0f, 0.0f), v = u;
        if (staged) {
            u = staged[(2 * r) * 32 * WARPS];
            v = staged[(2 * r + 1) * 32 * WARPS];
        } else {
            if (p.c0) u.x = __ldcg(Uin + o), v.x = __ldcg(Uin + plane + o);
            if (p.c1) u.y = __ldcg(Uin + o + 1), v.y = __ldcg(Uin + plane + o + 1);
        }
        if (p.c0 && p.c1) {
            *reinterpret_cast<float2 *>(Uout + o) = make_float2(u.x + d0.x, u.y + d1.x);
            *reinterpret_cast<float2 *>(Uout + plane + o) = make_float2(v.x + d0.y, v.y + d1.y);
        } else if (p.c0) {
            Uout[o] = u.x + d0.x;
            (Uout + plane)[o] = v.x + d0.y;
        } else if (p.c1) {
            Uout[o + 1] = u.y + d1.x;
            (Uout + plane)[o + 1] = v.y + d1.y;
        }
    }
}

// A region of 64 columns x VS * WARPS rows, its coefficients loaded straight
// into registers.  COH: the planes and U were written earlier in the launch.
// su: the block's flow stage (COH: none).
template <int VS, int WARPS, bool COH>
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
            const float2 i1 = ldf2<COH>(c + kCI11 * pl), i2 = ldf2<COH>(c + kCI22 * pl);
            const float2 a = ldf2<COH>(c + kCA12 * pl), g = ldf2<COH>(c + kCAS * pl);
            const float2 b1 = ldf2<COH>(c + kCB1 * pl), b2 = ldf2<COH>(c + kCB2 * pl);
            s.i11[r][0] = i1.x, s.i11[r][1] = i1.y;
            s.i22[r][0] = i2.x, s.i22[r][1] = i2.y;
            s.a12[r][0] = a.x, s.a12[r][1] = a.y;
            as[r + 1][0] = g.x, as[r + 1][1] = g.y;
            s.b[r][0] = pk(b1.x, b2.x);
            s.b[r][1] = pk(b1.y, b2.y);
        }
        const float *ca = c0 + kCAS * pl;
        const float2 z = make_float2(0.0f, 0.0f);
        const float2 gu = first ? z : ldf2<COH>(ca - pitch);
        const float2 gd = last ? z : ldf2<COH>(ca + VS * pitch);
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
                auto ld = [&](int k) { return in ? ldf<COH>(c + k * pl) : 0.0f; };
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
    if (!COH) stage_flow(p, Uin, plane, smem_u32(slot));
    clear_ends(ends);
    if (inside)
        edge_weights<VS, true>(s, as, lane, first, last, p.gx, p.gy, w, h);
    else
        edge_weights<VS, false>(s, as, lane, first, last, p.gx, p.gy, w, h);
    sor_sweeps<VS, WARPS>(s, ends, lane, wp, (p.gx + p.gy) & 1, n_half, omega);
    store_flow(p, s, Uin, Uoutb + (size_t)f * ufs, plane, COH ? nullptr : slot);
}

template <int VS>
__global__ void __launch_bounds__(kVThreads, 1)
var_sor_kernel(int w, int h, int pitch, const float *__restrict__ Uinb,
               float *__restrict__ Uoutb, size_t ufs, size_t plane,
               const float *__restrict__ coefb, size_t cfs, int R, int n_half, float omega)
{
    extern __shared__ float2 su[];
    __shared__ StripEnds<kVWarps> ends;
    sor_region<VS, kVWarps, false>(blockIdx.x, blockIdx.y, blockIdx.z, w, h, pitch, Uinb, Uoutb,
                                   ufs, plane, coefb, cfs, R, n_half, omega, ends, su);
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
    sor_region<kVS, kVWarps, false>(b % a.gx, r % a.gy, r / a.gy, a.w, a.h, a.pitch, a.Uin,
                                    a.Uout, a.ufs, a.plane, a.coef + kCoefShift, a.cfs, a.R,
                                    a.n_half, a.omega, ends, su);
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

__global__ void __launch_bounds__(kVThreads, 1)
var_sor_tma_kernel(const __grid_constant__ CUtensorMap cmap, int w, int h, int pitch,
                   const float *__restrict__ Uinb, float *__restrict__ Uoutb, size_t ufs,
                   size_t plane, int R, int nrx, int nry, int total, int n_half, float omega,
                   long long wait_limit, int *err)
{
    extern __shared__ __align__(1024) float tsm[];
    float *cbuf = tsm;  // [kCPlanes][kVR][kTmaBoxW]
    float2 *slot = reinterpret_cast<float2 *>(tsm + kTmaCoefFloats) + threadIdx.x;
    __shared__ StripEnds<kVWarps> ends;
    __shared__ __align__(8) unsigned long long mbar_s;
    const uint32_t mbar = smem_u32(&mbar_s);
    const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
    const int per_frame = nrx * nry, tile = kVR - 2 * R;
    const unsigned long long map_addr = (unsigned long long)&cmap;
    const uint32_t dst = smem_u32(cbuf);

    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    clear_ends(ends);
    __syncthreads();
    // the tensor map's column x + 1 is the level's column x
    auto issue = [&](int r) {  // thread 0: the tensor copy of region r
        const int f = r / per_frame, rem = r - f * per_frame;
        const int ry = rem / nrx, rx = rem - ry * nrx;
        const int bx0 = (rx * tile - R + kCoefShift) & ~3, by0 = ry * tile - R;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar),
                     "r"((unsigned)(kTmaCoefFloats * sizeof(float)))
                     : "memory");
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes "
            "[%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
            "l"(map_addr), "r"(bx0), "r"(by0), "r"(0), "r"(f), "r"(mbar)
            : "memory");
    };
    int r = blockIdx.x;
    if (t == 0 && r < total) issue(r);
    uint32_t parity = 0;
#pragma unroll 1
    for (; r < total; r += gridDim.x) {
        const bool ok = mbar_wait(mbar, parity, wait_limit);
        const int f = r / per_frame, rem = r - f * per_frame;
        const int ry = rem / nrx, rx = rem - ry * nrx;
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
        // every thread holds its coefficients: the buffer is free
        if (__syncthreads_or(!ok)) {
            if (t == 0) {
                atomicOr(err, kErrTimeout);
                // let the copy in flight land before the block exits (bounded
                // by the default limit, whatever the first wait's was)
                mbar_wait(mbar, parity, kWaitLimitDefault);
            }
            return;
        }
        parity ^= 1u;
        if (t == 0 && r + (int)gridDim.x < total) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue(r + gridDim.x);
        }
        const float *Uin = Uinb + (size_t)f * ufs;
        stage_flow(p, Uin, plane, smem_u32(slot));
        if (p.inside(lane, wp))
            edge_weights<kVS, true>(s, as, lane, first, last, p.gx, p.gy, w, h);
        else
            edge_weights<kVS, false>(s, as, lane, first, last, p.gx, p.gy, w, h);
        sor_sweeps<kVS, kVWarps>(s, ends, lane, wp, (p.gx + p.gy) & 1, n_half, omega);
        store_flow(p, s, Uin, Uoutb + (size_t)f * ufs, plane, slot);
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

// The whole variational refinement of a level in one launch.  The work is a
// list of items (iteration, region of 64 x 16 VS), iteration by iteration; a
// block claims them in order from a counter, the next one while it works on
// the last:
//  E. It waits for the previous iteration of the region and its eight
//     neighbours (the halo and the 2 px around are no wider than an interior).
//  A. It stages the flow of the region and 2 px around, and the warped image
//     there (positions outside the level are those of the nearest pixel
//     inside, which gives the replicated borders of the differences).
//  B. The warped image's derivatives and the smoothness weights, 1 px around.
//  C. Each thread builds the systems of its strip in registers, where the
//     sweeps use them: they never leave the SM.
//  D. The sweeps, then U + dU of the interior to the other flow buffer.
// The arithmetic is that of the per-iteration kernels, pixel by pixel with the
// same rounding, so the flow is the same bit for bit.
//
// Items are claimed by running blocks and in order, so whatever an item waits
// for is already claimed by a block that runs: the kernel ends with any number
// of blocks resident, beside any other kernel, and needs no cooperative launch
// (which, inside a CUDA graph, cost more than the ten launches it replaced).
//
// It pays where an iteration's two launches are latency: the launches
// themselves, and three round trips through L2 (flow, image, coefficients)
// before the sweeps start.  The halo's systems are built again by every region
// that holds them (1.9 times at 64 x 64, 3.2 at 64 x 32).  A 64 x 32 item takes
// about 12500 cycles: the wait and the release 3000, A 2400, B 1300, C 2700,
// the sweeps 2700.  Measured, with the launches of one iteration each in
// brackets: a 346 x 260 window 165 us (175; both inside a graph), outside a
// graph, where every launch costs more, 613 x 397 windows with all outputs 234
// us (315) and the flow block on 641 x 479 surfaces 401 us (497).
//
// ctl: [0] the claim counter, [1] blocks gone, [2 + r] finished iterations of
// region r.  The last block to leave sets them to 0 for the next launch.  Waits
// are bounded; a block whose wait runs out reports kErrTimeout and leaves.
constexpr int kLvW = kVR + 4;  // staged columns
template <int VS>
constexpr size_t level_smem_bytes()
{
    return (size_t)6 * kLvW * (VS * kVWarps + 4) * sizeof(float);
}

template <int VS, typename T>
__global__ void __launch_bounds__(kVThreads, 1)
var_level_kernel(const T *__restrict__ I0b, const T *__restrict__ I0xb,
                 const T *__restrict__ I0yb, const T *__restrict__ I1b, int w, int h, int pitch,
                 size_t pfs, float *Ua, float *Ub, size_t ufs, size_t plane, int outer, int n_half,
                 int R, int nrx, int nry, float delta, float gamma, float alpha_s, float omega,
                 int blocks, unsigned *ctl, long long wait_limit, int *err)
{
    constexpr int RH = VS * kVWarps, WH = RH + 4, NP = kLvW / 2;  // pairs of a staged row
    extern __shared__ __align__(16) float lsm[];
    float *sU = lsm, *sV = sU + kLvW * WH, *sW = sV + kLvW * WH;
    float *sIx = sW + kLvW * WH, *sIy = sIx + kLvW * WH, *sAs = sIy + kLvW * WH;
    __shared__ StripEnds<kVWarps> ends;
    const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
    __shared__ int s_item;
    const int per_frame = nrx * nry, total = outer * blocks;
    clear_ends(ends);
    const float wm1 = (float)(w - 1), hm1 = (float)(h - 1);
    auto pr = [](const float *a) { return *reinterpret_cast<const pair_t *>(a); };
    if (t == 0) s_item = (int)atomicAdd(ctl, 1u);
    __syncthreads();
    for (int item = s_item; item < total; item = s_item) {
        const unsigned next = t == 0 ? atomicAdd(ctl, 1u) : 0u;
        const int k = item / blocks, reg = item - k * blocks, f = reg / per_frame;
        const int rem = reg - f * per_frame, by = rem / nrx, bx = rem - by * nrx;
        const StripPlace<VS, kVWarps> p(bx, by, R, w, h, pitch, lane, wp);
        const int rx0 = p.gx - 2 * lane, ry0 = p.gy - wp * VS;
        const size_t po = (size_t)f * pfs;
        const T *I0 = I0b + po, *I0x = I0xb + po, *I0y = I0yb + po, *I1 = I1b + po;
        // the staged window lies in the level (block-uniform)
        const bool inside = rx0 >= 2 && ry0 >= 2 && rx0 + kVR + 2 <= w && ry0 + RH + 2 <= h;
        const float *a = ((k & 1) ? Ub : Ua) + (size_t)f * ufs;
        float *b = ((k & 1) ? Ua : Ub) + (size_t)f * ufs;
        // the strip's template values, which do not depend on the wait
        pair_t i0[VS], i0x[VS], i0y[VS];
#pragma unroll
        for (int r = 0; r < VS; ++r) {
            const int gx = p.gx, gy = p.gy + r, o = gy * pitch + gx;
            const bool in0 = inside || (gx >= 0 && gx < w && gy >= 0 && gy < h);
            const bool in1 = inside || (gx + 1 >= 0 && gx + 1 < w && gy >= 0 && gy < h);
            i0[r] = pk(in0 ? ldp(I0 + o) : 0.0f, in1 ? ldp(I0 + o + 1) : 0.0f);
            i0x[r] = pk(in0 ? ldp(I0x + o) : 0.0f, in1 ? ldp(I0x + o + 1) : 0.0f);
            i0y[r] = pk(in0 ? ldp(I0y + o) : 0.0f, in1 ? ldp(I0y + o + 1) : 0.0f);
        }
        // E
        bool late = false;
        if (k > 0 && t < 9) {
            const int nx = bx + t % 3 - 1, ny = by + t / 3 - 1;
            if (nx >= 0 && nx < nrx && ny >= 0 && ny < nry) {
                const unsigned *q = ctl + 2 + f * per_frame + ny * nrx + nx;
                late = true;
                for (long long it = 0; it < wait_limit; ++it) {
                    unsigned got;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];"
                                 : "=r"(got)
                                 : "l"(q)
                                 : "memory");
                    if ((int)got >= k) {
                        late = false;
                        break;
                    }
                }
            }
        }
        if (__syncthreads_or(late)) {
            if (t == 0) atomicOr(err, kErrTimeout);
            break;
        }
        // A
        constexpr int NI = NP * WH, KI = 3;
#pragma unroll 1
        for (int i0 = t; i0 < NI; i0 += kVThreads * KI) {
            pair_t u[KI], v[KI], x[KI], y[KI];
#pragma unroll
            for (int j = 0; j < KI; ++j) {
                const int i = min(i0 + kVThreads * j, NI - 1);
                const int row = i / NP, gx = rx0 - 2 + 2 * (i - row * NP), gy = ry0 - 2 + row;
                if (inside) {
                    const float *q = a + gy * pitch + gx;
                    const float2 uu = __ldcg(reinterpret_cast<const float2 *>(q));
                    const float2 vv = __ldcg(reinterpret_cast<const float2 *>(q + plane));
                    u[j] = pk(uu.x, uu.y);
                    v[j] = pk(vv.x, vv.y);
                    x[j] = pk((float)gx, (float)(gx + 1));
                    y[j] = dup((float)gy);
                } else {
                    const int c0 = clampi(gx, 0, w - 1), c1 = clampi(gx + 1, 0, w - 1);
                    const int cy = clampi(gy, 0, h - 1);
                    const float *q = a + cy * pitch;
                    u[j] = pk(__ldcg(q + c0), __ldcg(q + c1));
                    v[j] = pk(__ldcg(q + plane + c0), __ldcg(q + plane + c1));
                    x[j] = pk((float)c0, (float)c1);
                    y[j] = dup((float)cy);
                }
            }
            Taps2 tp[KI];
#pragma unroll
            for (int j = 0; j < KI; ++j)
                tp[j] = bil_taps2(I1, w, h, pitch, fadd2(x[j], u[j]), fadd2(y[j], v[j]));
#pragma unroll
            for (int j = 0; j < KI; ++j) {
                const int i = i0 + kVThreads * j;
                if (i < NI) {
                    *reinterpret_cast<pair_t *>(sU + 2 * i) = u[j];
                    *reinterpret_cast<pair_t *>(sV + 2 * i) = v[j];
                    *reinterpret_cast<pair_t *>(sW + 2 * i) = bil_lerp2(tp[j]);
                }
            }
        }
        __syncthreads();
        // B: rows 1 .. WH - 2 (the first and last column's left and right
        // neighbours are another row's; nothing reads those results)
#pragma unroll 1
        for (int i = NP + t; i < NP * (WH - 1); i += kVThreads) {
            const int e = 2 * i;
            const pair_t half = dup(0.5f);
            const float2 u = upk(pr(sU + e)), v = upk(pr(sV + e)), wc = upk(pr(sW + e));
            const float un = sU[e + 2], vn = sV[e + 2];
            const pair_t ix = pk(fsub(wc.y, sW[e - 1]), fsub(sW[e + 2], wc.x));
            const pair_t iy = fsub2(pr(sW + e + kLvW), pr(sW + e - kLvW));
            const pair_t ux = pk(fsub(u.y, u.x), fsub(un, u.y));
            const pair_t vx = pk(fsub(v.y, v.x), fsub(vn, v.y));
            const pair_t uy = fsub2(pr(sU + e + kLvW), pk(u.x, u.y));
            const pair_t vy = fsub2(pr(sV + e + kLvW), pk(v.x, v.y));
            const pair_t q = psi_prime2(ffma2(vy, vy, ffma2(vx, vx, ffma2(uy, uy, fmul2(ux, ux)))));
            *reinterpret_cast<pair_t *>(sIx + e) = fmul2(half, ix);
            *reinterpret_cast<pair_t *>(sIy + e) = fmul2(half, iy);
            *reinterpret_cast<pair_t *>(sAs + e) = fmul2(dup(alpha_s), q);
        }
        __syncthreads();
        // C
        Strip<VS> s;
#pragma unroll
        for (int r = 0; r < VS; ++r) {
            const int e = (wp * VS + r + 2) * kLvW + 2 * lane + 2;
            const int gx = p.gx, gy = p.gy + r;
            const pair_t half = dup(0.5f);
            auto cd2 = [&](pair_t hi, pair_t lo) { return fmul2(half, fsub2(hi, lo)); };
            const bool top = !inside && gy <= 0, bottom = !inside && gy + 1 >= h;
            const bool c0 = inside || (gx >= 0 && gx < w), c1 = inside || (gx + 1 >= 0 && gx + 1 < w);
            const bool row_in = inside || (gy >= 0 && gy < h);
            const bool in0 = c0 && row_in, in1 = c1 && row_in;
            const pair_t ix = pr(sIx + e), iy = pr(sIy + e);
            const pair_t ixu = top ? ix : pr(sIx + e - kLvW), ixd = bottom ? ix : pr(sIx + e + kLvW);
            const pair_t iyu = top ? iy : pr(sIy + e - kLvW), iyd = bottom ? iy : pr(sIy + e + kLvW);
            const float2 ixv = upk(ix);
            // clamped neighbours along x
            const bool l0 = inside || gx > 0, r0 = inside || gx + 1 < w;
            const bool l1 = inside || gx + 1 > 0, r1 = inside || gx + 2 < w;
            const pair_t Ixx = fmul2(half, pk(fsub(r0 ? ixv.y : ixv.x, l0 ? sIx[e - 1] : ixv.x),
                                              fsub(r1 ? sIx[e + 2] : ixv.y, l1 ? ixv.x : ixv.y)));
            const pair_t Ixy = cd2(ixd, ixu), Iyy = cd2(iyd, iyu);
            const pair_t Iz = fsub2(pr(sW + e), i0[r]);
            const pair_t Ixz = fsub2(ix, i0x[r]), Iyz = fsub2(iy, i0y[r]);
            const pair_t z2 = dup(kZeta2);
            const pair_t xx = fmul2(Ixx, Ixx), yy = fmul2(Ixy, Ixy);
            const float2 n1 = upk(fadd2(ffma2(iy, iy, fmul2(ix, ix)), z2));
            const float2 n2 =
                upk(fadd2(ffma2(Iyy, Iyy, ffma2(fmul2(dup(2.0f), Ixy), Ixy, xx)), z2));
            const pair_t nd = pk(rcp_normal(n1.x), rcp_normal(n1.y));
            const pair_t ng = pk(rcp_normal(n2.x), rcp_normal(n2.y));
            float2 adv =
                upk(fmul2(fmul2(dup(delta), nd), psi_prime2(fmul2(fmul2(nd, Iz), Iz))));
            float2 agv = upk(fmul2(fmul2(dup(gamma), ng),
                                   psi_prime2(fmul2(ng, ffma2(Iyz, Iyz, fmul2(Ixz, Ixz))))));
            const pair_t u = pr(sU + e), v = pr(sV + e);
            const float2 wx = upk(fadd2(pk((float)gx, (float)(gx + 1)), u));
            const float2 wy = upk(fadd2(dup((float)gy), v));
            if (wx.x < 0.0f || wx.x > wm1 || wy.x < 0.0f || wy.x > hm1) adv.x = agv.x = 0.0f;
            if (wx.y < 0.0f || wx.y > wm1 || wy.y < 0.0f || wy.y > hm1) adv.y = agv.y = 0.0f;
            const pair_t ad = pk(adv.x, adv.y), ag = pk(agv.x, agv.y);
            // edge weights, 0 where the edge leaves the level
            const pair_t as = pr(sAs + e);
            const float2 av = upk(as);
            const float mid = fmul(0.5f, fadd(av.x, av.y));
            const float wl = l0 ? fmul(0.5f, fadd(av.x, sAs[e - 1])) : 0.0f;
            const float wr = r1 ? fmul(0.5f, fadd(av.y, sAs[e + 2])) : 0.0f;
            const pair_t cl = pk(wl, l1 ? mid : 0.0f), cr = pk(r0 ? mid : 0.0f, wr);
            const pair_t cu = top ? 0 : fmul2(half, fadd2(as, pr(sAs + e - kLvW)));
            const pair_t cd = bottom ? 0 : fmul2(half, fadd2(as, pr(sAs + e + kLvW)));
            const pair_t sw = fadd2(fadd2(fadd2(cl, cr), cu), cd);
            auto smooth = [&](const float *q, pair_t c) {
                const float2 m = upk(c);
                const pair_t dl = pk(fsub(q[e - 1], m.x), fsub(m.x, m.y));
                const pair_t dr = pk(fsub(m.y, m.x), fsub(q[e + 2], m.y));
                return ffma2(cd, fsub2(pr(q + e + kLvW), c),
                             ffma2(cu, fsub2(pr(q + e - kLvW), c), ffma2(cr, dr, fmul2(cl, dl))));
            };
            const pair_t su = smooth(sU, u), sv = smooth(sV, v);
            const pair_t adx = fmul2(ad, ix), ady = fmul2(ad, iy), nag = neg2(ag);
            const float2 d1 = upk(fadd2(ffma2(ag, ffma2(Ixy, Ixy, xx), fmul2(adx, ix)), sw));
            const float2 d2 = upk(fadd2(ffma2(ag, ffma2(Iyy, Iyy, yy), fmul2(ady, iy)), sw));
            const float2 a12 =
                upk(ffma2(ag, ffma2(Ixy, Iyy, fmul2(Ixx, Ixy)), fmul2(adx, iy)));
            const float2 b1 = upk(ffma2(nag, ffma2(Ixy, Iyz, fmul2(Ixx, Ixz)),
                                        ffma2(neg2(adx), Iz, su)));
            const float2 b2 = upk(ffma2(nag, ffma2(Iyy, Iyz, fmul2(Ixy, Ixz)),
                                        ffma2(neg2(ady), Iz, sv)));
            s.i11[r][0] = in0 ? __fdividef(omega, d1.x) : 0.0f;
            s.i11[r][1] = in1 ? __fdividef(omega, d1.y) : 0.0f;
            s.i22[r][0] = in0 ? __fdividef(omega, d2.x) : 0.0f;
            s.i22[r][1] = in1 ? __fdividef(omega, d2.y) : 0.0f;
            s.a12[r][0] = in0 ? a12.x : 0.0f;
            s.a12[r][1] = in1 ? a12.y : 0.0f;
            s.b[r][0] = in0 ? pk(b1.x, b2.x) : 0;
            s.b[r][1] = in1 ? pk(b1.y, b2.y) : 0;
            // the region's own edges carry no weight, nor do pixels outside
            const float2 lv = upk(cl), uv = upk(cu), dv = upk(cd);
            s.wl[r][0] = lane > 0 && in0 ? lv.x : 0.0f;
            s.wl[r][1] = in1 ? lv.y : 0.0f;
            s.wr[r] = lane < 31 && in1 ? wr : 0.0f;
            const bool up_in = !(r == 0 && wp == 0);
            s.wu[r][0] = up_in && in0 ? uv.x : 0.0f;
            s.wu[r][1] = up_in && in1 ? uv.y : 0.0f;
            if (r == VS - 1) {
                s.wd[0] = wp < kVWarps - 1 && in0 ? dv.x : 0.0f;
                s.wd[1] = wp < kVWarps - 1 && in1 ? dv.y : 0.0f;
            }
        }
        // D
        sor_sweeps<VS, kVWarps>(s, ends, lane, wp, (p.gx + p.gy) & 1, n_half, omega);
#pragma unroll
        for (int r = 0; r < VS; ++r) {
            if (r < p.r0 || r >= p.r1) continue;
            const int e = (wp * VS + r + 2) * kLvW + 2 * lane + 2;
            float *q = b + (p.gy + r) * pitch + p.gx;
            const float2 u = upk(pr(sU + e)), v = upk(pr(sV + e));
            const float2 d0 = upk(s.d[r][0]), d1 = upk(s.d[r][1]);
            if (p.c0 && p.c1) {
                __stcg(reinterpret_cast<float2 *>(q), make_float2(u.x + d0.x, u.y + d1.x));
                __stcg(reinterpret_cast<float2 *>(q + plane), make_float2(v.x + d0.y, v.y + d1.y));
            } else if (p.c0) {
                __stcg(q, u.x + d0.x);
                __stcg(q + plane, v.x + d0.y);
            } else if (p.c1) {
                __stcg(q + 1, u.y + d1.x);
                __stcg(q + plane + 1, v.y + d1.y);
            }
        }
        if (t == 0) s_item = (int)next;
        __syncthreads();  // the block's stores, its reads of the stage
        if (t == 0)  // releases the whole block's stores, which the barrier ordered before it
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ctl + 2 + reg), "r"(k + 1)
                         : "memory");
    }
    // the last block to leave resets the counters
    __shared__ bool s_last;
    if (t == 0) {
        __threadfence();
        s_last = atomicInc(ctl + 1, gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        for (int i = t; i < blocks; i += kVThreads) ctl[2 + i] = 0;
        if (t == 0) ctl[0] = 0;
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

void make_coef_maps(float *work, const Geometry &geo, int frames, CoefMaps *m)
{
    for (int l = 0; l < kMaxLevels; ++l) m->ok[l] = false;
    EncodeTiledFn enc = encode_tiled();
    if (!enc || !work) return;
    for (int l = 0; l < geo.levels; ++l) {
        const Level &lv = geo.lv[l];
        const cuuint64_t dims[4] = {(cuuint64_t)lv.w + kCoefShift, (cuuint64_t)lv.h, (cuuint64_t)kCPlanes,
                                    (cuuint64_t)frames};
        const cuuint64_t strides[3] = {(cuuint64_t)lv.pitch * sizeof(float),
                                       (cuuint64_t)lv.plane * sizeof(float),
                                       (cuuint64_t)kCPlanes * lv.plane * sizeof(float)};
        const cuuint32_t box[4] = {(cuuint32_t)kTmaBoxW, (cuuint32_t)kVR, (cuuint32_t)kCPlanes,
                                   1};
        const cuuint32_t estr[4] = {1, 1, 1, 1};
        m->ok[l] = enc(&m->map[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, work, dims, strides, box,
                       estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
}

bool var_fused_supported(int var_sor)
{
    return kVR - 2 * sor_halo(var_sor) >= 16;
}

void init_var_attributes()
{
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevs) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        g_num_sms[dev] = n;
    }
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

int sor_halo(int var_sor) { return var_sor > 0 ? 2 * var_sor - 1 : 1; }
int sor_tile(int R) { return kVR - 2 * R; }
void coeff_tile_shape(int &x, int &y)
{
    x = kAX;
    y = kAY;
}
int coeff_planes() { return kCPlanes; }

void launch_seg_coeff(const SegTable<SegCoeff> &t, int blocks, bool half, cudaStream_t st)
{
    StageScope sc(kStVarCoeff, 1, st);
    if (half) seg_var_coeff_kernel<__half><<<blocks, dim3(kAX, kAY), 0, st>>>(t);
    else seg_var_coeff_kernel<float><<<blocks, dim3(kAX, kAY), 0, st>>>(t);
}

void launch_seg_sor(const SegTable<SegSor> &t, int blocks, cudaStream_t st)
{
    StageScope sc(kStVarSor, 1, st);
    seg_var_sor_kernel<<<blocks, kVThreads, flow_stage_bytes<kVS, kVWarps>(), st>>>(t);
}

float *launch_variational_fused(const void *I0, const void *I0x, const void *I0y,
                                const void *I1, const Level &lv, size_t pyr_frame_stride,
                                float *U, float *Utmp, size_t u_frame_stride, float *coef,
                                int frames, const FlowParams &fp, const CUtensorMap *coef_map,
                                int *err, cudaStream_t st)
{
    // the level's planes are packed: frame stride kCPlanes planes of this level
    const size_t coef_frame_stride = (size_t)kCPlanes * lv.plane;
    int dev = 0;
    cudaGetDevice(&dev);
    const int nsm = (dev >= 0 && dev < kMaxDevs && g_num_sms[dev] > 0) ? g_num_sms[dev] : 0;
    const int n_half = 2 * fp.var_sor;
    const int R = sor_halo(fp.var_sor);
    const int tile = sor_tile(R);           // interior side of a 64 x 64 region
    const int small = kVSmallRows - 2 * R;  // interior rows of a 64 x 32 region
    coef += kCoefShift;
    const dim3 cgrd((lv.w + kAX - 1) / kAX, (lv.h + kAY - 1) / kAY, frames);
    // the coefficient kernel's form depends on the level's width and the
    // stream's parameters only, so single, batched and grouped windows of a
    // level always run the same one (and give the same coefficients): by
    // default the column walk from 1024 px wide (the finest level of 1280 x
    // 720 frames), where it is the faster; smaller levels keep the tile form
    const bool column_walk = lv.w >= fp.coeff_cw_min_width;
    const int cw_rows = fp.coeff_cw_rows == 4 || fp.coeff_cw_rows == 16 ? fp.coeff_cw_rows
                                                                       : kCWRows;
    const dim3 wgrd((lv.w + kCWOut - 1) / kCWOut,
                    ((lv.h + cw_rows - 1) / cw_rows + kCWWarps - 1) / kCWWarps, frames);
    const dim3 sgrd((lv.w + tile - 1) / tile, (lv.h + tile - 1) / tile, frames);
    // small levels of a single frame: every outer iteration in one launch (same
    // flow bit for bit), where the regions fit one wave and a region's staged
    // window reaches no further than its neighbours' interiors; 64 x 32 regions
    // if they fit, else 64 x 64 (640 x 360: 112 of them, no slower than ten
    // launches inside a graph, 12 % faster outside one).  Not for levels of
    // more than one wave (1280 x 720: 171 us against 145), nor, unless asked
    // for, for several frames, whose launches fill the SMs (640 x 480, eight
    // frames: 1.21 against 1.20 ms a call)
    for (int vs : {kVSmallVS, kVS}) {
        const int ty = vs * kVWarps - 2 * R, nrx = (int)sgrd.x;
        const int nry = ty > 0 ? (lv.h + ty - 1) / ty : 0;
        const long long per = (long long)nrx * nry, blocks = per * frames;
        if (!fp.level_ctl || fp.var_outer < 1 || ty < R + 2 || tile < R + 2 || lv.w < 2 ||
            lv.h < 2 || nsm < 1 || blocks > std::min(nsm, kLevelBlocks) ||
            (frames > 1 && per > fp.var_cluster_max))
            continue;
        const bool small_form = vs == kVSmallVS;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)std::min<long long>(blocks, nsm), 1, 1);
        cfg.blockDim = dim3(kVThreads, 1, 1);
        cfg.dynamicSmemBytes =
            small_form ? level_smem_bytes<kVSmallVS>() : level_smem_bytes<kVS>();
        cfg.stream = st;
        cudaError_t e;
        {
            StageScope sc(kStVarSor, 1, st);
#define EBOF_LV(VS, T)                                                                          \
    cudaLaunchKernelEx(&cfg, var_level_kernel<VS, T>, (const T *)I0, (const T *)I0x,            \
                       (const T *)I0y, (const T *)I1, lv.w, lv.h, lv.pitch, pyr_frame_stride,   \
                       U, Utmp, u_frame_stride, lv.plane, fp.var_outer, n_half, R, nrx, nry,    \
                       fp.delta, fp.gamma, fp.alpha_s, fp.omega, (int)blocks, fp.level_ctl,     \
                       kWaitLimitDefault, err)
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
        if (column_walk) {
            StageScope sc(kStVarCoeff, 1, st);
#define EBOF_CW(R, T)                                                                          \
    var_coeff_cw_kernel<R, T><<<wgrd, dim3(32, kCWWarps), 0, st>>>(                             \
        (const T *)I0, (const T *)I0x, (const T *)I0y, (const T *)I1, lv.w, lv.h, lv.pitch,     \
        pyr_frame_stride, a, u_frame_stride, lv.plane, coef, coef_frame_stride, fp.delta,       \
        fp.gamma, fp.alpha_s, fp.omega)
            if (fp.half) {
                if (cw_rows == 4) EBOF_CW(4, __half);
                else if (cw_rows == 16) EBOF_CW(16, __half);
                else EBOF_CW(kCWRows, __half);
            } else {
                if (cw_rows == 4) EBOF_CW(4, float);
                else if (cw_rows == 16) EBOF_CW(16, float);
                else EBOF_CW(kCWRows, float);
            }
#undef EBOF_CW
        } else {
            StageScope sc(kStVarCoeff, 1, st);
            if (fp.half)
                var_coeff_kernel<__half><<<cgrd, dim3(kAX, kAY), 0, st>>>(
                    (const __half *)I0, (const __half *)I0x, (const __half *)I0y,
                    (const __half *)I1, lv.w, lv.h, lv.pitch, pyr_frame_stride, a,
                    u_frame_stride, lv.plane, coef, coef_frame_stride, fp.delta, fp.gamma,
                    fp.alpha_s, fp.omega);
            else
                var_coeff_kernel<float><<<cgrd, dim3(kAX, kAY), 0, st>>>(
                    (const float *)I0, (const float *)I0x, (const float *)I0y,
                    (const float *)I1, lv.w, lv.h, lv.pitch, pyr_frame_stride, a,
                    u_frame_stride, lv.plane, coef, coef_frame_stride, fp.delta, fp.gamma,
                    fp.alpha_s, fp.omega);
        }
        {
            StageScope sc(kStVarSor, 1, st);
            const int total = (int)(sgrd.x * sgrd.y * sgrd.z);
            const int row_waves = fp.sor_row_waves;
            const dim3 g1(sgrd.x, small > 0 ? (lv.h + small - 1) / small : 1, frames);
            if (coef_map && nsm > 0 && (long long)total >= (long long)fp.sor_tma_min_per_sm * nsm)
                var_sor_tma_kernel<<<std::min(nsm, total), kVThreads, kTmaSmemBytes, st>>>(
                    *coef_map, lv.w, lv.h, lv.pitch, a, b, u_frame_stride, lv.plane, R,
                    (int)sgrd.x, (int)sgrd.y, total, n_half, fp.omega,
                    fp.wait_limit >= 0 ? fp.wait_limit : kWaitLimitDefault, err);
            else if (small >= 8 && (long long)(g1.x * g1.y * g1.z) <= (long long)row_waves * nsm)
                var_sor_kernel<kVSmallVS>
                    <<<g1, kVThreads, flow_stage_bytes<kVSmallVS, kVWarps>(), st>>>(
                        lv.w, lv.h, lv.pitch, a, b, u_frame_stride, lv.plane, coef,
                        coef_frame_stride, R, n_half, fp.omega);
            else
                var_sor_kernel<kVS><<<sgrd, kVThreads, flow_stage_bytes<kVS, kVWarps>(), st>>>(
                    lv.w, lv.h, lv.pitch, a, b, u_frame_stride, lv.plane, coef,
                    coef_frame_stride, R, n_half, fp.omega);
        }
        float *t = a;
        a = b;
        b = t;
    }
    return a;
}

}  // namespace ebof
