// ps_internal.cuh -- device helpers shared by the libps translation units.
// Every TU of the library is compiled with -fmad=false: multiply-adds are
// written as explicit fmaf() so that the forward and the backward kernels,
// which recompute the same per-pixel candidate list, evaluate bit-identical
// arithmetic.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include "ps.h"

#define PS_CUDA_CHECK(expr)                                   \
    do {                                                      \
        cudaError_t e_ = (expr);                              \
        if (e_ != cudaSuccess) return PS_ERR_CUDA;            \
    } while (0)

#define PS_LAUNCH_CHECK()                                     \
    do {                                                      \
        cudaError_t e_ = cudaGetLastError();                  \
        if (e_ != cudaSuccess) return PS_ERR_CUDA;            \
    } while (0)

namespace ps {

// Programmatic dependent launch.  A kernel launched by launch_after may become resident while
// the kernel before it in the stream drains; after_previous(), first in it, lets the next one
// do the same and waits until the one before has finished and its writes are visible (at once
// if the launch was an ordinary one).  The kernels of a step are short enough for the gaps
// between them to count: an eager step of 64 planes in 8 views of 128x96 56 -> 43 us, a fitted
// render of 8 views 121 -> 110, a hard one of 64 views 261 -> 250.  Under capture the launches are
// ordinary: replayed steps were 0..2% slower with programmatic edges.
//
// Such a kernel is resident while the kernels before it still write, and its successors may be
// too.  Whatever a kernel of the chain writes is therefore read by ordinary loads through
// pointers without __restrict__: __ldg and const __restrict__ promise data that nobody writes
// during the kernel's life, so such a load may move above the wait or find an older line.  They
// are left for what is complete before the chain's first kernel (views, supervision, upstream
// gradients, parameters).
__device__ __forceinline__ void after_previous()
{
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                A... args)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(st, &cs);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = &at; cfg.numAttrs = cs == cudaStreamCaptureStatusNone ? 1 : 0;
    const cudaError_t r = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
    if (r != cudaSuccess) cudaGetLastError();      // reported here, not by the next launch's check
    return r;
}

constexpr int kRecFloats = 16;   // floats per record

__device__ __forceinline__ void set_status(int* st, ps_status code)
{
    if (st) atomicOr(st, 1 << (int)code);
}

// Global tile -> view by binary search over tile_off (views sorted by tile_off).
__device__ __forceinline__ int view_of_tile(const ps_view* views, int V, int tile)
{
    int lo = 0, hi = V - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(&views[mid].tile_off) <= tile) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The same by a whole warp: 32 probes per step instead of a chain of dependent loads; every step
// leaves the stride between two probes (one step up to 32 views, two up to 1,024).  A forward of
// 16,384 views of 32x32 took 833 us with view_of_tile, 4,952 with 32 consecutive views per step and
// 340 so; 64 views 26, 20, 20.
__device__ __forceinline__ int warp_view_of_tile(const ps_view* views, int V, int tile)
{
    const int lane = threadIdx.x & 31;
    int lo = 0, n = V;
    for (;;) {
        const int stride = (n + 31) >> 5;
        const int at = lane * stride;
        const bool in = at < n && __ldg(&views[lo + at].tile_off) <= tile;
        // (views are sorted by tile_off and view lo starts at or before the tile)
        const int k = __popc(__ballot_sync(0xffffffffu, in)) - 1;
        lo += k * stride;
        if (stride == 1) return lo;
        n = min(stride, n - k * stride);
    }
}

// One plane in camera coordinates, as stored in a record.
struct Rec {
    float4 n;    // n_c, s = n_c . p_c
    float4 vx;   // v^x_c, a_x = v^x_c . p_c
    float4 vy;   // v^y_c, a_y = v^y_c . p_c
    float4 r;    // r^x+, r^x-, r^y+, r^y-
};

// a / b as a times the approximate reciprocal of b, for 2^-126 <= |b| (what the caller asks of the
// result holds only there).  As accurate as __fdividef (2 ulp) and like it 0 for |b| > 2^126, without
// its care for subnormal b; a and the result may be subnormal.
__device__ __forceinline__ float quotient(float a, float b)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(b));
    return a * y;
}

// e^x = 2^(x log2 e), results below 2^-126 as 0: for a weight that is then below any w_min of at
// least kFlushFrom.  A smaller w_min takes __expf (`tiny`, the same for a whole launch), whose care
// for subnormal results costs a pair three instructions.  3,000 planes in 8 views of 640x480, a step
// at the first lambda: 382 us with __fdividef and __expf, 375 with quotient, 365 with both; 16 rooms
// 1,471, 1,442, 1,420; 10,000 planes in 64 views 5,044, 4,918, 4,822.  (The Eq. 5 weight keeps
// __expf: 2,134 us a step against 2,170 with the branch.)
constexpr float kFlushFrom = 4.7019774e-38f;     // 2^-124
__device__ __forceinline__ float weight_exp(float x, bool tiny)
{
    if (tiny) return __expf(x);
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x * 1.442695041f));
    return y;
}

// Evaluation of one (pixel ray, plane) pair: Eq. 4, 6-9 and the filter of
// Sec. 3.2.  d = (dx, dy, 1).  Returns true if the pair is a candidate.
struct PairEval {
    float t, w;        // depth, weight
    float m;           // margin of the active side
    float P;           // P_X or P_Y of the active side
    float den;         // d . n_c
    float dv;          // d . v_c of the active side
    bool sideX;        // active side is X (m_X < m_Y); ties go to Y
    bool pos;          // P > 0 on the active side (selects r^+)
    // both axes (used by the Gaussian weight of Eq. 5)
    float X, Y;        // P_X, P_Y
    float dvx, dvy;    // d . v^x_c, d . v^y_c
    float sX, sY;      // radius on the side of P_X, P_Y
};

struct SplatConst {
    float lam5;        // 5 lambda
    float w_min;
    float z_near, z_far;
    float reject;      // quick reject: margins below -reject cannot reach w_min
    int hard;          // PS_HARD
    int gauss;         // PS_GAUSSIAN: the Eq. 5 weight
    bool tiny;         // w_min < kFlushFrom
    float kappa;       // Eq. 5: w >= w_min only within kappa radii of the centre on each axis
};

// Every operation is executed for every lane and the filter is applied at the
// end: lanes of a warp leave at different tests, so early returns would only
// serialise the warp.  The selected values are the same as with early exits.
__device__ __forceinline__ bool eval_pair(const float4& n, const float4& vx, const float4& vy,
                                          const float4& r, float dx, float dy,
                                          const SplatConst& c, PairEval& o)
{
    const float den = fmaf(dx, n.x, fmaf(dy, n.y, n.z));
    const float t = quotient(n.w, den);
    const float dvx = fmaf(dx, vx.x, fmaf(dy, vx.y, vx.z));
    const float dvy = fmaf(dx, vy.x, fmaf(dy, vy.y, vy.z));
    const float X = fmaf(t, dvx, -vx.w);
    const float Y = fmaf(t, dvy, -vy.w);
    const float sXr = X > 0.f ? r.x : r.y, sYr = Y > 0.f ? r.z : r.w;
    o.X = X; o.Y = Y; o.dvx = dvx; o.dvy = dvy; o.sX = sXr; o.sY = sYr;
    if (c.gauss) {
        // Eq. 5 in the plane's frame, the one-sided radii as the scales
        const float ux = __fdividef(X, sXr), uy = __fdividef(Y, sYr);
        const float w = __expf(-0.5f * (ux * ux + uy * uy));
        o.t = t; o.w = w; o.m = 0.f; o.den = den;
        o.sideX = false; o.P = Y; o.dv = dvy; o.pos = Y > 0.f;
        return (fabsf(den) > 1e-6f) && (t > c.z_near && t < c.z_far) && (w >= c.w_min);
    }
    const float mX = sXr - fabsf(X);
    const float mY = sYr - fabsf(Y);
    const bool sx = mX < mY;
    const float m = sx ? mX : mY;
    // w = min(1, 2 sigmoid(5 lambda m)); below the clamp 2 sigmoid(x) = 2 e^x / (1 + e^x)
    const float e = weight_exp(c.lam5 * m, c.tiny);
    const float w = (m >= 0.f) ? 1.f : quotient(2.f * e, 1.f + e);
    // (hard edge: w = 1 for m >= 0, which is then the only condition on it)
    const bool ok = (fabsf(den) > 1e-6f) && (t > c.z_near && t < c.z_far) &&
                    (c.hard ? m >= 0.f : (!(m < -c.reject) && (w >= c.w_min)));
    o.t = t; o.w = w; o.m = m; o.den = den;
    o.sideX = sx;
    o.P = sx ? X : Y;
    o.dv = sx ? dvx : dvy;
    o.pos = o.P > 0.f;
    return ok;
}

// Minimum and maximum that are NaN if either argument is.
__device__ __forceinline__ float min_nan(float a, float b)
{
    float d;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

__device__ __forceinline__ float max_nan(float a, float b)
{
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// Rays through the pixel centres at the corners of a warp's pixel rectangle.
struct WarpRegion {
    float dxa, dxb, dya, dyb;
    float den_min;     // 0.01 x the longest of the four rays: den above it is accurate to 3e-5
};

// Conservative test whether a plane can pass the filter at any pixel of a
// warp's rectangle.  For a fixed plane, t = s / (d . n_c) and P = t (d . v_c) - a
// are linear-fractional in the ray d = (dx, dy, 1); if d . n_c keeps its sign
// over the rectangle they are monotone along every line, so their ranges over
// the rectangle are spanned by the four corner rays.  The corner values use
// the per-pixel formulas of eval_pair; the margins cover FP32 rounding.  t_low is
// the smallest depth at the corners, which bounds the depth at every pixel of the
// rectangle from below up to rounding (0 where d . n_c is too small for that).  A plane
// whose depths all lie below t_floor may not hit.
template <bool LOW>
__device__ __forceinline__ bool region_may_hit(const float4& n, const float4& vx, const float4& vy,
                                               const float4& r, const WarpRegion& g,
                                               const SplatConst& c, float& t_low, float t_floor = 0.f)
{
    float tmin = INFINITY, tmax = -INFINITY, xmin = INFINITY, xmax = -INFINITY;
    float ymin = INFINITY, ymax = -INFINITY;
    float dlo = INFINITY, dhi = -INFINITY;
    t_low = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float dx = (k & 1) ? g.dxb : g.dxa;
        const float dy = (k & 2) ? g.dyb : g.dya;
        const float den = fmaf(dx, n.x, fmaf(dy, n.y, n.z));
        dlo = min_nan(dlo, den); dhi = max_nan(dhi, den);      // NaN stays: no bound
        const float t = quotient(n.w, den);
        const float dvx = fmaf(dx, vx.x, fmaf(dy, vx.y, vx.z));
        const float dvy = fmaf(dx, vy.x, fmaf(dy, vy.y, vy.z));
        const float X = fmaf(t, dvx, -vx.w);
        const float Y = fmaf(t, dvy, -vy.w);
        tmin = fminf(tmin, t); tmax = fmaxf(tmax, t);
        xmin = fminf(xmin, X); xmax = fmaxf(xmax, X);
        ymin = fminf(ymin, Y); ymax = fmaxf(ymax, Y);
    }
    if (!(dlo > 2e-6f) && !(dhi < -2e-6f)) return true;       // d . n_c may vanish: no bound
    if constexpr (LOW) {
        if (dlo > g.den_min || dhi < -g.den_min) {
            t_low = tmin;
            if (tmax < t_floor) return false;
        }
    }
    if (tmax < c.z_near * 0.99999f || tmin > c.z_far * 1.00001f) return false;
    // support: r + reject around the rectangle, or kappa r for the Eq. 5 weight
    const float sc = c.gauss ? c.kappa : 1.f;
    const float rej = c.gauss ? 0.f : c.reject;
    const float mx = rej + 1e-5f * (fabsf(xmin) + fabsf(xmax) + fabsf(tmax)) + 1e-6f;
    const float my = rej + 1e-5f * (fabsf(ymin) + fabsf(ymax) + fabsf(tmax)) + 1e-6f;
    if (xmax < -(sc * r.y + mx) || xmin > sc * r.x + mx) return false;
    if (ymax < -(sc * r.w + my) || ymin > sc * r.z + my) return false;
    return true;
}

// Floats per record of the gradient accumulators: the gradients of s (0), of a turn about
// v^y (1) and about -v^x (2) that moves n_c, of a turn about n_c (3), of the radii (4-7),
// and for the Eq. 5 weight those of a_x and a_y (8, 9; the rectangle's follow from the radii).
__host__ __device__ constexpr int grad_stride(int gauss) { return gauss ? 12 : 8; }

// Fused mode: per-view loss sums are added into kSlots partial sums per view
// (spread over L2 slices, so that strips of one view do not serialise on one
// address), which the chain kernel adds up into view_sums.
constexpr int kSlots = 32;

__device__ __forceinline__ double slot_sum(const double* vs_slots, int v, int c)
{
    const double* sp = vs_slots + (size_t)v * kSlots * 4 + c;
    double t = 0.0;
    for (int i = 0; i < kSlots; ++i) t += sp[4 * i];        // in a fixed order
    return t;
}

// A plane's axes (Eq. 2-3): columns of the Hamilton matrix of its normalised quaternion.
struct PlaneAxes {
    float vx[3], vy[3], n[3];
    float w, x, y, z, norm;    // the normalised quaternion and the length it was divided by
};

// Returns false for a quaternion without a direction.
__device__ __forceinline__ bool plane_axes(float q0, float q1, float q2, float q3, PlaneAxes& o)
{
    const float qs = sqrtf(q0 * q0 + q1 * q1 + q2 * q2 + q3 * q3);
    const float w = q0 / qs, x = q1 / qs, y = q2 / qs, z = q3 / qs;
    o.w = w; o.x = x; o.y = y; o.z = z; o.norm = qs;
    o.vx[0] = 1.f - 2.f * (y * y + z * z); o.vx[1] = 2.f * (x * y + w * z); o.vx[2] = 2.f * (x * z - w * y);
    o.vy[0] = 2.f * (x * y - w * z); o.vy[1] = 1.f - 2.f * (x * x + z * z); o.vy[2] = 2.f * (y * z + w * x);
    o.n[0] = 2.f * (x * z + w * y); o.n[1] = 2.f * (y * z - w * x); o.n[2] = 1.f - 2.f * (x * x + y * y);
    return qs > 0.f && isfinite(qs);
}

// Adds one record's part of the centre's gradient.  The centre moves s = n_c . p_c, a_x and a_y
// with p_c = R c + t and the axes n_c = R n, ..., so the part is R^T R (gs n + gax v^x + gay v^y):
// for any 3x3 block R of the view's w2c, orthonormal or not.
__device__ __forceinline__ void add_centre(float (&g)[3], const PlaneAxes& a, float gs, float gax, float gay,
                                           const ps_view* vw)
{
    float R[9], u[3], y[3];
#pragma unroll
    for (int i = 0; i < 9; ++i) R[i] = __ldg(&vw->w2c[4 * (i / 3) + i % 3]);
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i] = fmaf(gs, a.n[i], fmaf(gax, a.vx[i], gay * a.vy[i]));
#pragma unroll
    for (int i = 0; i < 3; ++i) y[i] = fmaf(R[3 * i], u[0], fmaf(R[3 * i + 1], u[1], R[3 * i + 2] * u[2]));
#pragma unroll
    for (int i = 0; i < 3; ++i) g[i] = fmaf(R[i], y[0], fmaf(R[3 + i], y[1], fmaf(R[6 + i], y[2], g[i])));
}

// The torque and the radii of a plane's record gradients (sums over any of its records) ->
// quaternion 4 and radii 4 of the world parameters.
//
// A turn by theta in the plane's own frame moves v^x by theta_z v^y - theta_y n, v^y by theta_x n -
// theta_z v^x and n by theta_y v^x - theta_x v^y, and R takes them to the camera.  At a fixed centre
// what the gradients of n_c, v^x_c and v^y_c find along the others' axes are the moments (mx, my, mz)
// = record floats 1-3, whatever R is: the gradients of v^x_c and v^y_c are multiples of q = t d - p_c
// and that of n_c is one of q and the normal's, with n_c . q = 0, v^x_c . q = P_X, v^y_c . q = P_Y.
// With dq = quat (0, theta) / 2 the quaternion gradient is 2 quat (0, torque) / |quat|.
__device__ __forceinline__ void chain_turn(const PlaneAxes& a, float mx, float my, float mz, const float4& g3,
                                           int single_radii, float (&out)[8])
{
    const float tx = -my, ty = mx, tz = mz;
    const float s2 = 2.f / a.norm;
    out[0] = s2 * -(a.x * tx + a.y * ty + a.z * tz);
    out[1] = s2 * (a.w * tx + a.y * tz - a.z * ty);
    out[2] = s2 * (a.w * ty + a.z * tx - a.x * tz);
    out[3] = s2 * (a.w * tz + a.x * ty - a.y * tx);
    out[4] = single_radii ? g3.x + g3.y : g3.x;
    out[5] = single_radii ? 0.f : g3.y;
    out[6] = single_radii ? g3.z + g3.w : g3.z;
    out[7] = single_radii ? 0.f : g3.w;
}

// Adam with bias correction; values below `lowest` (NaN: none) are raised to it.
__device__ __forceinline__ void adam_value(float& p, float& m, float& v, float g, float lr, float b1, float b2,
                                           float eps, float bc1, float bc2, float lowest)
{
    m = fmaf(b1, m, (1.f - b1) * g);
    v = fmaf(b2, v, (1.f - b2) * g * g);
    const float mh = m / bc1, vh = v / bc2;
    p = p - lr * mh / (sqrtf(vh) + eps);
    if (p < lowest) p = lowest;
}

__device__ __forceinline__ void adam_update(float* __restrict__ p, float* __restrict__ m,
                                            float* __restrict__ v, long long i, float g, float lr, float b1,
                                            float b2, float eps, float bc1, float bc2, float lowest)
{
    float pi = p[i], mi = m[i], vi = v[i];
    adam_value(pi, mi, vi, g, lr, b1, b2, eps, bc1, bc2, lowest);
    m[i] = mi;
    v[i] = vi;
    p[i] = pi;
}

// Record r's part in the binning's counts: its number of tiles, where they start, and +1 / -1
// in the difference array where each row segment of its rectangle starts and ends.
struct BinCount {
    int* rec_cnt;
    int4* rec_info;
    int* diff;
    int n_tiles;
};

__device__ __forceinline__ void count_record(const BinCount& b, size_t r, const int4& rc, int tile_off, int tx,
                                             int v)
{
    int c = 0;
    int4 info = make_int4(0, 1, tx, v);
    if (rc.z >= rc.x && rc.w >= rc.y) {
        const int w = rc.z - rc.x + 1;
        c = w * (rc.w - rc.y + 1);
        const int first = tile_off + rc.y * tx + rc.x;
        info = make_int4(first, w, tx, v);
        if (w == tx) {
            // full rows: one contiguous run of c tiles
            atomicAdd(&b.diff[first], 1);
            if (first + c < b.n_tiles) atomicAdd(&b.diff[first + c], -1);
        } else {
            const int last = first + (rc.w - rc.y) * tx;   // first tile of the last row
            for (int a = first; a <= last; a += tx) {
                atomicAdd(&b.diff[a], 1);
                if (a + w < b.n_tiles) atomicAdd(&b.diff[a + w], -1);
            }
        }
    }
    b.rec_cnt[r] = c;
    b.rec_info[r] = info;
}

// What the entry points of a step ask of their arguments: PS_OK, or what they return before
// anything is launched.
ps_status check_project(const ps_planes* planes, const ps_frame* frame, const ps_settings* s, const float* rec,
                        const int* rect, const float* key);
ps_status check_bin(const ps_frame* frame, const ps_settings* s, const float* rec, const int* rect,
                    const float* key, const int* tile_ptr, const int* tile_ent, const float* tile_key,
                    long long capacity, const long long* d_required, void* ws, size_t ws_bytes);
ps_status check_fwd(const ps_frame* f, const ps_settings* s, const float* rec, const float* key,
                    const int* tile_ptr, const int* tile_ent, long long capacity, const float* depth,
                    const float* normal, void* ws, size_t ws_bytes);
ps_status check_loss(const ps_frame* f, const ps_settings* s, const float* depth, const float* normal,
                     const float* gt_depth, const float* gt_normal, const float* dLdD, const float* dLdN,
                     const double* view_sums);
ps_status check_bwd(const ps_planes* planes, const ps_frame* f, const ps_settings* s, const float* rec,
                    const float* key, const int* tile_ptr, const int* tile_ent, long long capacity,
                    const float* dLdD, const float* dLdN, const float* g_center, const float* g_quat,
                    const float* g_radii, void* ws, size_t ws_bytes);
ps_status check_fused(const ps_planes* planes, const ps_frame* f, const ps_settings* s, const float* rec,
                      const float* key, const int* tile_ptr, const int* tile_ent, long long capacity,
                      const float* gt_depth, const float* gt_normal, const float* g_radii, void* ws,
                      size_t ws_bytes);

// The parts of a step that ps_fit_step runs with less between them than the entry points do.
// project with `count` leaves the binning's counts as well (diff zeroed before).
ps_status project(const ps_planes* planes, const ps_frame* frame, const ps_settings* s, float* rec, int* rect,
                  float* key, const BinCount* count, int* d_status, cudaStream_t st);
// Where a binning with these arguments keeps its counts.
ps_status bin_count(const ps_frame* frame, long long capacity, void* ws, size_t ws_bytes, BinCount* out);
// counted: the counts are there.
ps_status bin_tiles(const ps_frame* frame, const ps_settings* s, const float* rec, const int* rect,
                    const float* key, int* tile_ptr, int* tile_ent, float* tile_key, long long capacity,
                    long long* d_required, void* ws, size_t ws_bytes, bool counted, int* d_status,
                    cudaStream_t st);
// ps_splat_fused without the chain: the record gradients, the work counter and the partial
// loss sums lie in ws as FusedWs says.  cleared: ws is zeroed (its first `bytes`).
struct FusedWs {
    float* g_rec;
    int* counter;
    double* slots;
    size_t bytes;
};
ps_status fused_ws(const ps_frame* f, const ps_settings* s, void* ws, size_t ws_bytes, FusedWs* out);
ps_status splat_fused(const ps_planes* planes, const ps_frame* f, const ps_settings* s, const float* rec,
                      const float* key, const int* tile_ptr, const int* tile_ent, long long capacity,
                      const float* gt_depth, const float* gt_normal, float* depth, float* normal, float* dL_dD,
                      float* dL_dN, float* g_radii, void* ws, size_t ws_bytes, bool cleared, int* d_status,
                      cudaStream_t st);
// The chain after splat_fused, with the views' loss sums.
ps_status chain_fused(const ps_planes* planes, const ps_frame* f, const ps_settings* s, double* view_sums,
                      float* g_center, float* g_quat, float* g_radii, void* ws, size_t ws_bytes,
                      cudaStream_t st);

// (t, id) lexicographic order of candidates.
__device__ __forceinline__ bool cand_less(float ta, int ia, float tb, int ib)
{
    return ta < tb || (ta == tb && ia < ib);
}

}  // namespace ps
