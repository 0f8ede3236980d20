// ps_init.cu -- nearest-neighbour distances for the initial plane radii.
//
// Sec. 3.1 starts every plane with all four radii equal to half the distance
// from its centre to the nearest other centre.  ps_nn_distance computes that
// distance exactly (the minimum over every other point, in FP32) for all
// points at once.  Up to kBruteMax points every pair is taken (k_nn_brute, one
// launch).  Beyond:
//   1. one CTA finds the bounding box and picks the cell edge of a uniform grid
//      (about one point per cell of the box's volume, thin boxes padded);
//   2. points are counted per hashed cell, every cell gets a run of that length
//      (the runs' order does not matter, so warps reserve them with an atomic),
//      the point ids are scattered into the runs;
//   3. each point's warp searches the cells around its own in shells of growing
//      Chebyshev radius r; a point within distance r * cell of the query lies in a
//      cell at most r away on every axis, so once the nearest point found is
//      within r * cell no unsearched cell can hold a nearer one.  Hash collisions
//      only add real points to a run, which never breaks the minimum.
// Both take the minimum of the same rounded squares, so they agree bit for bit.
#include "ps_internal.cuh"

namespace {

constexpr int kSetupThreads = 1024;
// All pairs up to here: radii of 3,000 centres take 11 us by pairs and 39 us by the grid,
// 8,192 31 and 44 us, 12,000 58 and 46 us (events around the call; from Python the first takes 17).  (One thread per point in the grid, its cells one
// after another, with the cells' runs from a one-CTA scan, took 81, 98 and 132 us.)
constexpr int kBruteMax = 10000;

struct NnHeader {
    float lo[3];
    float cell;
    float inv_cell;
    int r_max;          // shells beyond this radius cover the whole box
    unsigned mask;      // hash table size - 1
    unsigned used;      // points in the runs reserved so far
};

__host__ __device__ inline unsigned table_size(int n)
{
    unsigned t = 1024;
    while (t < 2u * (unsigned)n) t <<= 1;
    return t;
}

__device__ __forceinline__ unsigned cell_hash(int ix, int iy, int iz, unsigned mask)
{
    const unsigned h = ((unsigned)ix * 73856093u) ^ ((unsigned)iy * 19349663u) ^ ((unsigned)iz * 83492791u);
    return h & mask;
}

__device__ __forceinline__ void cell_of(const NnHeader& hd, float x, float y, float z, int& ix, int& iy,
                                        int& iz)
{
    ix = (int)floorf((x - hd.lo[0]) * hd.inv_cell);
    iy = (int)floorf((y - hd.lo[1]) * hd.inv_cell);
    iz = (int)floorf((z - hd.lo[2]) * hd.inv_cell);
}

// One CTA: bounding box, cell edge, shell limit, table mask.
__global__ void __launch_bounds__(kSetupThreads) k_nn_setup(const float* __restrict__ p, int n, NnHeader* hd)
{
    __shared__ float red[6][kSetupThreads / 32];
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float v = p[3 * i + c];
            mn[c] = fminf(mn[c], v);
            mx[c] = fmaxf(mx[c], v);
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        for (int o = 16; o > 0; o >>= 1) {
            mn[c] = fminf(mn[c], __shfl_xor_sync(0xffffffffu, mn[c], o));
            mx[c] = fmaxf(mx[c], __shfl_xor_sync(0xffffffffu, mx[c], o));
        }
        if (lane == 0) { red[c][w] = mn[c]; red[3 + c][w] = mx[c]; }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float lo[3], hi[3];
        for (int c = 0; c < 3; ++c) {
            lo[c] = red[c][0]; hi[c] = red[3 + c][0];
            for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
                lo[c] = fminf(lo[c], red[c][i]);
                hi[c] = fmaxf(hi[c], red[3 + c][i]);
            }
        }
        const float ex = hi[0] - lo[0], ey = hi[1] - lo[1], ez = hi[2] - lo[2];
        const float diag = sqrtf(ex * ex + ey * ey + ez * ez);
        // a flat or thin box (points on a plane or a line) is padded, so the cell
        // edge follows the spacing of the points rather than collapsing to zero
        const float pad = 1e-3f * diag + 1e-6f;
        const double vol = (double)fmaxf(ex, pad) * fmaxf(ey, pad) * fmaxf(ez, pad);
        float cell = (float)cbrt(vol / (double)(n > 0 ? n : 1));
        if (!(cell > 0.f)) cell = 1e-6f;
        for (int c = 0; c < 3; ++c) hd->lo[c] = lo[c];
        hd->cell = cell;
        hd->inv_cell = 1.f / cell;
        const float rm = ceilf(diag / cell) + 1.f;
        hd->r_max = rm < 1e6f ? (int)rm : 1000000;
        hd->mask = table_size(n) - 1;
        hd->used = 0;
    }
}

__global__ void k_nn_count(const float* __restrict__ p, int n, const NnHeader* __restrict__ hd,
                           unsigned* __restrict__ count)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const NnHeader h = *hd;
    int ix, iy, iz;
    cell_of(h, p[3 * i], p[3 * i + 1], p[3 * i + 2], ix, iy, iz);
    atomicAdd(&count[cell_hash(ix, iy, iz, h.mask)], 1u);
}

// Runs: start[t] = cursor[t] = the place of cell t's count[t] points.  A warp reserves
// 32 cells' worth at once.  (An exclusive prefix by one CTA took 7 us for 8,192 cells and
// grew with their number.)
__global__ void __launch_bounds__(256) k_nn_runs(const unsigned* __restrict__ count, NnHeader* hd,
                                                 unsigned* __restrict__ start,
                                                 unsigned* __restrict__ cursor)
{
    const unsigned t = blockIdx.x * 256 + threadIdx.x;      // the table size is a multiple of 256
    const int lane = threadIdx.x & 31;
    const unsigned v = count[t];
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    unsigned base = 0;
    if (lane == 31) base = atomicAdd(&hd->used, x);
    base = __shfl_sync(0xffffffffu, base, 31) + x - v;
    start[t] = base;
    cursor[t] = base;
}

__global__ void k_nn_scatter(const float* __restrict__ p, int n, const NnHeader* __restrict__ hd,
                             unsigned* __restrict__ cursor, int* __restrict__ sorted)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const NnHeader h = *hd;
    int ix, iy, iz;
    cell_of(h, p[3 * i], p[3 * i + 1], p[3 * i + 2], ix, iy, iz);
    const unsigned slot = atomicAdd(&cursor[cell_hash(ix, iy, iz, h.mask)], 1u);
    sorted[slot] = i;
}

__device__ __forceinline__ void nn_store(int i, float best, float* __restrict__ dist,
                                         float* __restrict__ radii, float scale, float r_lo, float r_hi)
{
    const float d = sqrtf(best);
    if (dist) dist[i] = d;
    if (radii) {
        // Sec. 3.1: all four radii start at scale x the nearest-centre distance
        const float r = fminf(fmaxf(scale * d, r_lo), r_hi);
        reinterpret_cast<float4*>(radii)[i] = make_float4(r, r, r, r);
    }
}

// Cell c of the shell of Chebyshev radius r (the whole cube for r = 1): the two faces
// dz = -r, r, then the ring of 8 r cells of every dz between them.
template <typename I>
__device__ __forceinline__ int3 shell_cell(I c, I r)
{
    if (r == 1) return make_int3((int)(c % 3) - 1, (int)(c / 3 % 3) - 1, (int)(c / 9) - 1);
    const I w = 2 * r + 1;
    if (c < 2 * w * w) {
        const I k = c % (w * w);
        return make_int3((int)(k % w - r), (int)(k / w - r), (int)(c < w * w ? -r : r));
    }
    c -= 2 * w * w;
    const I k = c % (8 * r), s = k / (2 * r), o = k % (2 * r);
    const I x = s == 0 ? o - r : (s == 1 ? r : (s == 2 ? r - o : -r));
    const I y = s == 0 ? -r : (s == 1 ? o - r : (s == 2 ? r : r - o));
    return make_int3((int)x, (int)y, (int)(c / (8 * r) - r + 1));
}

// One warp per point: the lanes share a shell's cells, so the chain of dependent loads
// (run, id, point) is walked once per shell instead of once per cell.
__global__ void __launch_bounds__(256) k_nn_query(const float* __restrict__ p, int n,
                                                  const NnHeader* __restrict__ hd,
                                                  const unsigned* __restrict__ start,
                                                  const unsigned* __restrict__ count,
                                                  const int* __restrict__ sorted,
                                                  float* __restrict__ dist, float* __restrict__ radii,
                                                  float scale, float r_lo, float r_hi)
{
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= n) return;
    const int lane = threadIdx.x & 31;
    const NnHeader h = *hd;
    const float x = p[3 * i], y = p[3 * i + 1], z = p[3 * i + 2];
    int cx, cy, cz;
    cell_of(h, x, y, z, cx, cy, cz);
    float best = INFINITY;       // squared distance
    for (int r = 1; r <= h.r_max; ++r) {
        const long long w = 2LL * r + 1;
        // (r_max is at most 10^6: a shell's cells are counted in 64 bits)
        const long long cells = r == 1 ? 27 : 2 * w * w + 8LL * r * (2 * r - 1);
        for (long long c = lane; c < cells; c += 32) {
            const int3 d = cells < (1LL << 31) ? shell_cell((int)c, r) : shell_cell(c, (long long)r);
            const unsigned t = cell_hash(cx + d.x, cy + d.y, cz + d.z, h.mask);
            const unsigned b = __ldg(&start[t]), e = b + __ldg(&count[t]);
            for (unsigned s = b; s < e; ++s) {
                const int j = __ldg(&sorted[s]);
                if (j == i) continue;
                const float ax = __ldg(&p[3 * j]) - x, ay = __ldg(&p[3 * j + 1]) - y,
                            az = __ldg(&p[3 * j + 2]) - z;
                const float d2 = fmaf(ax, ax, fmaf(ay, ay, az * az));
                best = fminf(best, d2);
            }
        }
        // squares are not negative: their bits order like their values
        best = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(best)));
        // (0.999: the cell coordinates are rounded FP32 products, so keep a margin)
        const float reach = (float)r * h.cell * 0.999f;
        if (best <= reach * reach) break;
    }
    if (lane == 0) nn_store(i, best, dist, radii, scale, r_lo, r_hi);
}

// Every pair, bound by the FP32 pipe: a CTA takes 8 queries, two per thread in the halves of packed FP32 pairs
// (add, multiply and fma of two pairs per instruction, each rounded as its scalar form),
// and 64 streams of points (8 groups of 4 threads in each of 8 warps) out of chunks in
// shared memory.
constexpr int kBruteQ = 8;
constexpr int kBruteChunk = 1024;

__device__ __forceinline__ unsigned long long pack2(float a, float b)
{
    return ((unsigned long long)__float_as_uint(b) << 32) | __float_as_uint(a);
}

__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b,
                                                   unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__global__ void __launch_bounds__(256) k_nn_brute(const float* __restrict__ p, int n,
                                                  float* __restrict__ dist, float* __restrict__ radii,
                                                  float scale, float r_lo, float r_hi)
{
    __shared__ float4 s_p[kBruteChunk];
    __shared__ float s_best[8][kBruteQ];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int q0 = blockIdx.x * kBruteQ;
    const int ia = q0 + 2 * (lane & 3), ib = ia + 1;         // this thread's queries
    const int ca = min(ia, n - 1), cb = min(ib, n - 1);
    // ax = p_j - p_i = p_j + (-p_i)
    const unsigned long long nx = pack2(-p[3 * ca], -p[3 * cb]);
    const unsigned long long ny = pack2(-p[3 * ca + 1], -p[3 * cb + 1]);
    const unsigned long long nz = pack2(-p[3 * ca + 2], -p[3 * cb + 2]);
    float ba = INFINITY, bb = INFINITY;
    for (int base = 0; base < n; base += kBruteChunk) {
        const int m = min(kBruteChunk, n - base);
        __syncthreads();
        for (int j = tid; j < m; j += 256) {
            const float* q = p + 3 * (size_t)(base + j);
            s_p[j] = make_float4(__ldg(q), __ldg(q + 1), __ldg(q + 2), 0.f);
        }
        __syncthreads();
        const bool own = base < q0 + kBruteQ && base + m > q0;   // the chunk holds the queries
#pragma unroll 4
        for (int j = w * 8 + (lane >> 2); j < m; j += 64) {
            const float4 v = s_p[j];
            const unsigned long long ax = add2(pack2(v.x, v.x), nx), ay = add2(pack2(v.y, v.y), ny),
                                     az = add2(pack2(v.z, v.z), nz);
            const unsigned long long d2 = fma2(ax, ax, fma2(ay, ay, mul2(az, az)));
            float da = __uint_as_float((unsigned)d2), db = __uint_as_float((unsigned)(d2 >> 32));
            if (own) {
                if (base + j == ia) da = INFINITY;
                if (base + j == ib) db = INFINITY;
            }
            ba = fminf(ba, da);
            bb = fminf(bb, db);
        }
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        ba = fminf(ba, __shfl_xor_sync(0xffffffffu, ba, o));
        bb = fminf(bb, __shfl_xor_sync(0xffffffffu, bb, o));
    }
    if (lane < 4) { s_best[w][2 * lane] = ba; s_best[w][2 * lane + 1] = bb; }
    __syncthreads();
    if (tid < kBruteQ && q0 + tid < n) {
        float best = s_best[0][tid];
#pragma unroll
        for (int k = 1; k < 8; ++k) best = fminf(best, s_best[k][tid]);
        nn_store(q0 + tid, best, dist, radii, scale, r_lo, r_hi);
    }
}

size_t nn_ws_bytes(int n)
{
    const size_t T = table_size(n);
    // header, counts [T], starts [T + 1], cursors [T], sorted ids [n]
    return 64 + sizeof(unsigned) * (3 * T + 1) + sizeof(int) * (size_t)n + 64;
}

}  // namespace

extern "C" size_t ps_nn_workspace_bytes(int n)
{
    if (n < 0) return 0;
    return nn_ws_bytes(n);
}

extern "C" ps_status ps_nn_distance(const float* points, int n, float scale, float r_lo, float r_hi,
                                    float* dist, float* radii, void* ws, size_t ws_bytes,
                                    ps_stream stream)
{
    if (n < 0) return PS_ERR_ARG;
    if (n == 0) return PS_OK;
    if (!points || (!dist && !radii) || !ws) return PS_ERR_ARG;
    if (radii && ((reinterpret_cast<uintptr_t>(radii) & 15) || !(scale >= 0.f) || !(r_lo <= r_hi)))
        return PS_ERR_ARG;
    if (ws_bytes < nn_ws_bytes(n) || (reinterpret_cast<uintptr_t>(ws) & 15)) return PS_ERR_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (n <= kBruteMax) {
        k_nn_brute<<<(n + kBruteQ - 1) / kBruteQ, 256, 0, st>>>(points, n, dist, radii, scale, r_lo, r_hi);
        PS_LAUNCH_CHECK();
        return PS_OK;
    }
    const unsigned T = table_size(n);
    char* base = static_cast<char*>(ws);
    NnHeader* hd = reinterpret_cast<NnHeader*>(base);
    unsigned* count = reinterpret_cast<unsigned*>(base + 64);
    unsigned* start = count + T;
    unsigned* cursor = start + T + 1;
    int* sorted = reinterpret_cast<int*>(cursor + T);
    PS_CUDA_CHECK(cudaMemsetAsync(count, 0, sizeof(unsigned) * T, st));
    k_nn_setup<<<1, kSetupThreads, 0, st>>>(points, n, hd);
    PS_LAUNCH_CHECK();
    const int blocks = (n + 255) / 256;
    k_nn_count<<<blocks, 256, 0, st>>>(points, n, hd, count);
    PS_LAUNCH_CHECK();
    k_nn_runs<<<T / 256, 256, 0, st>>>(count, hd, start, cursor);
    PS_LAUNCH_CHECK();
    k_nn_scatter<<<blocks, 256, 0, st>>>(points, n, hd, cursor, sorted);
    PS_LAUNCH_CHECK();
    k_nn_query<<<(n + 7) / 8, 256, 0, st>>>(points, n, hd, start, count, sorted, dist, radii, scale,
                                            r_lo, r_hi);
    PS_LAUNCH_CHECK();
    return PS_OK;
}
