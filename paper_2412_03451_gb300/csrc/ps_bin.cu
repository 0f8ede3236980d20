// ps_bin.cu -- per-tile lists of records, sorted near to far.
//
// Sec. 3.2 ("Blending Composition") sorts the intersections of a ray near to
// far.  The renderer gets there in two stages: here every tile receives the
// records whose screen rectangle covers it, each with a depth key that bounds
// from below every depth the plane can produce in that tile, sorted by it;
// the splat kernels then merge per pixel by exact depth.  Keys are unique per
// list as (key bits, record id), so the output does not depend on the order in
// which the atomics below land.
//
// Entry key (bit-exact specification, FP32 with correctly rounded + - * /
// only, no contraction): the rays of the pixel centres at the tile's four
// corner pixels, d = ((x + 0.5 - cx) / fx, (y + 0.5 - cy) / fy, 1); per ray
// den = (n_x d_x + n_y d_y) + n_z and t = s / den with the record's f32 n_c and
// s = n_c . p_c.  Over the tile the depth s / (d . n_c) of the plane is
// linear-fractional in the ray, so if den has one sign at all four corners (and
// |den| > 0.01 (|n_x d_x| + |n_y d_y| + |n_z|) at each, which keeps FP32
// cancellation small) its range over the tile is spanned by the corners:
// c = max(min t, z_near), or +inf if max t <= z_near (no depth in range);
// otherwise c = z_near.  The entry key is max(c, the record's key), both lower
// bounds of every depth the plane produces in the tile.  Unlike the record key
// alone (the smallest z of the whole widened quad), this bound is as tight as
// the tile: entries of large or oblique planes no longer all sort to the front
// of every list.
//
//   1. record counts: tiles covered by each record's rectangle (+ the record's
//      first global tile and rectangle width), then an exclusive scan over
//      records numbers every (record, tile) pair.  The same thread marks its
//      rectangle in a difference array over the flat (view-major, row-major)
//      tile index: +1 where each row segment starts, -1 one past its end (the
//      whole rectangle is one segment when it spans the full width);
//   2. scans: tile_ptr is the exclusive prefix of the inclusive prefix of the
//      difference array (the number of records covering each tile), total ->
//      d_required; two launches serve both scans (k_scan_sums, k_scan_apply);
//   3. scatter: one thread per pair writes its entry key and record id into a
//      slot of its tile (unordered, via per-tile cursors);
//   4. sort: each tile's slots by (key, record id), k_sort: a warp sorts lists of
//      up to kWarpSortCap entries in registers, four lists of up to 8 or two of up
//      to 16 at a time; a block sorts the longer ones it meets together (bitonic up
//      to kSortCap entries, an O(n^2) rank sort beyond).
// Every pair gets its own thread, so a plane covering a thousand tiles costs
// no more latency than one covering a single tile.
#include "ps_internal.cuh"

using namespace ps;

namespace {

constexpr int kSortCap = 4096;     // entries sorted in shared memory by a CTA (32 KB of u64)
constexpr int kWarpSortCap = 256;  // entries sorted by one warp, in registers (8 per lane)
constexpr int kSortWarps = 8;
constexpr int kSortTiles = 4;      // consecutive tiles per warp
constexpr int kScanThreads = 256;
constexpr int kScanItems = 9;      // elements per thread per scan tile (odd: a thread's run
                                   // starts 9 words after its neighbour's, no bank conflicts)
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr int kFlatBlocks = 152 * 8;
constexpr int kPairBlock = 256;       // pairs per scatter block = pairs per chunk of the chunk table
// The pair numbering is clamped here.  A total that reaches it exceeds every capacity; the pairs
// past it have no number, so nothing is scattered and the sort fills the truncated lists.
constexpr int kMaxPairs = 0x7fffffff;

inline long long n_chunks(long long capacity) { return capacity / kPairBlock + 2; }

struct BinWs {
    int* rec_cnt;       // [R + 1] tiles per record -> exclusive prefix (pair numbering)
    int4* rec_info;     // [R] first global tile, rectangle width in tiles, tiles_x, view
    int* tile_cnt;      // [n_tiles] difference array of the tile counts
    int* cursor;        // [n_tiles]
    int* chunk_first;   // [n_chunks] record holding pair c * kPairBlock
    longlong2* part;    // [scan tiles of records + of tiles] scan partial sums
    unsigned long long* ent_tmp;    // [capacity] unordered entries, (key bits, record id)
};

inline size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

inline int scan_tiles(long long n) { return (int)((n + kScanTile - 1) / kScanTile); }

inline BinWs carve(void* ws, int R, int n_tiles, long long capacity, size_t* bytes)
{
    char* p = static_cast<char*>(ws);
    size_t o = 0;
    auto take = [&](size_t n) { char* r = p + o; o += align_up(n); return r; };
    BinWs w;
    w.rec_cnt = reinterpret_cast<int*>(take(sizeof(int) * (size_t)(R + 1)));
    w.rec_info = reinterpret_cast<int4*>(take(sizeof(int4) * (size_t)(R > 0 ? R : 1)));
    w.tile_cnt = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n_tiles));
    w.cursor = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n_tiles));
    w.chunk_first = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n_chunks(capacity)));
    w.part = reinterpret_cast<longlong2*>(take(sizeof(longlong2) * (size_t)(scan_tiles(R) + scan_tiles(n_tiles))));
    w.ent_tmp = reinterpret_cast<unsigned long long*>(
        take(sizeof(unsigned long long) * (size_t)(capacity > 0 ? capacity : 1)));
    if (bytes) *bytes = o;
    return w;
}

inline size_t ws_bytes(int R, int n_tiles, long long capacity)
{
    size_t n;
    carve(nullptr, R, n_tiles, capacity, &n);
    return n;
}

// 1. record counts ---------------------------------------------------------------
__global__ void __launch_bounds__(128) k_rec_count(const int4* __restrict__ rect,
                                                   const ps_view* __restrict__ views, BinCount count)
{
    const int v = blockIdx.y;
    const ps_view* vw = views + v;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= __ldg(&vw->K)) return;
    const size_t r = (size_t)__ldg(&vw->rec_off) + k;
    count_record(count, r, __ldg(&rect[r]), __ldg(&vw->tile_off), __ldg(&vw->tiles_x), v);
}

// 2. scans ------------------------------------------------------------------------
// Exclusive prefixes of int arrays of any length, in tiles of kScanTile elements, in two
// launches that serve two jobs at once (the pair numbering and the tile offsets): the
// first sums every tile, the second adds the sums of the tiles before its own and scans.
// With `twice` the array is first replaced by its inclusive prefix (a difference array
// becomes the counts).  An element x at place j of a tile of m then adds x to the counts
// and x (m - j) to the tile's sum of counts, so both of a tile's sums (D, S) come without
// a scan, and the prefix before tile b is sum D_r for the counts and
// sum S_r + kScanTile (b - 1 - r) D_r for their sum.  Bound by latency:
// 38,400 tiles and 24,000 records take 2.0 + 3.2 us (a launch of two 8-CTA clusters, one
// per array, took 7.1 us), 307,200 and 640,000 2.8 + 5.7 us (three launches per pass over an
// array and one for the chunk table took 43 us).
struct ScanJob {
    const int* in;
    int n;
    int* out;             // [n + 1] exclusive prefix clamped to capacity, out[n] = total
    int* cursor;          // optional copy of out[0 .. n)
    long long capacity;
    long long* d_total;   // optional
    int* status;          // optional: PS_ERR_CAPACITY when the total exceeds capacity
    int twice;
    int* chunk_first;     // optional chunk table [n_chunk]: the record holding pair c * kPairBlock
    long long n_chunk;
    longlong2* part;      // [scan tiles]
    int blocks;           // scan tiles
};

// The block's totals of x and y (in every thread).
__device__ __forceinline__ void block_sum2(long long& x, long long& y, longlong2* s_warp)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = make_longlong2(x, y);
    __syncthreads();
    x = 0; y = 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) { x += s_warp[w].x; y += s_warp[w].y; }
    __syncthreads();
}

// Exclusive prefix of x over the block's threads.
template <typename T>
__device__ __forceinline__ T block_scan_excl(T x, T* s_warp)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    T before = 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) before += w < wid ? s_warp[w] : 0;
    __syncthreads();
    return before + incl - x;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(ScanJob j0, ScanJob j1)
{
    __shared__ longlong2 s_warp[kScanThreads / 32];
    after_previous();
    const bool second = (int)blockIdx.x >= j0.blocks;
    const ScanJob& a = second ? j1 : j0;
    const int b = (int)blockIdx.x - (second ? j0.blocks : 0);
    const int lo = b * kScanTile, m = min(kScanTile, a.n - lo);
    long long D = 0, S = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int j = i * kScanThreads + threadIdx.x;
        const int x = j < m ? a.in[lo + j] : 0;
        D += x;
        S += (long long)x * (m - j);
    }
    block_sum2(D, S, s_warp);
    if (threadIdx.x == 0) a.part[b] = make_longlong2(D, S);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(ScanJob j0, ScanJob j1)
{
    __shared__ int s_x[kScanTile];
    __shared__ longlong2 s_pair[kScanThreads / 32];
    __shared__ long long s_wide[kScanThreads / 32];
    __shared__ int s_int[kScanThreads / 32];
    after_previous();
    const bool second = (int)blockIdx.x >= j0.blocks;
    const ScanJob& a = second ? j1 : j0;
    const int b = (int)blockIdx.x - (second ? j0.blocks : 0);
    const int lo = b * kScanTile, m = min(kScanTile, a.n - lo);
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int j = i * kScanThreads + threadIdx.x;
        s_x[j] = j < m ? a.in[lo + j] : 0;       // (in and out may be the same array)
    }
    // carries from the tiles before: the counts' prefix cD and the offset cC
    long long cD = 0, cC = 0;
    for (int r = threadIdx.x; r < b; r += kScanThreads) {
        const longlong2 t = a.part[r];
        cD += t.x;
        cC += a.twice ? t.y + (long long)kScanTile * (b - 1 - r) * t.x : t.x;
    }
    block_sum2(cD, cC, s_pair);                  // (its barriers also cover s_x)
    int x[kScanItems];
    const int t0 = threadIdx.x * kScanItems;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) x[i] = s_x[t0 + i];
    if (a.twice) {
        int run = 0;
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) run += x[i];
        int c = (int)cD + block_scan_excl(run, s_int);
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            c += x[i];
            x[i] = t0 + i < m ? c : 0;
        }
    }
    long long sum = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) sum += x[i];
    long long v = cC + block_scan_excl(sum, s_wide);
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int at = (int)(v < a.capacity ? v : a.capacity);
        s_x[t0 + i] = at;
        v += x[i];
        if (a.chunk_first && t0 + i < m) {
            const long long hi = v < a.capacity ? v : a.capacity;
            for (long long c = ((long long)at + kPairBlock - 1) / kPairBlock;
                 c < a.n_chunk && c * kPairBlock < hi; ++c)
                a.chunk_first[c] = lo + t0 + i;
        }
    }
    if (b == a.blocks - 1 && threadIdx.x == kScanThreads - 1) {      // v: the total
        a.out[a.n] = (int)(v < a.capacity ? v : a.capacity);
        if (a.d_total) *a.d_total = v;
        if (a.status && v > a.capacity) set_status(a.status, PS_ERR_CAPACITY);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int j = i * kScanThreads + threadIdx.x;
        if (j < m) {
            a.out[lo + j] = s_x[j];
            if (a.cursor) a.cursor[lo + j] = s_x[j];
        }
    }
}

// 3. one thread per (record, tile) pair ----------------------------------------
__device__ __forceinline__ int pair_record(const int* off, int lo, int hi, int i)
{
    // last r in [lo, hi] with off[r] <= i (off is non-decreasing, off[lo] <= i)
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Pairs base .. base + kPairBlock - 1 of a block belong to records x .. y of the
// result: the chunk table gives the records holding this chunk's first pair and
// the next chunk's (an upper bound); beyond the table the whole record range is
// searched.  Every thread of the block computes the same two values (broadcast
// loads, no barrier) and then searches only that narrow range for its own pair.
__device__ __forceinline__ int2 chunk_record_range(const int* off, int R, int E, int base,
                                                   const int* chunk_first, long long n_chunk)
{
    const long long c = base / kPairBlock;
    const int lo = (c < n_chunk && c * kPairBlock < E) ? chunk_first[c]
                                                       : pair_record(off, 0, R - 1, base);
    const int hi = (c + 1 < n_chunk && (c + 1) * kPairBlock < E)
                       ? chunk_first[c + 1]
                       : pair_record(off, 0, R - 1, min(base + kPairBlock, E) - 1);
    return make_int2(lo, hi);
}

// The entry key of the specification above.
__device__ __forceinline__ float entry_key(float4 ns, const ps_view* __restrict__ vw, int tx, int ty,
                                           int tw, int th, float z_near)
{
    const float fx = __ldg(&vw->fx), fy = __ldg(&vw->fy), cx = __ldg(&vw->cx), cy = __ldg(&vw->cy);
    const float xs[2] = {(float)(tx * tw), (float)(tx * tw + tw - 1)};
    const float ys[2] = {(float)(ty * th), (float)(ty * th + th - 1)};
    int npos = 0, nneg = 0;
    bool weak = false;
    // the corners' den of largest and of smallest magnitude
    float dbig = 0.f, dsmall = INFINITY;
    const float dys[2] = {__fdiv_rn(__fsub_rn(__fadd_rn(ys[0], 0.5f), cy), fy),
                          __fdiv_rn(__fsub_rn(__fadd_rn(ys[1], 0.5f), cy), fy)};
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const float dx = __fdiv_rn(__fsub_rn(__fadd_rn(xs[a], 0.5f), cx), fx);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const float dy = dys[b];
            const float p1 = __fmul_rn(ns.x, dx), p2 = __fmul_rn(ns.y, dy);
            const float den = __fadd_rn(__fadd_rn(p1, p2), ns.z);
            const float mag = __fadd_rn(__fadd_rn(fabsf(p1), fabsf(p2)), fabsf(ns.z));
            if (!(fabsf(den) > __fmul_rn(0.01f, mag))) weak = true;
            npos += den > 0.f;
            nneg += den < 0.f;
            if (fabsf(den) > fabsf(dbig)) dbig = den;
            if (fabsf(den) < fabsf(dsmall)) dsmall = den;
        }
    }
    if (weak || (npos != 4 && nneg != 4)) return z_near;
    // With one sign of den at the four corners, t = s / den has one sign and its
    // magnitude falls as |den| grows; correctly rounded division is monotone and
    // odd, so the extremes of the four rounded quotients are the quotients by the
    // extreme dens: the same bits as taking all four.
    const float ta = __fdiv_rn(ns.w, dbig), tb = __fdiv_rn(ns.w, dsmall);
    const float tmin = fminf(ta, tb), tmax = fmaxf(ta, tb);
    if (!(tmax > z_near)) return INFINITY;
    return fmaxf(tmin, z_near);
}

__global__ void __launch_bounds__(kPairBlock) k_pair_scatter(const int* rec_off, int R, const int4* rec_info,
                                                             const int* tile_ptr, int* cursor,
                                                             unsigned long long* ent_tmp,
                                                             const float4* rec, const float* rec_key,
                                                             const ps_view* __restrict__ views,
                                                             int tw, int th, float z_near,
                                                             const int* chunk_first, long long n_chunk)
{
    after_previous();
    const int E = rec_off[R];
    if (E == kMaxPairs) return;
    // (unsigned: the step past the last block may pass the int range)
    for (unsigned base = blockIdx.x * kPairBlock; base < (unsigned)E; base += gridDim.x * kPairBlock) {
        const int2 rg = chunk_record_range(rec_off, R, E, (int)base, chunk_first, n_chunk);
        if (base + threadIdx.x < (unsigned)E) {
            const int i = (int)(base + threadIdx.x);
            const int r = pair_record(rec_off, rg.x, rg.y, i);
            const int4 info = rec_info[r];
            const int j = i - rec_off[r];
            const int t = info.x + (j / info.y) * info.z + (j % info.y);
            // the key first, so that the slot atomic's latency overlaps nothing it waits on
            const ps_view* vw = views + info.w;
            const int lt = t - __ldg(&vw->tile_off);
            const float k = fmaxf(entry_key(rec[4 * (size_t)r], vw, lt % info.z, lt / info.z, tw, th, z_near),
                                  rec_key[r]);
            const int lim = tile_ptr[t + 1];
            const int pos = atomicAdd(&cursor[t], 1);
            // tile_ptr is clamped to the capacity: positions past it belong to lists
            // that did not fit and are dropped (the status word says so)
            // (keys are positive or +inf, so their bits sort like the values)
            // (unsigned: a cursor may count past the int range)
            if ((unsigned)pos < (unsigned)lim) ent_tmp[pos] = ((unsigned long long)__float_as_uint(k) << 32) | (unsigned)r;
        }
    }
}

// 4. sort -----------------------------------------------------------------------
__device__ __forceinline__ void put(int* __restrict__ tile_ent, float* __restrict__ tile_key, int j,
                                    unsigned long long v)
{
    tile_ent[j] = (int)(unsigned)(v & 0xffffffffu);
    tile_key[j] = __uint_as_float((unsigned)(v >> 32));
}

// One step of a sorting network across lanes: the smaller of the pair goes to the lane
// with `lower` set if asc, to the other if not.
__device__ __forceinline__ unsigned long long cas(unsigned long long v, int mask, bool lower, bool asc)
{
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, v, mask);
    return ((v < o) == (lower == asc)) ? v : o;
}

// Bitonic network over E groups of W keys, key e * W + lane % W in v[e], sorting the
// 32 / W lists of a warp at once (E > 1 only for W = 32).  A merge of two ascending runs
// starts with the mirrored partner, so every run of up to 16 keys is ascending and a step
// needs one fixed predicate per lane; runs of 32 alternate in direction with e, which is
// known at compile time.
template <int W, int E>
__device__ __forceinline__ void warp_bitonic(unsigned long long (&v)[E], int lane)
{
#pragma unroll
    for (int k = 2; k <= W; k <<= 1) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const bool asc = k < 32 || E == 1 || (e & 1) == 0;
            v[e] = cas(v[e], k - 1, (lane & (k >> 1)) == 0, asc);
#pragma unroll
            for (int j = k >> 2; j > 0; j >>= 1) v[e] = cas(v[e], j, (lane & j) == 0, asc);
        }
    }
#pragma unroll
    for (int k = 2; k <= E; k <<= 1) {            // runs of 32 k keys
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if ((e & j) == 0) {
                    const bool asc = k == E || (e & k) == 0;
                    const unsigned long long a = v[e], b = v[e + j];
                    const bool sw = (a > b) == asc;
                    v[e] = sw ? b : a;
                    v[e + j] = sw ? a : b;
                }
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const bool asc = k == E || (e & k) == 0;
#pragma unroll
            for (int j = 16; j > 0; j >>= 1) v[e] = cas(v[e], j, (lane & j) == 0, asc);
        }
    }
}

// Sorts the list of n slots from b (W = 32: the warp's one list; else this lane's group's).
template <int W, int E>
__device__ __forceinline__ void warp_sort_list(const unsigned long long* ent_tmp,
                                               int* __restrict__ tile_ent, float* __restrict__ tile_key,
                                               int b, int n, int lane)
{
    unsigned long long v[E];
    const int i = lane & (W - 1);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = e * W + i < n ? ent_tmp[b + e * W + i] : ~0ull;
    warp_bitonic<W, E>(v, lane);
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (e * W + i < n) put(tile_ent, tile_key, b + e * W + i, v[e]);
}

__device__ void sort_long_list(const unsigned long long* ent_tmp,
                               int* __restrict__ tile_ent, float* __restrict__ tile_key, int b, int n,
                               unsigned long long* s)
{
    const int tid = threadIdx.x, NT = blockDim.x;
    if (n <= kSortCap) {
        int N = 2;
        while (N < n) N <<= 1;
        for (int i = tid; i < N; i += NT) s[i] = i < n ? ent_tmp[b + i] : ~0ull;
        __syncthreads();
        for (int k = 2; k <= N; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = tid; i < N; i += NT) {
                    const int ixj = i ^ j;
                    if (ixj > i) {
                        const unsigned long long x = s[i], y = s[ixj];
                        const bool up = (i & k) == 0;
                        if ((x > y) == up) { s[i] = y; s[ixj] = x; }
                    }
                }
                __syncthreads();
            }
        }
        for (int i = tid; i < n; i += NT) put(tile_ent, tile_key, b + i, s[i]);
        __syncthreads();    // the block's next list reuses s
        return;
    }
    // rank of each element = number of smaller keys (keys are unique)
    for (int i0 = 0; i0 < n; i0 += NT) {
        const int i = i0 + tid;
        const unsigned long long ki = i < n ? ent_tmp[b + i] : 0ull;
        int rank = 0;
        for (int c0 = 0; c0 < n; c0 += kSortCap) {
            const int cn = min(kSortCap, n - c0);
            __syncthreads();
            for (int j = tid; j < cn; j += NT) s[j] = ent_tmp[b + c0 + j];
            __syncthreads();
            if (i < n)
                for (int j = 0; j < cn; ++j) rank += s[j] < ki;
        }
        if (i < n) put(tile_ent, tile_key, b + rank, ki);
    }
    __syncthreads();    // the block's next list reuses s
}

// Bound by instruction issue, so short lists share a warp: at lambda 300 the lists of 3,000
// planes in 8 views of 640x480 take 5.2 us (one list per warp and a second launch for the
// long ones: 13.5 us), those of 16 uneven rooms 31 us (96 us), of 10,000 planes in 64 views
// at lambda 20 118 us (169 us).
__global__ void __launch_bounds__(kSortWarps * 32) k_sort(const int* tile_ptr, int n_tiles,
                                                          const int* pairs,
                                                          const unsigned long long* ent_tmp,
                                                          int* __restrict__ tile_ent,
                                                          float* __restrict__ tile_key)
{
    __shared__ unsigned long long s[kSortCap];
    __shared__ int s_list[kSortWarps * kSortTiles];
    __shared__ int s_cnt;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) s_cnt = 0;
    after_previous();
    __syncthreads();
    if (*pairs == kMaxPairs) {
        // nothing was scattered: every entry is record 0, behind every depth
        const int t = blockIdx.x * kSortWarps * kSortTiles;
        const int e = tile_ptr[min(t + kSortWarps * kSortTiles, n_tiles)];
        for (int j = tile_ptr[t] + (int)threadIdx.x; j < e; j += kSortWarps * 32)
            put(tile_ent, tile_key, j, (unsigned long long)__float_as_uint(INFINITY) << 32);
        return;
    }
    const int t0 = (blockIdx.x * kSortWarps + w) * kSortTiles;
    // lane l < kSortTiles + 1: the start of tile t0 + l's list (past the last tile: its end)
    const int ptr = tile_ptr[min(t0 + min(lane, kSortTiles), n_tiles)];
    const int len = __shfl_down_sync(0xffffffffu, ptr, 1) - ptr;      // lanes < kSortTiles
    const int n4[kSortTiles] = {__shfl_sync(0xffffffffu, len, 0), __shfl_sync(0xffffffffu, len, 1),
                                __shfl_sync(0xffffffffu, len, 2), __shfl_sync(0xffffffffu, len, 3)};
    if (max(max(n4[0], n4[1]), max(n4[2], n4[3])) <= 8) {
        const int q = lane >> 3;
        const int b = __shfl_sync(0xffffffffu, ptr, q), n = __shfl_sync(0xffffffffu, len, q);
        warp_sort_list<8, 1>(ent_tmp, tile_ent, tile_key, b, n, lane);
    } else {
#pragma unroll 1
        for (int p = 0; p < kSortTiles; p += 2) {
            const int na = __shfl_sync(0xffffffffu, len, p), nb = __shfl_sync(0xffffffffu, len, p + 1);
            if (max(na, nb) <= 16) {
                const int q = p + (lane >> 4);
                const int b = __shfl_sync(0xffffffffu, ptr, q), n = __shfl_sync(0xffffffffu, len, q);
                warp_sort_list<16, 1>(ent_tmp, tile_ent, tile_key, b, n, lane);
                continue;
            }
#pragma unroll 1
            for (int q = p; q < p + 2; ++q) {
                const int b = __shfl_sync(0xffffffffu, ptr, q), n = __shfl_sync(0xffffffffu, len, q);
                if (n <= 0) continue;
                if (n <= 32) warp_sort_list<32, 1>(ent_tmp, tile_ent, tile_key, b, n, lane);
                else if (n <= 64) warp_sort_list<32, 2>(ent_tmp, tile_ent, tile_key, b, n, lane);
                else if (n <= 128) warp_sort_list<32, 4>(ent_tmp, tile_ent, tile_key, b, n, lane);
                else if (n <= kWarpSortCap) warp_sort_list<32, 8>(ent_tmp, tile_ent, tile_key, b, n, lane);
                else if (lane == 0) s_list[atomicAdd(&s_cnt, 1)] = t0 + q;
            }
        }
    }
    __syncthreads();
    const int cnt = s_cnt;
    for (int q = 0; q < cnt; ++q) {
        const int t = s_list[q];
        const int b = tile_ptr[t];
        sort_long_list(ent_tmp, tile_ent, tile_key, b, tile_ptr[t + 1] - b, s);
    }
}

}  // namespace

extern "C" size_t ps_bin_workspace_bytes(const ps_frame* frame, long long capacity)
{
    if (!frame || frame->n_tiles < 0 || frame->n_records < 0 || capacity < 0) return 0;
    return ws_bytes(frame->n_records, frame->n_tiles, capacity);
}

ps_status ps::bin_count(const ps_frame* frame, long long capacity, void* ws, size_t ws_bytes_, BinCount* out)
{
    if (!frame || !ws || frame->n_tiles <= 0 || frame->n_records < 0) return PS_ERR_ARG;
    if (capacity < 0 || capacity >= (1LL << 31) - 1) return PS_ERR_ARG;
    if (ws_bytes_ < ws_bytes(frame->n_records, frame->n_tiles, capacity)) return PS_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(ws) & 255) return PS_ERR_ARG;
    const BinWs w = carve(ws, frame->n_records, frame->n_tiles, capacity, nullptr);
    *out = BinCount{w.rec_cnt, w.rec_info, w.tile_cnt, frame->n_tiles};
    return PS_OK;
}

ps_status ps::check_bin(const ps_frame* frame, const ps_settings* s, const float* rec, const int* rect,
                        const float* key, const int* tile_ptr, const int* tile_ent, const float* tile_key,
                        long long capacity, const long long* d_required, void* ws, size_t ws_bytes_)
{
    if (!frame || !s || !rec || !rect || !key || !tile_ptr || !d_required || !ws || !frame->views)
        return PS_ERR_ARG;
    if (capacity > 0 && (!tile_ent || !tile_key)) return PS_ERR_ARG;
    if (s->tile_w <= 0 || s->tile_h <= 0 || !(s->z_near > 0.f)) return PS_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(rec) & 15) return PS_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(rect) & 15) return PS_ERR_ARG;
    BinCount cnt;
    return bin_count(frame, capacity, ws, ws_bytes_, &cnt);
}

ps_status ps::bin_tiles(const ps_frame* frame, const ps_settings* s, const float* rec, const int* rect,
                        const float* key, int* tile_ptr, int* tile_ent, float* tile_key, long long capacity,
                        long long* d_required, void* ws, size_t ws_bytes_, bool counted, int* d_status,
                        cudaStream_t st)
{
    const ps_status e = check_bin(frame, s, rec, rect, key, tile_ptr, tile_ent, tile_key, capacity, d_required,
                                  ws, ws_bytes_);
    if (e != PS_OK) return e;
    BinCount cnt;
    bin_count(frame, capacity, ws, ws_bytes_, &cnt);
    const int R = frame->n_records;
    BinWs w = carve(ws, R, frame->n_tiles, capacity, nullptr);
    const long long nch = n_chunks(capacity);
    if (!counted) {
        PS_CUDA_CHECK(cudaMemsetAsync(w.tile_cnt, 0, sizeof(int) * (size_t)frame->n_tiles, st));
        if (R > 0) {
            dim3 grid((frame->max_K + 127) / 128, frame->n_views);
            k_rec_count<<<grid, 128, 0, st>>>(reinterpret_cast<const int4*>(rect), frame->views, cnt);
            PS_LAUNCH_CHECK();
        }
    }
    // Pair numbering: offsets clamp at the int range (still non-decreasing); the tile total
    // then exceeds every capacity and nothing is scattered (kMaxPairs).
    const int tr = scan_tiles(R), tt = scan_tiles(frame->n_tiles);
    const ScanJob jr{w.rec_cnt, R, w.rec_cnt, nullptr, kMaxPairs, nullptr, nullptr, 0,
                     w.chunk_first, nch, w.part, tr};
    const ScanJob jt{w.tile_cnt, frame->n_tiles, tile_ptr, w.cursor, capacity, d_required,
                     d_status, 1, nullptr, 0, w.part + tr, tt};
    PS_CUDA_CHECK(launch_after(k_scan_sums, tr + tt, kScanThreads, 0, st, jr, jt));
    PS_CUDA_CHECK(launch_after(k_scan_apply, tr + tt, kScanThreads, 0, st, jr, jt));
    if (R > 0 && capacity > 0) {
        PS_CUDA_CHECK(launch_after(k_pair_scatter, kFlatBlocks, kPairBlock, 0, st, w.rec_cnt, R, w.rec_info, tile_ptr,
                                   w.cursor, w.ent_tmp, reinterpret_cast<const float4*>(rec), key, frame->views,
                                   s->tile_w, s->tile_h, s->z_near, w.chunk_first, nch));
        constexpr int per = kSortWarps * kSortTiles;
        PS_CUDA_CHECK(launch_after(k_sort, (frame->n_tiles + per - 1) / per, kSortWarps * 32, 0, st, tile_ptr,
                                   frame->n_tiles, w.rec_cnt + R, w.ent_tmp, tile_ent, tile_key));
    }
    return PS_OK;
}

extern "C" ps_status ps_bin_tiles(const ps_frame* frame, const ps_settings* s, const float* rec,
                                  const int* rect, const float* key, int* tile_ptr, int* tile_ent,
                                  float* tile_key, long long capacity, long long* d_required,
                                  void* ws, size_t ws_bytes_, int* d_status, ps_stream stream)
{
    return ps::bin_tiles(frame, s, rec, rect, key, tile_ptr, tile_ent, tile_key, capacity, d_required, ws,
                         ws_bytes_, false, d_status, reinterpret_cast<cudaStream_t>(stream));
}
