// ps_conv.cu -- the seed network's 3x3 stride-2 convolutions as implicit GEMMs on
// the tensor cores: the im2col matrix never exists in memory.
//
//   y[p, co] = relu(bias[co] + sum over taps (ky, kx) and ci of
//              x[b, 2 oy - 1 + ky, 2 ox - 1 + kx, ci] w[co, (3 ky + kx) C + ci])
//
// with output positions p = (b, oy, ox), activations NHWC bf16 and FP32
// accumulation.  The tap order and the 16-wide K steps are those of an im2col
// matrix product, so the results equal ps_seed_im2col + ps_gemm_bf16 bit for bit; so
// do the gradients of the convolutions' weights and inputs.
// Measured: the network's forward on 4,480 patches (64 views of 640x480) 6,766 -> 377 us
// (the element-wise im2col alone took 5,870 us); a training step of 256 patches 6,812 ->
// 426 us (the weight gradients, one to nine CTAs each, took most of 5,400 us).
#include "ps_tc.cuh"

using namespace ps;

namespace {

constexpr int kCh = 64;                       // channels of every activation (and output channels)
constexpr int kRows = 128;                    // output positions per tile
constexpr int kTile = kRows * kCh * 2;        // bytes of a tile of 128 positions (16 KB)
constexpr int kWTap = kCh * kCh * 2;          // bytes of one tap's weights (8 KB)
constexpr int kTaps = 9;
constexpr int kSide = 64;                     // the first layer's input side (64 x 64 x 4)
constexpr int kPatch = kSide * kSide * 4 * 2; // bytes of an input patch (32 KB)
constexpr int kTmemCols = 128;                // two accumulators of 64 columns

__host__ __device__ constexpr int first_smem() { return kPatch + 2 * kTile + kWTap + 1024; }

// The pixels that tap (ky, kx) reads for the output positions from row y0 of patch b0
// on, from a tap_map: pixel 2 o - 1 + k is entry o - 1 of the odd pixels for k = 0, o of
// the even ones for k = 1, o of the odd ones for k = 2; entry -1 is filled with zeros.
__device__ __forceinline__ void load_tap(uint32_t dst, const CUtensorMap* tm, int tap, int y0, int b0, uint32_t bar)
{
    const int ky = tap / 3, kx = tap - 3 * ky;
    tma_load_5d(dst, tm, kx == 1 ? 0 : kCh, kx == 0 ? -1 : 0, ky == 1 ? 0 : 1, ky == 0 ? y0 - 1 : y0, b0, bar);
}

// bias + ReLU of 32 accumulator columns, packed to bf16 and parked in a tile of
// 128-byte rows with the 128-byte swizzle (16-byte chunk c of row r at chunk
// c ^ (r & 7)): the layout a TMA tile store reads; no bank conflicts.
__device__ __forceinline__ void park_relu32(uint8_t* tile, int row, int half, const float (&v)[32],
                                            const float* __restrict__ bias)
{
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = 8 * c + 2 * j;
            const __nv_bfloat162 h = __floats2bfloat162_rn(fmaxf(v[k] + bias[32 * half + k], 0.f),
                                                           fmaxf(v[k + 1] + bias[32 * half + k + 1], 0.f));
            w[j] = *reinterpret_cast<const uint32_t*>(&h);
        }
        const int chunk = (4 * half + c) ^ (row & 7);
        *reinterpret_cast<uint4*>(tile + row * 128 + chunk * 16) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// im2col row of one output position of the first layer (36 of 64 columns; 48 are
// multiplied): nine 8-byte pixels from the patch in shared memory, zeros outside.
__device__ __forceinline__ void first_row(uint8_t* tile, int row, const uint2* __restrict__ patch, int oy, int ox)
{
    uint2 px[12];
#pragma unroll
    for (int tap = 0; tap < 12; ++tap) {
        px[tap] = make_uint2(0u, 0u);
        const int y = 2 * oy - 1 + tap / 3, x = 2 * ox - 1 + tap % 3;
        if (tap < kTaps && y >= 0 && x >= 0) px[tap] = patch[y * kSide + x];
    }
#pragma unroll
    for (int c = 0; c < 6; ++c)
        *reinterpret_cast<uint4*>(tile + row * 128 + ((c ^ (row & 7)) << 4)) =
            make_uint4(px[2 * c].x, px[2 * c].y, px[2 * c + 1].x, px[2 * c + 1].y);
}

// First layer: [B, 64, 64, 4] -> [B, 32, 32, 64].  K is 36, so the work is the
// 128-byte output rows: bound by the write of y (587 of 734 MB at 4,480 patches).
// One CTA of 128 threads takes a patch at a time (32 KB by one bulk copy) and walks
// its eight tiles of 128 positions: every thread builds its position's im2col row
// in shared memory (a TMA box cannot: a pixel is 8 bytes), three MMAs, then the
// thread's output row goes to the same buffer and leaves by a TMA tile store that
// overlaps the next tile.  Three CTAs per SM hide each other's waits.  copy, if not
// null, receives the input patches (the backward's copy; one more bulk store).
__global__ void __launch_bounds__(128) k_conv_first(const uint8_t* __restrict__ x, uint8_t* __restrict__ copy,
                                                    const __grid_constant__ CUtensorMap tmW,
                                                    const __grid_constant__ CUtensorMap tmY,
                                                    const float* __restrict__ bias, int B, int* err)
{
    extern __shared__ uint8_t s_dyn[];
    __shared__ __align__(8) uint64_t bar[3];           // patch, weights, MMA
    __shared__ uint32_t tmem_base;
    __shared__ float s_bias[kCh];
    uint8_t* sm = s_dyn + (((smem_u32(s_dyn) + 1023u) & ~1023u) - smem_u32(s_dyn));
    uint8_t* patch = sm;
    uint8_t* buf[2] = {sm + kPatch, sm + kPatch + kTile};
    uint8_t* wt = sm + kPatch + 2 * kTile;
    const int tid = threadIdx.x, warp = tid >> 5;
    const uint32_t bp = smem_u32(&bar[0]), bw = smem_u32(&bar[1]), bm = smem_u32(&bar[2]);

    if (warp == 0) tmem_alloc(&tmem_base, kTmemCols);
    if (tid == 0) {
        mbar_init(bp, 1);
        mbar_init(bw, 1);
        mbar_init(bm, 1);
        mbar_init_fence();
    }
    if (tid < kCh) s_bias[tid] = bias[tid];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    bool ok = true;
    if (tid == 0) {
        mbar_expect(bw, kWTap);
        tma_load_2d(smem_u32(wt), &tmW, 0, 0, bw);
    }
    ok = !__syncthreads_or(!mbar_wait(bw, 0));
    uint32_t np = 0, nm = 0;                           // patch loads issued, tiles multiplied
    for (int b = blockIdx.x; ok && b < B; b += gridDim.x) {
        if (tid == 0) {
            bulk_wait_read<2>();                       // the last patch's copy has left (older than two stores)
            mbar_expect(bp, kPatch);
            bulk_load(smem_u32(patch), x + (size_t)b * kPatch, kPatch, bp);
        }
        ok = mbar_wait(bp, np++ & 1);
        if (__syncthreads_or(!ok)) { ok = false; break; }
        if (tid == 0 && copy) {
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                         :: "l"(copy + (size_t)b * kPatch), "r"(smem_u32(patch)), "r"(kPatch) : "memory");
            bulk_commit();
        }
        for (int t = 0; t < 8; ++t) {
            uint8_t* tile = buf[t & 1];
            if (tid == 0) bulk_wait_read<1>();         // the store that last read this buffer
            __syncthreads();
            first_row(tile, tid, reinterpret_cast<const uint2*>(patch), 4 * t + (tid >> 5), tid & 31);
            fence_async_smem();
            tc_fence_before();
            __syncthreads();
            const uint32_t acc = tmem + (uint32_t)(t & 1) * kCh;
            if (tid == 0) {
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    mma_bf16(acc, smem_desc_k(smem_u32(tile) + 32 * k), smem_desc_k(smem_u32(wt) + 32 * k),
                             instr_desc(kRows, kCh), k > 0);
                mma_commit(bm);
            }
            ok = mbar_wait(bm, nm++ & 1);
            if (__syncthreads_or(!ok)) { ok = false; break; }
            tc_fence_after();
            float v[32];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                tmem_ld32(acc + ((uint32_t)(warp * 32) << 16) + 32 * h, v);
                park_relu32(tile, tid, h, v, s_bias);
            }
            fence_async_smem();
            __syncthreads();
            if (tid == 0) {
                tma_store_2d(&tmY, smem_u32(tile), 0, (b * 8 + t) * kRows);
                bulk_commit();
            }
        }
    }
    if (tid == 0) {
        if (!ok) {
            if (err) atomicOr(err, 1 << PS_ERR_TIMEOUT);
            // what is in flight gets another bounded wait before the memory is given up
            mbar_wait(bw, 0);
            if (np) mbar_wait(bp, (np - 1) & 1);
            if (nm) mbar_wait(bm, (nm - 1) & 1);
        }
        bulk_wait<0>();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, kTmemCols);
}

constexpr int kStages = 7;                    // input tiles in flight of an inner layer
constexpr int kInnerThreads = 192;            // copy warp, MMA warp, four epilogue warps

__host__ __device__ constexpr int inner_smem() { return kTaps * kWTap + kStages * kTile + 2 * kTile + 1024; }

// Inner layers: [B, 2 So, 2 So, 64] -> [B, So, So, 64], So = 16, 8 or 4.  Bound by the
// 2.25 reads of every input element out of L2 (each is used by 2.25 taps on
// average).  Persistent CTAs, one per SM, keep the layer's weights (72 KB) in shared
// memory; a copy warp streams one 16 KB tile per tap -- a TMA box of every second
// pixel in x and y (zero fill outside the image), which lands as the tap's im2col
// slice -- through a ring of 7; an MMA warp issues four M 128, N 64, K 16
// steps per slice into one of two accumulators; four warps apply bias and ReLU and
// send the tile out by TMA while the next tile is multiplied.  Every wait is bounded;
// a wait that runs out ends its role, reports PS_ERR_TIMEOUT and drains what it issued.
struct InnerArgs {
    const float* bias;
    int n_tiles;
    int so_log2;             // output side
    int* err;
};

__global__ void __launch_bounds__(kInnerThreads, 1) k_conv_inner(const __grid_constant__ CUtensorMap tmX,
                                                                 const __grid_constant__ CUtensorMap tmW,
                                                                 const __grid_constant__ CUtensorMap tmY,
                                                                 InnerArgs a)
{
    extern __shared__ uint8_t s_dyn[];
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages], acc_full[2], acc_empty[2], w_full;
    __shared__ uint32_t tmem_base;
    __shared__ float s_bias[kCh];
    __shared__ int failed, out_failed;                 // out_failed: written by the epilogue warps alone
    uint8_t* sm = s_dyn + (((smem_u32(s_dyn) + 1023u) & ~1023u) - smem_u32(s_dyn));
    const uint32_t wt = smem_u32(sm), ring = wt + kTaps * kWTap;
    uint8_t* out = sm + kTaps * kWTap + kStages * kTile;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) tmem_alloc(&tmem_base, kTmemCols);
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&acc_full[s]), 1);
            mbar_init(smem_u32(&acc_empty[s]), 128);
        }
        mbar_init(smem_u32(&w_full), 1);
        mbar_init_fence();
        failed = out_failed = 0;
    }
    if (tid < kCh) s_bias[tid] = a.bias[tid];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    int issued = 0;                                    // slices (copy warp)

    if (warp == 0) {
        if (elect_one()) {
            mbar_expect(smem_u32(&w_full), kTaps * kWTap);
#pragma unroll
            for (int tap = 0; tap < kTaps; ++tap) tma_load_2d(wt + tap * kWTap, &tmW, tap * kCh, 0, smem_u32(&w_full));
        }
        bool ok = true;
        int s = 0;
        uint32_t par = 1;                              // parity of the slot's last release
        for (int tile = blockIdx.x; ok && tile < a.n_tiles; tile += gridDim.x) {
            const int p0 = tile * kRows;
            const int b0 = p0 >> (2 * a.so_log2), y0 = (p0 >> a.so_log2) & ((1 << a.so_log2) - 1);
#pragma unroll
            for (int tap = 0; tap < kTaps; ++tap) {
                if (issued >= kStages) ok = ok && mbar_wait(smem_u32(&empty[s]), par);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (elect_one()) {
                    mbar_expect(smem_u32(&full[s]), kTile);
                    load_tap(ring + s * kTile, &tmX, tap, y0, b0, smem_u32(&full[s]));
                }
                __syncwarp();
                ++issued;
                if (++s == kStages) { s = 0; par ^= 1; }
            }
        }
        if (!ok && lane == 0) failed = 1;
    } else if (warp == 1) {
        bool ok = mbar_wait(smem_u32(&w_full), 0);
        int it = 0, s = 0;
        uint32_t par = 0;
        for (int tile = blockIdx.x; ok && tile < a.n_tiles; tile += gridDim.x, ++it) {
            const int acc = it & 1;
            if (it >= 2) ok = mbar_wait(smem_u32(&acc_empty[acc]), (uint32_t)(((it >> 1) - 1) & 1));
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after();
            for (int tap = 0; ok && tap < kTaps; ++tap) {
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&full[s]), par));
                if (!ok) break;
                tc_fence_after();
                const uint64_t da = smem_desc_k(ring + s * kTile), db = smem_desc_k(wt + tap * kWTap);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < kCh / 16; ++k)
                        mma_bf16(tmem + acc * kCh, da + 2 * k, db + 2 * k, instr_desc(kRows, kCh), tap > 0 || k > 0);
                    mma_commit(smem_u32(&empty[s]));
                    if (tap == kTaps - 1) mma_commit(smem_u32(&acc_full[acc]));
                }
                __syncwarp();
                if (++s == kStages) { s = 0; par ^= 1; }
            }
        }
        if (!ok && lane == 0) failed = 1;
    } else {
        const int quad = warp & 3;                     // the tensor-memory lanes this warp may read
        const int row = quad * 32 + lane;
        bool ok = true;
        int it = 0;
        for (int tile = blockIdx.x; tile < a.n_tiles; tile += gridDim.x, ++it) {
            const int acc = it & 1;
            uint8_t* park = out + acc * kTile;
            ok = mbar_wait(smem_u32(&acc_full[acc]), (uint32_t)((it >> 1) & 1));
            if (!ok) *reinterpret_cast<volatile int*>(&out_failed) = 1;
            if (tid == 64) bulk_wait_read<1>();        // the store that last read this buffer
            // between the barriers no thread writes the flag, so all four warps read the same
            asm volatile("bar.sync 1, 128;" ::: "memory");
            ok = *reinterpret_cast<volatile int*>(&out_failed) == 0;
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (!ok) break;
            tc_fence_after();
            float v[32];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + acc * kCh + 32 * h, v);
                park_relu32(park, row, h, v, s_bias);
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&acc_empty[acc]));
            fence_async_smem();
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (tid == 64) {
                tma_store_2d(&tmY, smem_u32(park), 0, tile * kRows);
                bulk_commit();
            }
        }
        if (tid == 64) bulk_wait<0>();
    }
    __syncthreads();
    if ((failed || out_failed) && tid == 0) {
        if (a.err) atomicOr(a.err, 1 << PS_ERR_TIMEOUT);
        // copies and MMAs in flight get another bounded wait before the memory is given up
        mbar_wait(smem_u32(&w_full), 0);
        for (int j = issued > kStages ? issued - kStages : 0; j < issued; ++j) {
            mbar_wait(smem_u32(&full[j % kStages]), (uint32_t)((j / kStages) & 1));
            mbar_wait(smem_u32(&empty[j % kStages]), (uint32_t)((j / kStages) & 1), 1 << 16);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, kTmemCols);
}

// ---------------------------------------------------------------------------
// Backward.
//
// Weight gradients gw[co, k] = sum over positions p of dz[p, co] A[p, k], A the im2col
// matrix: a 64 x 576 (64 x 36) result summed over up to 10^6 rows.  An FP32
// accumulator's last bits depend on the order of that sum, and its size makes them
// count: the tensor core truncates, so at 262,144 rows one chain and a sum split over
// the SMs differ by 3e-4.  The chain in order of p is kept (results equal
// ps_gemm_bf16's on transposed copies bit for bit) and the outputs are split instead:
//   inner layers: one CTA per tap, 64 x 64 outputs; tap tile and dz tile come straight
//     from the forward's TMA boxes and are read MN-major (no transposed copies);
//   first layer: one CTA per 8 columns x 8 channels, 40 in all, from operands stored in
//     blocks of 8 columns (16 bytes x P rows, contiguous bulk copies; the unswizzled
//     core-matrix layout): its chain of P / 16 steps is the longest, and a step costs
//     the smallest the instruction takes, M 64 (8 rows real, the others' sums dropped)
//     and N 8: 27 cycles in groups of 64 (a wait and a commit cost 160 between groups).
// All layers run in one launch, the first layer's CTAs first, so the shorter chains
// hide behind the longest.  (Split over 152 SMs with the parts added afterwards the
// three kernels took 72 us at 256 patches, but changed the gradients by up to 6e-4.)
constexpr int kRing = 128 * 1024;             // bytes of operand tiles in flight
constexpr int kChunk = 64;                    // positions per stage of an inner layer
constexpr int kChunkTile = kChunk * kCh * 2;  // 8 KB
constexpr int kFirstK = 36;                   // columns of the first layer's weights
constexpr int kBlocksK = 5;                   // its blocks of 8 columns (the last half empty)
constexpr int kFirstChunk = 1024;             // positions per stage of the first layer
constexpr int kFirstTile = kFirstChunk * 16;  // 16 KB per block of 8 columns
constexpr int kFirstCtas = kBlocksK * (kCh / 8);
constexpr int kWgradCtas = kFirstCtas + 3 * kTaps;
constexpr int kMaxStages = kRing / (2 * kChunkTile);

__host__ __device__ constexpr int wgrad_smem() { return kRing + 1024; }

struct WgradMaps { CUtensorMap x[3], z[3]; };  // inner layers 1, 2, 3

struct WgradArgs {
    const uint8_t* xb;       // first layer: [5][P][8] bf16 im2col columns
    const uint8_t* zb;       // [8][P][8] bf16 masked output gradients
    float* gw[4];            // [64][36], 3 x [64][576]
    long long P0;            // positions of the first layer
    int B;
    int* err;
};

__global__ void __launch_bounds__(kInnerThreads, 1) k_wgrad(const __grid_constant__ WgradMaps maps, WgradArgs a)
{
    extern __shared__ uint8_t s_dyn[];
    __shared__ __align__(8) uint64_t full[kMaxStages], empty[kMaxStages], done;
    __shared__ uint32_t tmem_base;
    __shared__ int failed;
    const uint32_t base = (smem_u32(s_dyn) + 1023u) & ~1023u;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool first = blockIdx.x < kFirstCtas;
    const int inner = first ? 0 : (blockIdx.x - kFirstCtas) / kTaps;        // 0, 1, 2: layers 1, 2, 3
    const int tap = first ? 0 : (blockIdx.x - kFirstCtas) % kTaps;
    const int kb = blockIdx.x >> 3, cb = blockIdx.x & 7;                    // first layer: column and channel block
    const int so_log2 = 4 - inner, so = 1 << so_log2;
    const int n = first ? (int)(a.P0 / kFirstChunk) : a.B * so * so / kChunk;   // stages
    const int tile = first ? kFirstTile : kChunkTile;
    const int stages = kRing / (2 * tile);

    if (warp == 0) tmem_alloc(&tmem_base, kCh);
    if (tid == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        mbar_init(smem_u32(&done), 1);
        mbar_init_fence();
        failed = 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    int issued = 0;
    bool ok = true;
    if (warp == 0) {
        const CUtensorMap* tx = &maps.x[inner];
        const CUtensorMap* tz = &maps.z[inner];
        const uint8_t* xb = a.xb + (size_t)kb * a.P0 * 16;
        const uint8_t* zb = a.zb + (size_t)cb * a.P0 * 16;
        int s = 0;
        uint32_t par = 1;                              // parity of the stage's last release
        for (int i = 0; i < n; ++i) {
            if (i >= stages) ok = mbar_wait(smem_u32(&empty[s]), par);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const uint32_t st = base + s * 2 * tile, f = smem_u32(&full[s]);
            const int p0 = i * kChunk, b0 = p0 >> (2 * so_log2), y0 = (p0 >> so_log2) & (so - 1);
            if (elect_one()) {
                mbar_expect(f, 2 * tile);
                if (first) {
                    bulk_load(st, xb + (size_t)i * kFirstTile, kFirstTile, f);
                    bulk_load(st + kFirstTile, zb + (size_t)i * kFirstTile, kFirstTile, f);
                } else {
                    load_tap(st, tx, tap, y0, b0, f);
                    tma_load_2d(st + kChunkTile, tz, 0, p0, f);
                }
            }
            __syncwarp();
            ++issued;
            if (++s == stages) { s = 0; par ^= 1; }
        }
        if (!ok && lane == 0) failed = 1;
    } else if (warp == 1) {
        int s = 0;
        uint32_t par = 0;
        for (int i = 0; ok && i < n; ++i) {
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&full[s]), par));
            if (!ok) break;
            tc_fence_after();
            const uint32_t st = base + s * 2 * tile;
            if (first) {
                // groups of 8 rows are 128 bytes apart; the 7 blocks past A's only real one
                // lie in the next groups
                const uint64_t da = smem_desc_blocks(st, 128), db = smem_desc_blocks(st + kFirstTile, 128);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < kFirstChunk / 16; ++k)
                        mma_bf16(tmem, da + 16 * k, db + 16 * k, instr_desc(64, 8, 1, 1), i > 0 || k > 0);
                    mma_commit(smem_u32(&empty[s]));
                    if (i == n - 1) mma_commit(smem_u32(&done));
                }
            } else {
                const uint64_t da = smem_desc_mn(st, kChunkTile), db = smem_desc_mn(st + kChunkTile, kChunkTile);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < kChunk / 16; ++k)
                        mma_bf16(tmem, da + 128 * k, db + 128 * k, instr_desc(64, kCh, 1, 1), i > 0 || k > 0);
                    mma_commit(smem_u32(&empty[s]));
                    if (i == n - 1) mma_commit(smem_u32(&done));
                }
            }
            __syncwarp();
            if (++s == stages) { s = 0; par ^= 1; }
        }
        if (!ok && lane == 0) failed = 1;
    } else if (warp >= 2) {
        ok = mbar_wait(smem_u32(&done), 0, 16 * kWaitPolls);      // the whole chain
        if (!ok) failed = 1;
        if (__all_sync(0xffffffffu, ok)) {
            tc_fence_after();
            // a 64-row result: row m in lane 32 (m / 16) + m % 16
            const int quad = warp & 3, row = quad * 16 + lane;
            float v[32];
            if (first) {
                tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16), v);
                const int k = 8 * kb + row;
                if (row < 8 && quad == 0 && k < kFirstK) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) a.gw[0][(8 * cb + j) * kFirstK + k] = v[j];
                }
            } else {
                float* gw = a.gw[1 + inner] + tap * kCh + row;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + 32 * h, v);
                    if (lane < 16) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) gw[(32 * h + j) * kTaps * kCh] = v[j];
                    }
                }
            }
        }
    }
    __syncthreads();
    if (failed && tid == 0) {
        if (a.err) atomicOr(a.err, 1 << PS_ERR_TIMEOUT);
        // copies and MMAs in flight get another bounded wait before the memory is given up
        for (int j = issued > stages ? issued - stages : 0; j < issued; ++j) {
            mbar_wait(smem_u32(&full[j % stages]), (uint32_t)((j / stages) & 1), 1 << 16);
            mbar_wait(smem_u32(&empty[j % stages]), (uint32_t)((j / stages) & 1), 1 << 16);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, kCh);
}

__device__ __forceinline__ void store32(float* dst, const float (&v)[32])
{
#pragma unroll
    for (int j = 0; j < 32; j += 4)
        *reinterpret_cast<float4*>(dst + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
}

// Input gradient of an inner layer, the ReLU mask of the layer below and that layer's
// bias gradient, in one pass.  A pixel (2h + py, 2w + px) receives from the taps of
// matching parity only: 1, 2, 2 or 4 of the 9 for the four (py, px) classes.  One CTA
// takes 128 positions (h, w) of one class: a K-major dz tile per tap, shifted by 0 or 1
// in h and w (zero fill past the edge), against the tap's weights MN-major, each tap
// into its own accumulator; the accumulators are added in tap order in FP32 (the sums
// of im2col's adjoint, bit for bit), masked by the activation, rounded to bf16 and
// written; the FP32 values' column sums are added to gb.
constexpr int kPitch = 68;                    // floats per parked row (conflict-free float4 rows)
__host__ __device__ constexpr int dgrad_smem() { return 4 * kTile + 4 * kWTap + 1024; }

struct DgradArgs {
    const uint4* y;          // [B][2 so][2 so][64] bf16: the activation below
    uint4* dz;               // same shape: its masked gradient, bf16
    long long block;         // 0: dz in rows of 64 channels; else blocks of 8 channels, so many rows each
    float* gb;               // [64], added to
    int so_log2;
    int* err;
};

__global__ void __launch_bounds__(128) k_dgrad(const __grid_constant__ CUtensorMap tmZ,
                                               const __grid_constant__ CUtensorMap tmW, DgradArgs a)
{
    extern __shared__ uint8_t s_dyn[];
    __shared__ __align__(8) uint64_t full[4], done;
    __shared__ uint32_t tmem_base;
    __shared__ float s_gb[4][kCh];
    uint8_t* sm = s_dyn + (((smem_u32(s_dyn) + 1023u) & ~1023u) - smem_u32(s_dyn));
    const uint32_t za = smem_u32(sm), wa = za + 4 * kTile;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cls = 3 - blockIdx.y, py = cls >> 1, px = cls & 1;      // the 4-tap class first
    const int ny = 1 + py, nx = 1 + px, taps = ny * nx;
    const int so = 1 << a.so_log2;

    if (warp == 0) tmem_alloc(&tmem_base, 256);
    if (tid == 0) {
        for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&full[i]), 1);
        mbar_init(smem_u32(&done), 1);
        mbar_init_fence();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    const int p0 = blockIdx.x * kRows;
    bool ok = true;
    if (tid == 0) {
        const int b0 = p0 >> (2 * a.so_log2), h0 = (p0 >> a.so_log2) & (so - 1);
        for (int i = 0; i < taps; ++i) {
            // odd side: taps 0 (one further) and 2 (same position); even side: tap 1
            const int iy = i / nx, ix = i - iy * nx;
            const int ky = py ? 2 * iy : 1, kx = px ? 2 * ix : 1;
            const uint32_t f = smem_u32(&full[i]);
            mbar_expect(f, kTile + kWTap);
            tma_load_4d(za + i * kTile, &tmZ, 0, px && ix == 0 ? 1 : 0, h0 + (py && iy == 0 ? 1 : 0), b0, f);
            tma_load_2d(wa + i * kWTap, &tmW, (3 * ky + kx) * kCh, 0, f);
        }
        int i = 0;
        for (; i < taps; ++i) {
            ok = mbar_wait(smem_u32(&full[i]), 0);
            if (!ok) break;
            tc_fence_after();
            const uint64_t da = smem_desc_k(za + i * kTile), db = smem_desc_mn(wa + i * kWTap, kWTap);
#pragma unroll
            for (int k = 0; k < kCh / 16; ++k)
                mma_bf16(tmem + i * kCh, da + 2 * k, db + 128 * k, instr_desc(kRows, kCh, 0, 1), k > 0);
        }
        mma_commit(smem_u32(&done));
        for (; i < taps; ++i) mbar_wait(smem_u32(&full[i]), 0);      // after a time-out: copies in flight
    }
    ok = mbar_wait(smem_u32(&done), 0) && ok;
    if (__syncthreads_or(!ok)) {
        if (tid == 0 && a.err) atomicOr(a.err, 1 << PS_ERR_TIMEOUT);
    } else {
        tc_fence_after();
        float* park = reinterpret_cast<float*>(sm);       // over the dz tiles, which the MMAs have read
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float s[32], v[32];
            const uint32_t t = tmem + ((uint32_t)(warp * 32) << 16) + 32 * h;
            tmem_ld32(t, s);
            for (int i = 1; i < taps; ++i) {
                tmem_ld32(t + i * kCh, v);
#pragma unroll
                for (int j = 0; j < 32; ++j) s[j] += v[j];
            }
            store32(park + tid * kPitch + 32 * h, s);
        }
        __syncthreads();
        // eight threads per row, 16 rows at a time: whole 128-byte rows of y and dz
        const int c8 = tid & 7;
        float sum[8] = {};
        for (int r = tid >> 3; r < kRows; r += 16) {
            const int p = p0 + r;
            const int w = p & (so - 1), hh = (p >> a.so_log2) & (so - 1), b = p >> (2 * a.so_log2);
            const size_t pix = ((size_t)b * 2 * so + 2 * hh + py) * 2 * so + 2 * w + px;
            const uint4 yv = __ldg(&a.y[pix * 8 + c8]);
            const uint32_t yw[4] = {yv.x, yv.y, yv.z, yv.w};
            const float4 g0 = *reinterpret_cast<const float4*>(park + r * kPitch + 8 * c8);
            const float4 g1 = *reinterpret_cast<const float4*>(park + r * kPitch + 8 * c8 + 4);
            float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
            uint32_t out[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const __nv_bfloat162 ya = *reinterpret_cast<const __nv_bfloat162*>(&yw[j]);
                g[2 * j] = __low2float(ya) > 0.f ? g[2 * j] : 0.f;
                g[2 * j + 1] = __high2float(ya) > 0.f ? g[2 * j + 1] : 0.f;
                sum[2 * j] += g[2 * j];
                sum[2 * j + 1] += g[2 * j + 1];
                const __nv_bfloat162 z = __floats2bfloat162_rn(g[2 * j], g[2 * j + 1]);
                out[j] = *reinterpret_cast<const uint32_t*>(&z);
            }
            a.dz[a.block ? (size_t)c8 * a.block + pix : pix * 8 + c8] = make_uint4(out[0], out[1], out[2], out[3]);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], 8);
            sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], 16);
            if (lane < 8) s_gb[warp][8 * c8 + j] = sum[j];
        }
        __syncthreads();
        if (tid < kCh) atomicAdd(&a.gb[tid], (s_gb[0][tid] + s_gb[1][tid]) + (s_gb[2][tid] + s_gb[3][tid]));
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, 256);
}

// Linear layer, backward, apart from its input gradient (a GEMM on the operands made
// here): bf16 copies of dout (zero-padded to 128 columns) and of the transposed weights,
// the weight and bias gradients (bf16 operands, FP32 sums), the zeroed bias gradients
// of the convolutions, to which the next kernels add, and the first layer's im2col
// columns in blocks of 8 for k_wgrad.
constexpr int kOut = 96;
constexpr int kOutPad = 128;
constexpr int kHeadTile = 4;                  // output columns per weight-gradient block

struct HeadArgs {
    const float* dout;               // [B][96]
    const float* w;                  // [96][64]
    const __nv_bfloat16* h;          // [B][64]
    __nv_bfloat16* dout16;           // [B][128]
    __nv_bfloat16* wt;               // [64][128]
    float* gw;                       // [96][64]
    float* gb;                       // [96]
    float* gb_conv[4];               // [64] each
    const uint2* x;                  // [B][64][64] pixels of 4 bf16
    uint4* xb;                       // [5][B * 1024][8] bf16
    int B;
};

__global__ void __launch_bounds__(256) k_head_grads(HeadArgs a)
{
    __shared__ float red[3][kHeadTile][kCh + 1];
    const int tid = threadIdx.x;
    if (blockIdx.x < kOut / kHeadTile) {
        const int o0 = blockIdx.x * kHeadTile, c = tid & 63, g = tid >> 6;
        float s[kHeadTile] = {}, sb[kHeadTile] = {};
        for (int b = g; b < a.B; b += 4) {
            const float4 d4 = __ldg(reinterpret_cast<const float4*>(a.dout + (size_t)b * kOut + o0));
            const float d[kHeadTile] = {d4.x, d4.y, d4.z, d4.w};
            const float h = __bfloat162float(a.h[(size_t)b * kCh + c]);
#pragma unroll
            for (int i = 0; i < kHeadTile; ++i) {
                s[i] = fmaf(__bfloat162float(__float2bfloat16(d[i])), h, s[i]);
                sb[i] += d[i];
            }
        }
        if (g > 0) {
#pragma unroll
            for (int i = 0; i < kHeadTile; ++i) {
                red[g - 1][i][c] = s[i];
                if (c == 0) red[g - 1][i][kCh] = sb[i];
            }
        }
        __syncthreads();
        if (g == 0) {
#pragma unroll
            for (int i = 0; i < kHeadTile; ++i) {
                a.gw[(o0 + i) * kCh + c] = (s[i] + red[0][i][c]) + (red[1][i][c] + red[2][i][c]);
                if (c == 0) a.gb[o0 + i] = (sb[i] + red[0][i][kCh]) + (red[1][i][kCh] + red[2][i][kCh]);
            }
        }
        return;
    }
    const int block = blockIdx.x - kOut / kHeadTile, n = gridDim.x - kOut / kHeadTile;
    if (block == 0) a.gb_conv[tid >> 6][tid & 63] = 0.f;
    const long long total = (long long)(a.B + kCh) * kOutPad;
    for (long long i = (long long)block * 256 + tid; i < total; i += (long long)n * 256) {
        const int c = (int)(i % kOutPad);
        const long long r = i / kOutPad;
        if (r < a.B) a.dout16[i] = __float2bfloat16(c < kOut ? a.dout[r * kOut + c] : 0.f);
        else {
            const int k = (int)(r - a.B);
            a.wt[k * kOutPad + c] = __float2bfloat16(c < kOut ? a.w[c * kCh + k] : 0.f);
        }
    }
    const long long P = (long long)a.B * 1024;
    for (long long p = (long long)block * 256 + tid; p < P; p += (long long)n * 256) {
        const uint2* patch = a.x + (p >> 10) * (kSide * kSide);
        const int oy = (int)(p >> 5) & 31, ox = (int)p & 31;
        uint2 px[10];
#pragma unroll
        for (int tap = 0; tap < 10; ++tap) {
            px[tap] = make_uint2(0u, 0u);
            const int y = 2 * oy - 1 + tap / 3, x = 2 * ox - 1 + tap % 3;
            if (tap < kTaps && y >= 0 && x >= 0) px[tap] = __ldg(&patch[y * kSide + x]);
        }
#pragma unroll
        for (int g = 0; g < kBlocksK; ++g)
            a.xb[g * P + p] = make_uint4(px[2 * g].x, px[2 * g].y, px[2 * g + 1].x, px[2 * g + 1].y);
    }
}

// Pooling, backward, with the last convolution's ReLU mask and bias gradient:
// dz[b, s, c] = bf16((y > 0) dh[b, c] / 16), gb[c] += the FP32 values.
__global__ void __launch_bounds__(256) k_pool_relu_bwd(const float* __restrict__ dh, const uint4* __restrict__ y,
                                                       int rows, uint4* __restrict__ dz, float* __restrict__ gb)
{
    __shared__ float s_gb[8][kCh];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, c8 = tid & 7;
    float sum[8] = {};
    for (long long r = (long long)blockIdx.x * 32 + (tid >> 3); r < rows; r += (long long)gridDim.x * 32) {
        const uint4 yv = __ldg(&y[r * 8 + c8]);
        const uint32_t yw[4] = {yv.x, yv.y, yv.z, yv.w};
        const float* g = dh + (r >> 4) * kCh + 8 * c8;
        uint32_t out[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const __nv_bfloat162 ya = *reinterpret_cast<const __nv_bfloat162*>(&yw[j]);
            const float g0 = __low2float(ya) > 0.f ? __ldg(&g[2 * j]) / 16.f : 0.f;
            const float g1 = __high2float(ya) > 0.f ? __ldg(&g[2 * j + 1]) / 16.f : 0.f;
            sum[2 * j] += g0;
            sum[2 * j + 1] += g1;
            const __nv_bfloat162 z = __floats2bfloat162_rn(g0, g1);
            out[j] = *reinterpret_cast<const uint32_t*>(&z);
        }
        dz[r * 8 + c8] = make_uint4(out[0], out[1], out[2], out[3]);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], 8);
        sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], 16);
        if (lane < 8) s_gb[warp][8 * c8 + j] = sum[j];
    }
    __syncthreads();
    if (tid < kCh) {
        float s = 0.f;
        for (int i = 0; i < 8; ++i) s += s_gb[i][tid];
        atomicAdd(&gb[tid], s);
    }
}

// bf16 copies of all five weight blocks, the first layer's zero-padded from 36 to 64
// columns, in one launch.
struct SyncArgs {
    const float* params;
    __nv_bfloat16* w[5];
};

__global__ void __launch_bounds__(256) k_sync_weights(SyncArgs a)
{
    // offsets of the weight blocks in the flat parameters: each is followed by its bias
    constexpr int kOff[5] = {0, 64 * 37, 64 * 37 + 64 * 577, 64 * 37 + 2 * 64 * 577, 64 * 37 + 3 * 64 * 577};
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < 64 * 64) {
        const int r = i >> 6, c = i & 63;
        a.w[0][i] = __float2bfloat16(c < kFirstK ? a.params[r * kFirstK + c] : 0.f);
        return;
    }
    int j = i - 64 * 64;
#pragma unroll
    for (int l = 1; l < 5; ++l) {
        const int n = l < 4 ? 64 * 576 : kOut * 64;
        if (j < n) { a.w[l][j] = __float2bfloat16(a.params[kOff[l] + j]); return; }
        j -= n;
    }
}

// Rows of 64 channels [rows][64], boxes of box_rows rows.
bool rows_map(CUtensorMap* m, const void* ptr, long long rows, int box_rows)
{
    const cuuint64_t dim[2] = {kCh, (cuuint64_t)rows}, stride[1] = {kCh * 2};
    const cuuint32_t box[2] = {kCh, (cuuint32_t)box_rows};
    return encode_map(m, ptr, 2, dim, stride, box);
}

// A layer's weights [64][K], boxes of 64 x 64.
bool weight_map(CUtensorMap* m, const void* ptr, int K)
{
    const cuuint64_t dim[2] = {(cuuint64_t)K, kCh}, stride[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {kCh, kCh};
    return encode_map(m, ptr, 2, dim, stride, box);
}

// Boxes of `positions` consecutive positions of a side x side grid.
struct GridBox { cuuint32_t w, h, n; };
GridBox grid_box(int side, int positions)
{
    const int rows = positions < side * side ? positions / side : side;
    return GridBox{(cuuint32_t)side, (cuuint32_t)rows, (cuuint32_t)(positions / (rows * side))};
}

// Activations [B][so][so][64], every position.
bool grid_map(CUtensorMap* m, const void* ptr, int B, int so, int positions)
{
    const GridBox g = grid_box(so, positions);
    const cuuint64_t row = (cuuint64_t)so * kCh * 2;
    const cuuint64_t dim[4] = {kCh, (cuuint64_t)so, (cuuint64_t)so, (cuuint64_t)B}, stride[3] = {kCh * 2, row, so * row};
    const cuuint32_t box[4] = {kCh, g.w, g.h, g.n};
    return encode_map(m, ptr, 4, dim, stride, box);
}

// A convolution's input [B][2 so][2 so][64]: the pixels one tap reads for consecutive
// output positions are every second one in x and y.  The parities are dimensions of
// their own -- (x parity, channel), x / 2, y parity, y / 2, patch -- so that the box is
// dense: with element steps of 2 instead the copies took twice as long.
bool tap_map(CUtensorMap* m, const void* ptr, int B, int so, int positions)
{
    const GridBox g = grid_box(so, positions);
    const cuuint64_t row = (cuuint64_t)2 * so * kCh * 2;
    const cuuint64_t dim[5] = {2 * kCh, (cuuint64_t)so, 2, (cuuint64_t)so, (cuuint64_t)B};
    const cuuint64_t stride[4] = {2 * kCh * 2, row, 2 * row, 2 * so * row};
    const cuuint32_t box[5] = {kCh, g.w, 1, g.h, g.n};
    return encode_map(m, ptr, 5, dim, stride, box);
}

cudaError_t set_smem(const void* fn, int bytes) { return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); }

cudaError_t sm_count(int* n)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    return e != cudaSuccess ? e : cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev);
}

}  // namespace

extern "C" ps_status ps_seed_conv_fwd(const void* x, int B, int side, int C, const void* w, const float* bias,
                                      void* y, void* x_copy, int* d_err, ps_stream stream)
{
    if (!x || !w || !bias || !y || B <= 0 || B >= (1 << 20)) return PS_ERR_ARG;
    const bool first = C == 4 && side == kSide;
    const bool inner = C == kCh && (side == 32 || side == 16 || side == 8);
    if (!first && !inner) return PS_ERR_ARG;
    const int so = side / 2;
    const long long P = (long long)B * so * so;
    if (P % kRows) return PS_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(x_copy)) & 15)
        return PS_ERR_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const bool unaligned = (reinterpret_cast<uintptr_t>(x) & 15) != 0;
    if (unaligned) {
        // a copy engine takes any alignment: read the copy instead
        if (!x_copy) return PS_ERR_ARG;
        PS_CUDA_CHECK(cudaMemcpyAsync(x_copy, x, (size_t)B * side * side * C * 2, cudaMemcpyDeviceToDevice, st));
        x = x_copy;
        x_copy = nullptr;
    }
    int sms = 0;
    PS_CUDA_CHECK(sm_count(&sms));
    CUtensorMap tw, ty;
    if (!rows_map(&ty, y, P, kRows)) return PS_ERR_CUDA;
    if (first) {
        if (!weight_map(&tw, w, kCh)) return PS_ERR_CUDA;
        PS_CUDA_CHECK(set_smem((const void*)k_conv_first, first_smem()));
        k_conv_first<<<B < 3 * sms ? B : 3 * sms, 128, first_smem(), st>>>(
            static_cast<const uint8_t*>(x), static_cast<uint8_t*>(x_copy), tw, ty, bias, B, d_err);
    } else {
        if (x_copy) return PS_ERR_ARG;
        CUtensorMap tx;
        if (!weight_map(&tw, w, kTaps * kCh) || !tap_map(&tx, x, B, so, kRows)) return PS_ERR_CUDA;
        PS_CUDA_CHECK(set_smem((const void*)k_conv_inner, inner_smem()));
        const int n_tiles = (int)(P / kRows);
        InnerArgs a{bias, n_tiles, 31 - __builtin_clz((unsigned)so), d_err};
        k_conv_inner<<<n_tiles < sms ? n_tiles : sms, kInnerThreads, inner_smem(), st>>>(tx, tw, ty, a);
    }
    PS_LAUNCH_CHECK();
    return PS_OK;
}

namespace {

constexpr int kSide_[4] = {64, 32, 16, 8};   // input side of each convolution

// Offsets of a layer's weights and bias in the flat parameter (and gradient) buffer.
inline size_t weight_off(int l) { return l == 0 ? 0 : (size_t)64 * 37 + (size_t)(l - 1) * 64 * 577; }
inline size_t bias_off(int l) { return weight_off(l) + (l == 0 ? 64 * 36 : l < 4 ? 64 * 576 : kOut * 64); }

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct BwdWs {
    __nv_bfloat16* dz[4];    // masked gradients of the four activations
    __nv_bfloat16* dout16;
    __nv_bfloat16* wt;
    float* dh;
    uint8_t* xb;             // the first layer's im2col columns, blocked
    size_t bytes;
};

BwdWs bwd_ws(void* ws, int B)
{
    char* p = static_cast<char*>(ws);
    BwdWs w;
    size_t o = 0;
    auto take = [&](size_t n) { char* r = p + o; o += align256(n); return r; };
    for (int l = 0; l < 4; ++l) w.dz[l] = reinterpret_cast<__nv_bfloat16*>(take((size_t)B * kSide_[l] * kSide_[l] / 4 * kCh * 2));
    w.dout16 = reinterpret_cast<__nv_bfloat16*>(take((size_t)B * kOutPad * 2));
    w.wt = reinterpret_cast<__nv_bfloat16*>(take((size_t)kCh * kOutPad * 2));
    w.dh = reinterpret_cast<float*>(take((size_t)B * kCh * 4));
    w.xb = reinterpret_cast<uint8_t*>(take((size_t)B * 1024 * kBlocksK * 16));
    w.bytes = o;
    return w;
}

}  // namespace

extern "C" size_t ps_seed_backward_ws_bytes(int B)
{
    if (B <= 0 || B >= (1 << 20)) return 0;
    return bwd_ws(nullptr, B).bytes;
}

extern "C" ps_status ps_seed_backward(const float* params, const void* const* w16, const void* x, const void* const* y,
                                      const void* h16, const float* dout, int B, float* grad, void* ws,
                                      size_t ws_bytes, int* d_err, ps_stream stream)
{
    if (!params || !w16 || !x || !y || !h16 || !dout || !grad || !ws || B <= 0 || B >= (1 << 20) || (B % 64))
        return PS_ERR_ARG;
    if (ws_bytes < ps_seed_backward_ws_bytes(B)) return PS_ERR_ARG;
    uintptr_t al = reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(h16);
    for (int l = 0; l < 4; ++l) {
        if (!w16[l] || !y[l]) return PS_ERR_ARG;
        al |= reinterpret_cast<uintptr_t>(w16[l]) | reinterpret_cast<uintptr_t>(y[l]);
    }
    al |= reinterpret_cast<uintptr_t>(dout);
    if ((al & 15) || (reinterpret_cast<uintptr_t>(ws) & 255)) return PS_ERR_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int sms = 0;
    PS_CUDA_CHECK(sm_count(&sms));
    const BwdWs w = bwd_ws(ws, B);

    HeadArgs ha;
    ha.dout = dout; ha.w = params + weight_off(4); ha.h = static_cast<const __nv_bfloat16*>(h16);
    ha.dout16 = w.dout16; ha.wt = w.wt; ha.gw = grad + weight_off(4); ha.gb = grad + bias_off(4);
    for (int l = 0; l < 4; ++l) ha.gb_conv[l] = grad + bias_off(l);
    ha.x = static_cast<const uint2*>(x); ha.xb = reinterpret_cast<uint4*>(w.xb);
    ha.B = B;
    const int copy_blocks = 4 * B < 8 * sms ? 4 * B : 8 * sms;       // 256 of B x 1024 positions per step
    k_head_grads<<<kOut / kHeadTile + copy_blocks, 256, 0, st>>>(ha);
    PS_LAUNCH_CHECK();
    const ps_status e = ps_gemm_bf16(w.dout16, w.wt, nullptr, w.dh, nullptr, B, kCh, kOutPad, kCh, 0, 0, d_err, stream);
    if (e != PS_OK) return e;
    const int rows = B * 16;
    k_pool_relu_bwd<<<rows / 32 < 2 * sms ? rows / 32 : 2 * sms, 256, 0, st>>>(
        w.dh, static_cast<const uint4*>(y[3]), rows, reinterpret_cast<uint4*>(w.dz[3]), grad + bias_off(3));
    PS_LAUNCH_CHECK();

    PS_CUDA_CHECK(set_smem((const void*)k_dgrad, dgrad_smem()));
    PS_CUDA_CHECK(set_smem((const void*)k_wgrad, wgrad_smem()));
    WgradMaps maps;
    for (int l = 3; l >= 1; --l) {
        const int so = kSide_[l] / 2;
        const long long P = (long long)B * so * so;
        CUtensorMap tw, tg;
        if (!tap_map(&maps.x[l - 1], y[l - 1], B, so, kChunk) || !rows_map(&maps.z[l - 1], w.dz[l], P, kChunk))
            return PS_ERR_CUDA;
        if (!grid_map(&tg, w.dz[l], B, so, kRows) || !weight_map(&tw, w16[l], kTaps * kCh)) return PS_ERR_CUDA;
        DgradArgs da{static_cast<const uint4*>(y[l - 1]), reinterpret_cast<uint4*>(w.dz[l - 1]),
                     l == 1 ? (long long)B * 1024 : 0, grad + bias_off(l - 1), 31 - __builtin_clz((unsigned)so), d_err};
        k_dgrad<<<dim3((unsigned)(P / kRows), 4), 128, dgrad_smem(), st>>>(tg, tw, da);
        PS_LAUNCH_CHECK();
    }
    WgradArgs wa;
    wa.xb = w.xb; wa.zb = reinterpret_cast<const uint8_t*>(w.dz[0]);
    for (int l = 0; l < 4; ++l) wa.gw[l] = grad + weight_off(l);
    wa.P0 = (long long)B * 1024; wa.B = B; wa.err = d_err;
    k_wgrad<<<kWgradCtas, kInnerThreads, wgrad_smem(), st>>>(maps, wa);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

extern "C" ps_status ps_seed_sync_weights(const float* params, void* const* w16, ps_stream stream)
{
    if (!params || !w16) return PS_ERR_ARG;
    SyncArgs a;
    a.params = params;
    for (int l = 0; l < 5; ++l) {
        if (!w16[l]) return PS_ERR_ARG;
        a.w[l] = static_cast<__nv_bfloat16*>(w16[l]);
    }
    constexpr int n = 64 * 64 + 3 * 64 * 576 + kOut * 64;
    k_sync_weights<<<(n + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(a);
    PS_LAUNCH_CHECK();
    return PS_OK;
}
