// ps_conv.cu -- the seed network's 3x3 stride-2 convolutions as implicit GEMMs on
// the tensor cores: the im2col matrix never exists in memory.
//
//   y[p, co] = relu(bias[co] + sum over taps (ky, kx) and ci of
//              x[b, 2 oy - 1 + ky, 2 ox - 1 + kx, ci] w[co, (3 ky + kx) C + ci])
//
// with output positions p = (b, oy, ox), activations NHWC bf16 and FP32
// accumulation.  The tap order and the 16-wide K steps are those of an im2col
// matrix product, so the results equal ps_seed_im2col + ps_gemm_bf16 bit for bit.
// The network's forward on 4,480 patches (64 views of 640x480): 6,766 -> 421 us (the
// element-wise im2col alone took 5,870 us); on 256 patches 391 -> 52 us.
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
    ok = mbar_wait(bw, 0);
    uint32_t np = 0, nm = 0;                           // patches loaded, tiles multiplied
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
        if (tid == 0) {
            bulk_wait_read<2>();                       // the last patch's copy has left (older than two stores)
            mbar_expect(bp, kPatch);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         :: "r"(smem_u32(patch)), "l"(x + (size_t)b * kPatch), "r"(kPatch), "r"(bp) : "memory");
        }
        ok = ok && mbar_wait(bp, np++ & 1);
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
        if (!ok) break;
    }
    if (tid == 0) {
        if (!ok) {
            if (err) atomicOr(err, 1 << PS_ERR_TIMEOUT);
            // what is in flight gets another bounded wait before the memory is given up
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
// pixel (element step 2 in x and y; zero fill outside the image), which lands as the
// tap's im2col slice -- through a ring of 7; an MMA warp issues four M 128, N 64, K 16
// steps per slice into one of two accumulators; four warps apply bias and ReLU and
// send the tile out by TMA while the next tile is multiplied.  Every wait is bounded;
// a wait that runs out ends its role, reports PS_ERR_TIMEOUT and drains what it issued.
struct InnerArgs {
    const float* bias;
    int n_tiles;
    int so;                  // output side
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
    const int per_patch = a.so * a.so;                 // positions per patch
    int issued = 0;                                    // slices (copy warp)

    if (warp == 0) {
        if (lane == 0) {
            mbar_expect(smem_u32(&w_full), kTaps * kWTap);
            for (int tap = 0; tap < kTaps; ++tap) tma_load_2d(wt + tap * kWTap, &tmW, tap * kCh, 0, smem_u32(&w_full));
            bool ok = true;
            for (int tile = blockIdx.x; ok && tile < a.n_tiles; tile += gridDim.x) {
                const int p0 = tile * kRows;
                const int b0 = p0 / per_patch, y0 = 2 * ((p0 - b0 * per_patch) / a.so);
                for (int tap = 0; ok && tap < kTaps; ++tap) {
                    const int s = issued % kStages, u = issued / kStages;
                    if (u > 0) ok = mbar_wait(smem_u32(&empty[s]), (uint32_t)((u - 1) & 1));
                    if (!ok) break;
                    mbar_expect(smem_u32(&full[s]), kTile);
                    tma_load_4d(ring + s * kTile, &tmX, 0, tap % 3 - 1, y0 + tap / 3 - 1, b0, smem_u32(&full[s]));
                    ++issued;
                }
            }
            if (!ok) failed = 1;
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            bool ok = mbar_wait(smem_u32(&w_full), 0);
            int n = 0, it = 0;
            for (int tile = blockIdx.x; ok && tile < a.n_tiles; tile += gridDim.x, ++it) {
                const int acc = it & 1;
                if (it >= 2) ok = mbar_wait(smem_u32(&acc_empty[acc]), (uint32_t)(((it >> 1) - 1) & 1));
                tc_fence_after();
                for (int tap = 0; ok && tap < kTaps; ++tap, ++n) {
                    const int s = n % kStages;
                    ok = mbar_wait(smem_u32(&full[s]), (uint32_t)((n / kStages) & 1));
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int k = 0; k < kCh / 16; ++k)
                        mma_bf16(tmem + acc * kCh, smem_desc_k(ring + s * kTile + 32 * k),
                                 smem_desc_k(wt + tap * kWTap + 32 * k), instr_desc(kRows, kCh), tap > 0 || k > 0);
                    mma_commit(smem_u32(&empty[s]));
                }
                if (ok) mma_commit(smem_u32(&acc_full[acc]));
            }
            if (!ok) failed = 1;
        }
        __syncwarp();
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
        for (int j = issued > kStages ? issued - kStages : 0; j < issued; ++j) {
            mbar_wait(smem_u32(&full[j % kStages]), (uint32_t)((j / kStages) & 1));
            mbar_wait(smem_u32(&empty[j % kStages]), (uint32_t)((j / kStages) & 1), 1 << 16);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_free(tmem, kTmemCols);
}

// Rows of 64 channels [rows][64], boxes of box_rows rows.
bool rows_map(CUtensorMap* m, const void* ptr, long long rows, int box_rows)
{
    const cuuint64_t dim[2] = {kCh, (cuuint64_t)rows}, stride[1] = {kCh * 2};
    const cuuint32_t box[2] = {kCh, (cuuint32_t)box_rows}, step[2] = {1, 1};
    return encode_map(m, ptr, 2, dim, stride, box, step);
}

// A layer's weights [64][K], boxes of 64 x 64.
bool weight_map(CUtensorMap* m, const void* ptr, int K)
{
    const cuuint64_t dim[2] = {(cuuint64_t)K, kCh}, stride[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {kCh, kCh}, step[2] = {1, 1};
    return encode_map(m, ptr, 2, dim, stride, box, step);
}

// Activations [B][side][side][64] read at every step-th pixel: boxes of `positions`
// consecutive positions of the (side / step)^2 grid.
bool grid_map(CUtensorMap* m, const void* ptr, int B, int side, int step_, int positions)
{
    const int so = side / step_;
    const int rows = positions < so * so ? positions / so : so, patches = positions / (rows * so);
    const cuuint64_t dim[4] = {kCh, (cuuint64_t)side, (cuuint64_t)side, (cuuint64_t)B};
    const cuuint64_t stride[3] = {kCh * 2, (cuuint64_t)side * kCh * 2, (cuuint64_t)side * side * kCh * 2};
    const cuuint32_t box[4] = {kCh, (cuuint32_t)(so * step_), (cuuint32_t)(rows * step_), (cuuint32_t)patches};
    const cuuint32_t step[4] = {1, (cuuint32_t)step_, (cuuint32_t)step_, 1};
    return encode_map(m, ptr, 4, dim, stride, box, step);
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
        if (!weight_map(&tw, w, kTaps * kCh) || !grid_map(&tx, x, B, side, 2, kRows)) return PS_ERR_CUDA;
        PS_CUDA_CHECK(set_smem((const void*)k_conv_inner, inner_smem()));
        const int n_tiles = (int)(P / kRows);
        InnerArgs a{bias, n_tiles, so, d_err};
        k_conv_inner<<<n_tiles < sms ? n_tiles : sms, kInnerThreads, inner_smem(), st>>>(tx, tw, ty, a);
    }
    PS_LAUNCH_CHECK();
    return PS_OK;
}
