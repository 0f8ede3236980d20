// ps_step.cu -- one optimisation step (Sec. 3.3) enqueued by one call.
//
// The step is project, bin, fused splat, chain, Adam, each with something small before or
// after it: the schedule's advance, zeroed counts, accumulators and gradients.  Where lists
// are short those launches and the gaps between them are a tenth of a step, and an eager step
// of a small scene is bound by the host that enqueues them.  So k_begin advances the schedule
// and zeroes everything the step accumulates into, the projection leaves the binning's counts,
// and k_chain_adam takes the records' gradients to the world parameters and updates them: 8
// launches instead of 13.  64 planes in 8 views of 128x96, eager, by events: 162 us by nine calls,
// 62 by one call of the same launches, 39 now (launches overlapped as in launch_after; a step
// among others from Python takes 50-57, bound by the host); 3,000 planes in 8 views of 640x480 at
// lambda 300, replayed from a graph: 171 -> 167 us, 158 with the loads of k_chain_adam ahead of
// its chain and the splat's grouped strips.
#include <math.h>

#include "ps_internal.cuh"

using namespace ps;

namespace {

struct BeginArgs {
    uint4* zero[2];          // 16-byte aligned ranges and their lengths in 16 bytes
    long long n[2];
    float* zero_f;           // a range of floats
    long long n_f;
    ps_step_state* state;    // schedule: *state = sched[min(*iter, n_sched - 1)], ++*iter
    const ps_step_state* sched;
    int n_sched;
    int* iter;
};

__global__ void __launch_bounds__(256) k_begin(BeginArgs a)
{
    after_previous();
    const long long t = (long long)blockIdx.x * 256 + threadIdx.x, stride = (long long)gridDim.x * 256;
#pragma unroll
    for (int r = 0; r < 2; ++r)
        for (long long i = t; i < a.n[r]; i += stride) a.zero[r][i] = make_uint4(0u, 0u, 0u, 0u);
    for (long long i = t; i < a.n_f; i += stride) a.zero_f[i] = 0.f;
    if (a.sched && t == 0) {
        const int i = *a.iter;
        *a.state = a.sched[i < a.n_sched ? i : a.n_sched - 1];
        *a.iter = i + 1;
    }
}

constexpr int kChainThreads = 128;
constexpr int kChainLanes = 8;                               // lanes per plane
constexpr int kChainPlanes = kChainThreads / kChainLanes;

struct ChainAdamArgs {
    const ps_view* views;
    int n_views, P;
    const float* g_rec;
    int gauss, single_radii;
    float *params, *grad, *m, *v;    // [center 3 P | quat 4 P | radii 4 P]
    float lr, b1, b2, eps, bc1, bc2, r_min;
    const ps_step_state* d_state;    // if set, bc1 and bc2 come from here
    const double* vs_slots;
    double* view_sums;
    int plane_blocks;                // blocks of planes; the rest add up the views' loss sums
};

// Eight lanes per plane add up its records over the views of its scene (the centre's part by each
// view's rotation), one lane chains the sum, then the block writes its planes' gradients and updates their parameters in order of
// address.  grad holds the radii's direct part (pairs at P = 0) on entry.  Bound by the latency
// of its dependent loads, so what Adam reads is loaded before the chain.  3,000 planes in 8 views:
// 7.8 -> 5.6 us; 64 planes, a whole eager step 42 -> 37.
__global__ void __launch_bounds__(kChainThreads) k_chain_adam(ChainAdamArgs a)
{
    __shared__ float s_g[kChainPlanes][12];
    after_previous();
    if ((int)blockIdx.x >= a.plane_blocks) {
        const int t = ((int)blockIdx.x - a.plane_blocks) * kChainThreads + (int)threadIdx.x;
        if (t < 4 * a.n_views) a.view_sums[t] = slot_sum(a.vs_slots, t >> 2, t & 3);
        return;
    }
    const int p0 = blockIdx.x * kChainPlanes, at = threadIdx.x / kChainLanes, p = p0 + at;
    const int j = threadIdx.x % kChainLanes;
    // this thread's parameters: centres, then quaternions, then radii of the block's planes
    const int n = min(kChainPlanes, a.P - p0);
    constexpr int kPer = (11 * kChainPlanes + kChainThreads - 1) / kChainThreads;
    long long idx[kPer];
    float pv[kPer], mv[kPer], vv[kPer], gv[kPer];
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        const int t = threadIdx.x + e * kChainThreads;
        idx[e] = t < 3 * n ? 3LL * p0 + t
               : t < 7 * n ? 3LL * a.P + 4LL * p0 + t - 3 * n : 7LL * a.P + 4LL * p0 + t - 7 * n;
        if (t < 11 * n) {
            pv[e] = a.params[idx[e]]; mv[e] = a.m[idx[e]]; vv[e] = a.v[idx[e]];
            gv[e] = t < 7 * n ? 0.f : a.grad[idx[e]];
        }
    }
    // centre 3, moments 3, radii 4
    float g[10] = {};
    PlaneAxes ax;
    bool ok = false;
    if (p < a.P) {
        const float* q = a.params + 3 * (size_t)a.P + 4 * (size_t)p;
        ok = plane_axes(q[0], q[1], q[2], q[3], ax);
        // planes of a scene are consecutive and its views too: the last view whose planes start
        // at or before p is the last view of p's scene, if that scene has views at all
        int lo = 0, hi = a.n_views - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&a.views[mid].plane_off) <= p) lo = mid; else hi = mid - 1;
        }
        const int k = p - __ldg(&a.views[lo].plane_off), scene = __ldg(&a.views[lo].scene);
        if (k >= 0 && k < __ldg(&a.views[lo].K)) {
            for (int v = lo - j; v >= 0 && __ldg(&a.views[v].scene) == scene; v -= kChainLanes) {
                const size_t r = (size_t)__ldg(&a.views[v].rec_off) + k;
                const float4* q = reinterpret_cast<const float4*>(a.g_rec + r * grad_stride(a.gauss));
                const float4 x = q[0], y = q[1];
                // rectangle: every pair's gradient of P is that of its radius, negative on the + side
                float gax = y.x - y.y, gay = y.z - y.w;
                if (a.gauss) { const float4 z = q[2]; gax = z.x; gay = z.y; }
                float gc[3] = {g[0], g[1], g[2]};
                add_centre(gc, ax, x.x, gax, gay, a.views + v);
                g[0] = gc[0]; g[1] = gc[1]; g[2] = gc[2];
                g[3] += x.y; g[4] += x.z; g[5] += x.w;
                g[6] += y.x; g[7] += y.y; g[8] += y.z; g[9] += y.w;
            }
        }
    }
#pragma unroll
    for (int o = kChainLanes / 2; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 10; ++c) g[c] += __shfl_xor_sync(0xffffffffu, g[c], o);
    if (j == 0 && p < a.P) {
        float out[8];
        chain_turn(ax, g[3], g[4], g[5], make_float4(g[6], g[7], g[8], g[9]), a.single_radii, out);
#pragma unroll
        for (int c = 0; c < 11; ++c) s_g[at][c] = !ok ? 0.f : c < 3 ? g[c] : out[c - 3];
    }
    __syncthreads();
    const float bc1 = a.d_state ? a.d_state->bc1 : a.bc1, bc2 = a.d_state ? a.d_state->bc2 : a.bc2;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        const int t = threadIdx.x + e * kChainThreads;
        if (t >= 11 * n) continue;
        const int u = t < 3 * n ? 0 : t < 7 * n ? t - 3 * n : t - 7 * n;
        const float gi = t < 3 * n ? s_g[t / 3][t % 3]
                       : t < 7 * n ? s_g[u >> 2][3 + (u & 3)] : gv[e] + s_g[u >> 2][7 + (u & 3)];
        const long long i = idx[e];
        a.grad[i] = gi;
        adam_value(pv[e], mv[e], vv[e], gi, a.lr, a.b1, a.b2, a.eps, bc1, bc2, t < 7 * n ? -INFINITY : a.r_min);
        a.params[i] = pv[e]; a.m[i] = mv[e]; a.v[i] = vv[e];
    }
}

// Plane splitting's sums and Adam on the finished gradient, by the entry points.
ps_status adam_parameters(int n_planes, const ps_settings* s, const ps_fit_buffers* b, float lr, float b1, float b2,
                          float eps, float r_min, int step, ps_stream stream)
{
    const long long g = 7LL * n_planes, n = 11LL * n_planes;     // the radii's first value, all values
    ps_status e;
    if (b->split_acc) {
        e = ps_radii_grad_accum(b->grad + g, b->split_scale, 1.f, n_planes, b->split_acc, stream);
        if (e != PS_OK) return e;
    }
    if (s->d_state)
        return ps_adam_step_state(b->params, b->grad, b->m, b->v, n, lr, b1, b2, eps, s->d_state, r_min, g, stream);
    e = ps_adam_step(b->params, b->grad, b->m, b->v, g, lr, b1, b2, eps, step, NAN, stream);
    if (e != PS_OK) return e;
    return ps_adam_step(b->params + g, b->grad + g, b->m + g, b->v + g, n - g, lr, b1, b2, eps, step, r_min, stream);
}

// From so many records per plane on (the mean number of views of a scene) the chain goes record by
// record, as ps_splat_fused's does, and Adam by its own launches: eight lanes would walk a plane's
// views too long.  64 planes in views of 32x32, an eager step by k_chain_adam and by records: 64
// views 68 and 71 us, 128 80 and 78, 256 105 and 92, 1,024 242 and 176, 4,096 839 and 497.
constexpr int kManyViews = 128;

}  // namespace

extern "C" ps_status ps_fit_step(int n_planes, const ps_frame* frame, const ps_settings* s,
                                 const ps_fit_buffers* b, int fused, float lr, float b1, float b2,
                                 float eps, float r_min, int step, ps_stream stream)
{
    if (n_planes < 0 || !frame || !s || !b || !b->params || !b->grad || !b->m || !b->v || step < 1)
        return PS_ERR_ARG;
    if (b->d_sched && (!b->d_state || !b->d_iter || b->n_sched < 1)) return PS_ERR_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const size_t P = (size_t)n_planes;
    ps_planes pl{};
    pl.n_planes = n_planes;
    pl.center = b->params; pl.quat = b->params + 3 * P; pl.radii = b->params + 7 * P;
    float *gc = b->grad, *gq = b->grad + 3 * P, *gr = b->grad + 7 * P;
    // every argument first: nothing is launched, and the schedule not advanced, for a refused step
    ps_status e = check_project(&pl, frame, s, b->rec, b->rect, b->key);
    if (e != PS_OK) return e;
    e = check_bin(frame, s, b->rec, b->rect, b->key, b->tile_ptr, b->tile_ent, b->tile_key, b->capacity,
                  b->d_required, b->bin_ws, b->bin_ws_bytes);
    if (e != PS_OK) return e;
    if (fused) {
        if (!b->view_sums) return PS_ERR_ARG;
        e = check_fused(&pl, frame, s, b->rec, b->tile_key, b->tile_ptr, b->tile_ent, b->capacity, b->gt_depth,
                        b->gt_normal, gr, b->bwd_ws, b->bwd_ws_bytes);
    } else {
        e = check_fwd(frame, s, b->rec, b->tile_key, b->tile_ptr, b->tile_ent, b->capacity, b->depth, b->normal,
                      b->fwd_ws, b->fwd_ws_bytes);
        if (e != PS_OK) return e;
        e = check_loss(frame, s, b->depth, b->normal, b->gt_depth, b->gt_normal, b->dL_dD, b->dL_dN, b->view_sums);
        if (e != PS_OK) return e;
        e = check_bwd(&pl, frame, s, b->rec, b->tile_key, b->tile_ptr, b->tile_ent, b->capacity, b->dL_dD,
                      b->dL_dN, gc, gq, gr, b->bwd_ws, b->bwd_ws_bytes);
    }
    if (e != PS_OK) return e;
    if (fused) {
        BinCount count;
        FusedWs w;
        bin_count(frame, b->capacity, b->bin_ws, b->bin_ws_bytes, &count);
        fused_ws(frame, s, b->bwd_ws, b->bwd_ws_bytes, &w);
        BeginArgs a{};
        // (the counts' buffer is padded to 256 bytes, the splat's range is whole 16 bytes)
        a.zero[0] = reinterpret_cast<uint4*>(count.diff); a.n[0] = (count.n_tiles + 3) / 4;
        a.zero[1] = static_cast<uint4*>(b->bwd_ws); a.n[1] = (long long)(w.bytes / 16);
        const bool many = frame->n_records >= kManyViews * (long long)n_planes;
        a.zero_f = many ? b->grad : gr; a.n_f = (many ? 11LL : 4LL) * n_planes;
        a.state = b->d_state; a.sched = b->d_sched; a.n_sched = b->n_sched; a.iter = b->d_iter;
        const long long most = a.n[1] > a.n[0] ? a.n[1] : a.n[0];
        const long long blocks = (most + 255) / 256;
        k_begin<<<(unsigned)(blocks < 152 * 4 ? blocks : 152 * 4), 256, 0, st>>>(a);
        PS_LAUNCH_CHECK();
        if ((e = project(&pl, frame, s, b->rec, b->rect, b->key, &count, b->d_status, st)) != PS_OK) return e;
        e = bin_tiles(frame, s, b->rec, b->rect, b->key, b->tile_ptr, b->tile_ent, b->tile_key, b->capacity,
                      b->d_required, b->bin_ws, b->bin_ws_bytes, true, b->d_status, st);
        if (e != PS_OK) return e;
        e = splat_fused(&pl, frame, s, b->rec, b->tile_key, b->tile_ptr, b->tile_ent, b->capacity, b->gt_depth,
                        b->gt_normal, nullptr, nullptr, nullptr, nullptr, gr, b->bwd_ws, b->bwd_ws_bytes, true,
                        b->d_status, st);
        if (e != PS_OK) return e;
        if (many) {
            e = chain_fused(&pl, frame, s, b->view_sums, gc, gq, gr, b->bwd_ws, b->bwd_ws_bytes, st);
            return e == PS_OK ? adam_parameters(n_planes, s, b, lr, b1, b2, eps, r_min, step, stream) : e;
        }
        ChainAdamArgs c{};
        c.views = frame->views; c.n_views = frame->n_views; c.P = n_planes;
        c.g_rec = w.g_rec;
        c.gauss = (s->flags & PS_GAUSSIAN) ? 1 : 0; c.single_radii = (s->flags & PS_SINGLE_RADII) ? 1 : 0;
        c.params = b->params; c.grad = b->grad; c.m = b->m; c.v = b->v;
        c.lr = lr; c.b1 = b1; c.b2 = b2; c.eps = eps;
        c.bc1 = (float)(1.0 - pow((double)b1, (double)step));
        c.bc2 = (float)(1.0 - pow((double)b2, (double)step));
        c.r_min = isnan(r_min) ? -INFINITY : r_min;
        c.d_state = s->d_state;
        c.vs_slots = w.slots; c.view_sums = b->view_sums;
        c.plane_blocks = (n_planes + kChainPlanes - 1) / kChainPlanes;
        const int grid = c.plane_blocks + (4 * frame->n_views + kChainThreads - 1) / kChainThreads;
        PS_CUDA_CHECK(launch_after(k_chain_adam, grid, kChainThreads, 0, st, c));
        return b->split_acc ? ps_radii_grad_accum(gr, b->split_scale, 1.f, n_planes, b->split_acc, stream) : PS_OK;
    }
    if (b->d_sched) {
        e = ps_step_advance(b->d_state, b->d_sched, b->n_sched, b->d_iter, stream);
        if (e != PS_OK) return e;
    }
    e = ps_project_cull(&pl, frame, s, b->rec, b->rect, b->key, b->d_status, stream);
    if (e != PS_OK) return e;
    e = ps_bin_tiles(frame, s, b->rec, b->rect, b->key, b->tile_ptr, b->tile_ent, b->tile_key, b->capacity,
                     b->d_required, b->bin_ws, b->bin_ws_bytes, b->d_status, stream);
    if (e != PS_OK) return e;
    PS_CUDA_CHECK(cudaMemsetAsync(b->grad, 0, sizeof(float) * 11 * P, st));
    e = ps_splat_fwd(frame, s, b->rec, b->tile_key, b->tile_ptr, b->tile_ent, b->capacity, b->depth,
                     b->normal, nullptr, b->fwd_ws, b->fwd_ws_bytes, b->d_status, stream);
    if (e != PS_OK) return e;
    e = ps_loss(frame, s, b->depth, b->normal, b->gt_depth, b->gt_normal, b->dL_dD, b->dL_dN, b->view_sums,
                stream);
    if (e != PS_OK) return e;
    e = ps_splat_bwd(&pl, frame, s, b->rec, b->tile_key, b->tile_ptr, b->tile_ent, b->capacity, b->dL_dD,
                     b->dL_dN, gc, gq, gr, b->bwd_ws, b->bwd_ws_bytes, b->d_status, stream);
    if (e != PS_OK) return e;
    return adam_parameters(n_planes, s, b, lr, b1, b2, eps, r_min, step, stream);
}
