// The order of the units of a two-stage search (screen.cuh): whether its slabs follow the norms, and the units
// by ascending norm as far as a document reaches.
//
// One block.  Documents (screen_window_kernel counted them) and units are counted in SC_BINS steps between the
// smallest norm and the largest; from the two follow the work of a sweep in that order and how far the slabs
// should go: a few documents that reach much further than the rest are better evaluated whole than have
// everybody's slabs made for them.  Then the units up to there are counted once more in finer steps, dropped at their
// places, and each step -- a few units -- is sorted by counting.  (norm, unit) is unique, so the order does not
// depend on how the threads ran.  Where it promises nothing the kernel stops after the first counting and the slabs
// follow the map.  Bound by the latency of one block.
#include "screen.cuh"

#include <math_constants.h>

namespace bmu {

static const int ORDER_THREADS = 1024;
static const uint32_t ORDER_STEP_MAX = 256;          // units in one fine step, at most
// Costs in units of one (document, unit) pair of the sweep, 2.5 ps.  A pair of a document that is evaluated whole
// (screen_dense.cu, 15 ps); a weight of a slab's image that is read alone (17 ps, scattered sectors) or as a part of
// whole rows (0.6 ps per weight of the map and launch of 26 slabs).
static const float ORDER_WHOLE = 6.f, ORDER_ALONE = 6.7f, ORDER_ROWS = 0.0095f;
// The largest share of a full sweep that one by norm may cost: a block goes as far as the furthest of its 128
// documents, its slabs' candidates are single units, and it gains from nothing that a map's neighbours share.
static const float ORDER_SHARE = 0.4f;

__device__ __forceinline__ uint32_t order_scan(uint32_t v, uint32_t *s_warp)      // exclusive, over the block
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, inc, m);
        if (lane >= m) inc += x;
    }
    __syncthreads();
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    return inc - v + __reduce_add_sync(0xffffffffu, lane < warp ? s_warp[lane] : 0u);
}

// f(unit, norm) for all units, those of 4,096 at a time before the next
template <typename F>
__device__ __forceinline__ void order_units(const float *__restrict__ norms, int64_t M, F f)
{
    if ((reinterpret_cast<uintptr_t>(norms) & 15) == 0) {
        const int64_t n4 = M / 4;
#pragma unroll 2
        for (int64_t i = threadIdx.x; i < n4; i += ORDER_THREADS) {
            const float4 t = __ldg(reinterpret_cast<const float4 *>(norms) + i);
            f(4 * i, t.x); f(4 * i + 1, t.y); f(4 * i + 2, t.z); f(4 * i + 3, t.w);
        }
        if (4 * n4 + threadIdx.x < M) f(4 * n4 + threadIdx.x, __ldg(norms + 4 * n4 + threadIdx.x));
    } else {
        for (int64_t j = threadIdx.x; j < M; j += ORDER_THREADS) f(j, __ldg(norms + j));
    }
}

__global__ void __launch_bounds__(ORDER_THREADS)
screen_order_kernel(const float *__restrict__ norms, int64_t D, int64_t M, int64_t N, int64_t launches,
                    const uint32_t *__restrict__ status, float *scalars, const float *__restrict__ earlier, int shared,
                    int32_t *__restrict__ units, float *__restrict__ unit_norm, u64 *__restrict__ tmp,
                    int32_t *__restrict__ rank_of, int2 *__restrict__ picks, uint32_t *__restrict__ tickets)
{
    static_assert(SC_BINS == 4 * ORDER_THREADS, "four steps a thread");
    __shared__ uint32_t bins[SC_BINS], s_warp[32], s_most, s_kept, s_cursor[SC_MAX_LAUNCHES];
    __shared__ u64 s_best;
    uint32_t *sc = reinterpret_cast<uint32_t *>(scalars);
    const int lane = threadIdx.x & 31;
    const bool stand = scalars[7] == 0.f, followed = earlier && screen_ordered(earlier);
    const ScreenSteps steps(scalars, norms);
    __syncthreads();
    // (images in the order of the norms are of no use to slabs that follow the map)
    if (followed && threadIdx.x == 0) scalars[7] = 1.f;
    // (an earlier search of the same codebook has decided for this one too)
    if (screen_whole(scalars) || !(steps.top > steps.lo) || !(steps.top < CUDART_INF_F) || (earlier && !followed)) return;
    for (int b = threadIdx.x; b < SC_BINS; b += ORDER_THREADS) bins[b] = 0u;
    if (threadIdx.x == 0) { s_most = 0u; s_best = ~0ull; }
    __syncthreads();
    order_units(norms, M, [&](int64_t, float n) {
        if (n >= steps.lo && n <= steps.top) atomicAdd(bins + steps.of(n), 1u);
        else if (n < steps.lo) s_most = 0xffffffffu;         // a unit at minus infinity
    });
    __syncthreads();
    // how far to go: up to the end of a step, or all the way
    const uint4 docs = __ldg(reinterpret_cast<const uint4 *>(status + STATUS_REACH) + threadIdx.x);
    const uint32_t d4[4] = {docs.x, docs.y, docs.z, docs.w};
    uint32_t u4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u4[i] = bins[4 * threadIdx.x + i];
    uint32_t within = order_scan(d4[0] + d4[1] + d4[2] + d4[3], s_warp);
    uint32_t below = order_scan(u4[0] + u4[1] + u4[2] + u4[3], s_warp);
    const float slab_cost = (float)D * fminf(ORDER_ALONE * SC_SLAB, ORDER_ROWS * (float)M);
    const float whole_cost = ORDER_WHOLE * (float)M;
    u64 best = ~0ull;
    float work[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        within += d4[i]; below += u4[i];
        work[i] = (float)d4[i] * (float)below;
        const float cost = (float)((below + SC_SLAB - 1) / SC_SLAB) * slab_cost + (float)(N - within) * whole_cost;
        if (d4[i]) best = min(best, (u64)__float_as_uint(cost) << 32 | (uint32_t)(4 * threadIdx.x + i));
    }
    if (threadIdx.x == ORDER_THREADS - 1) {                  // all the way: no document is left over
        const float cost = (float)((M + SC_SLAB - 1) / SC_SLAB) * slab_cost;
        best = min(best, (u64)__float_as_uint(cost) << 32 | (uint32_t)SC_BINS);
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, m));
    if (lane == 0) atomicMin(&s_best, best);
    __syncthreads();
    int cut = (int)(uint32_t)s_best;
    bool keep = false;
    if (followed) {
        // the earlier order serves if it goes far enough
        const float old = earlier[SC_TOP];
        const int b = old >= steps.top ? SC_BINS : steps.of(old) - 1;
        if (b >= cut) { keep = true; cut = b; }
    }
    // the work up to there, and that of the documents left over
    float part = 0.f;
    uint32_t n_in = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) if (4 * (int)threadIdx.x + i <= cut) { part += work[i]; n_in += d4[i]; }
    n_in = __reduce_add_sync(0xffffffffu, n_in);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) part += __shfl_xor_sync(0xffffffffu, part, m);
    __syncthreads();
    if (lane == 0) { s_warp[threadIdx.x >> 5] = __float_as_uint(part); s_cursor[threadIdx.x >> 5] = n_in; }
    __syncthreads();
    part = 0.f;
    n_in = 0u;
    for (int w = 0; w < 32; ++w) { part += __uint_as_float(s_warp[w]); n_in += s_cursor[w]; }
    const float over = (float)(N - n_in) * (cut >= SC_BINS ? (float)M : whole_cost);
    if (!followed && part + over > ORDER_SHARE * (float)N * (float)M) return;
    if (s_most) return;
    for (int64_t i = threadIdx.x; i < launches * (SC_PARTS + 1); i += ORDER_THREADS) tickets[i] = 0u;
    if (keep) {
        if (threadIdx.x == 0) {
            const uint32_t kept = reinterpret_cast<const uint32_t *>(earlier)[SC_KEPT];
            sc[SC_KEPT] = kept; sc[SC_NEEDED] = (kept + SC_SLAB - 1) / SC_SLAB; sc[SC_TOP] = __float_as_uint(earlier[SC_TOP]);
            sc[SC_STAND] = stand ? 1u : 0u; sc[SC_ORDERED] = 1u;
        }
        return;
    }
    float hi = steps.top;
    if (cut < SC_BINS) hi = fminf(hi, steps.lo + (float)(cut + 1) * ((steps.top - steps.lo) / (float)SC_BINS));
    // (searches to come may reach a little further)
    if (shared) hi = fminf(steps.top, hi + 0.125f * (hi - steps.lo));
    const ScreenSteps fine(steps.lo, hi > steps.lo ? hi : steps.top);
    for (int b = threadIdx.x; b < SC_BINS; b += ORDER_THREADS) bins[b] = 0u;
    __syncthreads();
    order_units(norms, M, [&](int64_t, float n) { if (n <= hi) atomicAdd(bins + fine.of(n), 1u); });
    __syncthreads();
    uint32_t most = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) { u4[i] = bins[4 * threadIdx.x + i]; most = max(most, u4[i]); }
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0) atomicMax(&s_most, most);
    uint32_t run = order_scan(u4[0] + u4[1] + u4[2] + u4[3], s_warp);
#pragma unroll
    for (int i = 0; i < 4; ++i) { bins[4 * threadIdx.x + i] = run; run += u4[i]; }
    if (threadIdx.x == ORDER_THREADS - 1) s_kept = run;
    for (int64_t i = threadIdx.x; i < launches; i += ORDER_THREADS) s_cursor[i] = 0u;
    __syncthreads();
    if (s_most > ORDER_STEP_MAX) return;
    const uint32_t kept = s_kept, needed = (kept + SC_SLAB - 1) / SC_SLAB;
    order_units(norms, M, [&](int64_t j, float n) {
        if (n <= hi) tmp[atomicAdd(bins + fine.of(n), 1u)] = make_key(n, (int32_t)j);
    });
    __syncthreads();
    // (now bins[b] is where step b ends, that is where b + 1 begins)
    for (uint32_t x = threadIdx.x; x < needed * SC_SLAB; x += ORDER_THREADS) {
        if (x >= kept) { units[x] = -1; unit_norm[x] = CUDART_INF_F; picks[x] = make_int2(-1, (int)x); continue; }
        const u64 mine = tmp[x];
        const float n = ordered_to_float((uint32_t)(mine >> 32));
        const int b = fine.of(n);
        const uint32_t beg = b ? bins[b - 1] : 0u, end = bins[b];
        uint32_t at = beg;
        for (uint32_t y = beg; y < end; ++y) at += tmp[y] < mine;
        units[at] = (int32_t)(uint32_t)mine;
        unit_norm[at] = n;
        rank_of[(uint32_t)mine] = (int32_t)at;
    }
    __syncthreads();
    // the units of each launch, nearly in the order of the map
    const int64_t slabs = (M + SC_SLAB - 1) / SC_SLAB, q = slabs / launches, rem = slabs % launches;
    order_units(norms, M, [&](int64_t j, float n) {
        if (!(n <= hi)) return;
        const int32_t r = rank_of[j];
        const int s = r / SC_SLAB, k = launches == 1 ? 0 : (int)(s < rem * (q + 1) ? s / (q + 1) : rem + (s - rem * (q + 1)) / q);
        const int64_t slab0 = k * q + (k < rem ? k : rem);
        picks[slab0 * SC_SLAB + atomicAdd(s_cursor + k, 1u)] = make_int2((int)j, r);
    });
    if (threadIdx.x == 0) {
        sc[SC_KEPT] = kept; sc[SC_NEEDED] = needed; sc[SC_TOP] = __float_as_uint(hi);
        sc[SC_STAND] = 0u; sc[SC_ORDERED] = 1u;
    }
}

int launch_screen_order(const float *norms, int64_t D, int64_t M, int64_t N, int64_t launches, char *cb,
                        const ScreenLayout &cl, float *scalars, const float *earlier, bool shared,
                        const uint32_t *status, uint32_t *tickets, cudaStream_t s)
{
    { screen_order_kernel<<<1, ORDER_THREADS, 0, s>>>(
        norms, D, M, N, launches, status, scalars, earlier, shared, reinterpret_cast<int32_t *>(cb + cl.units),
        reinterpret_cast<float *>(cb + cl.unit_norm), reinterpret_cast<u64 *>(cb + cl.unit_tmp),
        reinterpret_cast<int32_t *>(cb + cl.rank_of), reinterpret_cast<int2 *>(cb + cl.picks), tickets); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

}  // namespace bmu
