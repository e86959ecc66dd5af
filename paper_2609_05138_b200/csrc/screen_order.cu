// The order of the units of a two-stage search (screen.cuh): whether its slabs follow the norms, and the units
// by ascending norm as far as a document reaches.
//
// One block.  The units and the sets of 128 documents are counted in SC_BINS steps between the smallest norm and the
// largest; from the two follow what the sweeps of both orders take, and up to which reach a set should be swept
// by norm.  Then the units up to there are counted once more in finer steps, dropped at their places, and each
// step -- a few units -- is sorted by counting.  (norm, unit) is unique, so the order does not depend on how the
// threads ran.  Where the norms promise nothing the kernel stops after the first counting.  Bound by the latency of one
// block: 8 us for 5,625 units, 14 where 4,096 are sorted.
#include "screen.cuh"

#include <math_constants.h>

namespace bmu {

static const int ORDER_THREADS = 1024;
static const uint32_t ORDER_STEP_MAX = 256;          // units in one fine step, at most
// What it costs, in ns of the whole chip: a slab for a set of documents, in the order of the map and of the norms
// (whose candidates are looked up once more), and to begin with a set; 10^-3 ns a weight of an image, in the order of
// the map and, read alone or with its neighbours, of the norms.  (30 .. 50 ns a slab measured, by the length of the lists;
// 0.85, 17 and 5.5 ps a weight.)
static const float ORDER_SLAB = 40.f, ORDER_SLAB_BY_NORM = 46.f, ORDER_SET = 30.f;
static const float ORDER_BESIDE = 30000.f;
// ... and 10^-3 ns for a unit and a document that is evaluated whole.  Such documents are few here and come with the
// codebook's latency from DRAM: 60,000 documents on fp16 256 x 256 2,962 us so, 3,008 at 15 and 3,043 at 34, 120,000 on
// 64 x 64 840, 860 and 830, 100,000 on 512 x 512 12.84, 12.88 and 13.05 ms.
static const float ORDER_WHOLE = 26.f;
static const float ORDER_IMAGE = 0.9f, ORDER_IMAGE_ALONE = 12.f, ORDER_IMAGE_NEAR = 5.5f;

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
screen_order_kernel(const float *__restrict__ norms, int64_t D, int64_t M, int64_t N, int64_t launches, int32_t cap, float *scalars,
                    const float *earlier, const uint32_t *status, const uint32_t *set_reach, int sets,
                    int32_t *__restrict__ units, float *__restrict__ unit_norm, u64 *__restrict__ tmp,
                    int32_t *__restrict__ rank_of, int2 *__restrict__ picks, uint32_t *__restrict__ tickets,
                    uint32_t *__restrict__ nat_list)
{
    static_assert(SC_BINS == 4 * ORDER_THREADS, "four steps a thread");
    __shared__ uint32_t bins[SC_BINS], s_sets[SC_BINS], s_warp[32], s_most, s_kept, s_far, s_within, s_cursor[SC_MAX_LAUNCHES];
    __shared__ u64 s_best;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    uint32_t *sc = reinterpret_cast<uint32_t *>(scalars);
    const int lane = threadIdx.x & 31;
    const ScreenSteps steps(scalars);
    if (screen_whole(scalars) || !(steps.top > steps.lo) || !(steps.top < CUDART_INF_F)) return;
    const bool ordered_before = earlier && screen_ordered(earlier), codes = scalars[3] != 0.f, map_stands = scalars[7] == 0.f;
    for (int b = threadIdx.x; b < SC_BINS; b += ORDER_THREADS) bins[b] = s_sets[b] = 0u;
    if (threadIdx.x == 0) { s_most = s_far = 0u; s_best = ~0ull; }
    __syncthreads();
    order_units(norms, M, [&](int64_t, float n) {
        if (n >= steps.lo && n <= steps.top) atomicAdd(bins + steps.of(n), 1u);
        else if (n < steps.lo) s_most = 0xffffffffu;         // a unit at minus infinity
    });
    for (int i = threadIdx.x; i < sets; i += ORDER_THREADS) {
        const uint32_t v = set_reach[i];
        if (v == 0u) continue;                               // none of its documents needs a slab
        const float t = ordered_to_float(v);
        atomicAdd(t < steps.top ? s_sets + steps.of(t) : &s_far, 1u);
    }
    __syncthreads();
    // sets and their slabs up to each step, and what both sweeps and images would take
    const int all = (int)((M + SC_SLAB - 1) / SC_SLAB);
    uint32_t d4[4], slabs4[4], below = 0, within = 0, swept = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) { slabs4[i] = bins[4 * threadIdx.x + i]; below += slabs4[i]; }
    below = order_scan(below, s_warp);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        below += slabs4[i];
        slabs4[i] = (below + SC_SLAB - 1) / SC_SLAB;
        d4[i] = s_sets[4 * threadIdx.x + i];
        within += d4[i]; swept += d4[i] * slabs4[i];
    }
    within = order_scan(within, s_warp);
    swept = order_scan(swept, s_warp);
    const uint32_t mine = d4[0] + d4[1] + d4[2] + d4[3];
    if (threadIdx.x == ORDER_THREADS - 1) s_within = within + mine;
    __syncthreads();
    const uint32_t total = s_within + s_far;
    const uint4 docs = reinterpret_cast<const uint4 *>(status + STATUS_REACH)[threadIdx.x];
    const uint32_t n4[4] = {docs.x, docs.y, docs.z, docs.w};
    uint32_t docs_in = order_scan(docs.x + docs.y + docs.z + docs.w, s_warp);
    const float near = fminf(1.f, 0.016f * (float)M * (float)launches / (float)(all * SC_SLAB));
    const float image = (float)D * (float)SC_SLAB * (ORDER_IMAGE_NEAR + ORDER_IMAGE_ALONE * near) * 1e-3f;
    const float map_image = map_stands ? 0.f : (float)D * (float)M * ORDER_IMAGE * 1e-3f;
    const uint32_t made = ordered_before && codes ? (reinterpret_cast<const uint32_t *>(earlier)[SC_KEPT] + SC_SLAB - 1) / SC_SLAB : 0u;
    u64 best = ~0ull;
    // up to a step; what reaches further in the order of the map, by sets, or evaluated whole, by documents
    auto offer = [&](int step, uint32_t slabs, uint32_t n, uint32_t n_slabs, uint32_t n_docs) {
        if (slabs > (uint32_t)cap) return;
        const float first = (slabs <= made ? 0.f : (float)slabs * image) + (float)n_slabs * ORDER_SLAB_BY_NORM + (float)n * ORDER_SET;
        const float rest = (float)(total - n);
        const float map = first + (total > n ? map_image + rest * (float)all * ORDER_SLAB : 0.f);
        const float whole = first + rest * ((float)slabs * ORDER_SLAB_BY_NORM + ORDER_SET) + (float)(N - n_docs) * (float)M * (ORDER_WHOLE * 1e-3f);
        best = min(best, (u64)__float_as_uint(fminf(map, whole)) << 32 | (uint32_t)(2 * step + (whole < map)));
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        within += d4[i]; swept += d4[i] * slabs4[i]; docs_in += n4[i];
        if (d4[i] | n4[i]) offer(4 * threadIdx.x + i, slabs4[i], within, swept, docs_in);
    }
    if (threadIdx.x == ORDER_THREADS - 1) offer(SC_BINS, all, total, swept + s_far * all, (uint32_t)N);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, m));
    if (lane == 0) atomicMin(&s_best, best);
    __syncthreads();
    // (in favour of the one order: what the other costs beside it, and a sixth)
    const float natural = map_image + (float)total * (float)all * ORDER_SLAB;
    if (s_most || s_best == ~0ull || 1.2f * __uint_as_float((uint32_t)(s_best >> 32)) + ORDER_BESIDE > natural) return;
    const int cut = (int)((uint32_t)s_best >> 1);
    const bool whole = s_best & 1u;
    const float top = cut == SC_BINS ? CUDART_INF_F : steps.lo + (float)(cut + 1) * ((steps.top - steps.lo) / (float)SC_BINS);
    const float hi = fminf(top, steps.top);
    const bool keep = ordered_before && hi <= earlier[SC_SORTED];
    uint32_t kept = keep ? reinterpret_cast<const uint32_t *>(earlier)[SC_KEPT] : 0u;
    if (!keep) {
        const ScreenSteps fine(steps.lo, hi > steps.lo ? hi : steps.top);
        for (int b = threadIdx.x; b < SC_BINS; b += ORDER_THREADS) bins[b] = 0u;
        __syncthreads();
        order_units(norms, M, [&](int64_t, float n) { if (n <= hi) atomicAdd(bins + fine.of(n), 1u); });
        __syncthreads();
        uint32_t most = 0, u4[4];
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
        kept = s_kept;
        if (s_most > ORDER_STEP_MAX || kept > (uint32_t)cap * SC_SLAB) return;
        const uint32_t needed = (kept + SC_SLAB - 1) / SC_SLAB;
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
    }
    // the sets that reach further, in their order
    uint32_t n_nat = 0;
    for (int i0 = 0; i0 < sets; i0 += ORDER_THREADS) {
        const uint32_t v = i0 + (int)threadIdx.x < sets ? set_reach[i0 + threadIdx.x] : 0u;
        const bool far = v != 0u && !whole && !(ordered_to_float(v) <= top);
        const uint32_t at = order_scan(far, s_warp);
        if (far) nat_list[n_nat + at] = i0 + threadIdx.x;
        __syncthreads();
        if (threadIdx.x == ORDER_THREADS - 1) s_far = at + far;
        __syncthreads();
        n_nat += s_far;
    }
    for (int64_t i = threadIdx.x; i < launches * (SC_PARTS + 1); i += ORDER_THREADS) tickets[i] = 0u;
    if (threadIdx.x == 0) {
        sc[SC_ORDERED] = 1u; sc[SC_KEPT] = kept; sc[SC_NEEDED] = (kept + SC_SLAB - 1) / SC_SLAB;
        scalars[SC_TOP] = whole ? CUDART_INF_F : top; scalars[SC_DOC_TOP] = whole ? top : CUDART_INF_F;
        scalars[SC_SORTED] = keep ? earlier[SC_SORTED] : hi;
        sc[SC_STAND] = keep && codes;
        sc[SC_NAT] = n_nat; sc[SC_NATMADE] = n_nat > 0 || map_stands;
    }
}

// All of the map swept in its own order takes no more than the other costs beside it: the kernel would say so for every
// codebook (4,000 documents on 1,024 units, D = 4,096: 105 us with its launches, 95 without them).
bool screen_order_possible(int64_t D, int64_t M, int64_t N)
{
    const double sets = (double)((N + SC_DOCS - 1) / SC_DOCS), slabs = (double)((M + SC_SLAB - 1) / SC_SLAB);
    return M >= SC_ORDER_MIN && 1e-3 * ORDER_IMAGE * (double)D * (double)M + ORDER_SLAB * sets * slabs > 0.999 * ORDER_BESIDE;
}

int launch_screen_order(const float *norms, int64_t D, int64_t M, int64_t N, int64_t launches, char *cb,
                        const ScreenLayout &cl, float *scalars, const float *earlier, const uint32_t *status,
                        const uint32_t *set_reach, int sets, uint32_t *tickets, uint32_t *nat_list, cudaStream_t s)
{
    const int64_t slabs = (M + SC_SLAB - 1) / SC_SLAB, q = slabs / launches, rem = slabs % launches, k = cl.ord_launches;
    ScreenLaunch l(1, ORDER_THREADS, s, true);
    BMU_CUDA(cudaLaunchKernelEx(
        &l.c, screen_order_kernel, norms, D, M, N, launches, (int32_t)(k * q + (k < rem ? k : rem)), scalars, earlier, status,
        set_reach, sets, reinterpret_cast<int32_t *>(cb + cl.units), reinterpret_cast<float *>(cb + cl.unit_norm),
        reinterpret_cast<u64 *>(cb + cl.unit_tmp), reinterpret_cast<int32_t *>(cb + cl.rank_of),
        reinterpret_cast<int2 *>(cb + cl.picks), tickets, nat_list));
    BMU_LAUNCHED();
    return BMU_OK;
}

}  // namespace bmu
