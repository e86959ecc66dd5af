// Documents the screen cannot help with (screen.cuh): evaluated against all units, exactly, by the whole
// chip.  The verify stage hands over those with more candidate groups than screen_dense_groups -- exact
// or near ties all over the map, as after an epoch with a wide neighbourhood, weights the 8-bit image does
// not resolve, lists too long for its sums -- and those without any candidate (distances that are not
// finite).  Where most of a sample of the documents would come here, all do, and nothing is screened.
//
// A warp takes a document and a piece of 256 units (128 where rows are not whole 16-byte pieces): every
// lane owns eight of them and adds its part of each listed row of W, fp32 sums in the row's order, ids
// through shared memory.  Pieces outside, documents inside, so that all warps in flight share one piece or
// two: rows of W in L2, those of frequent features in L1 (two or four pieces per warp, a quarter slower).  Keys meet in the per-document state; the
// warp that arrives last at a document (a ticket each) writes its outputs.
//
// Bound by the L2 -> SM path, less what L1 holds: all of 50,000 documents of 80 ids on 4,096 units take 2.6
// ms (6.2e12 updates/s), on 16,384 units 12 (5.4e12); the planned kernel with ids packed and sorted by a
// tiling pass makes 6.7 and 6.9e12.  Five blocks of four warps, or four units per lane: 5-20 % slower.
#include "screen.cuh"

#include <cuda_fp16.h>
#include <math_constants.h>

#include <type_traits>

namespace bmu {

static const int DENSE_WARPS = 16, DENSE_BLOCKS = 2;         // warps per block, blocks per SM

// adds sixteen bytes of a row: four fp32 or eight fp16 weights
__device__ __forceinline__ void dense_add16(u64 *acc, const ulonglong2 v, float)
{
    add2(acc[0], v.x);
    add2(acc[1], v.y);
}
__device__ __forceinline__ void dense_add16(u64 *acc, const ulonglong2 v, __half)
{
    const uint32_t x[4] = {(uint32_t)v.x, (uint32_t)(v.x >> 32), (uint32_t)v.y, (uint32_t)(v.y >> 32)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 t = __half22float2(*reinterpret_cast<const __half2 *>(&x[i]));
        add2(acc[i], ((u64)__float_as_uint(t.y) << 32) | __float_as_uint(t.x));
    }
}
__device__ __forceinline__ float dense_ld(const float *p) { return __ldg(p); }
__device__ __forceinline__ float dense_ld(const __half *p) { return __half2float(__ldg(p)); }

template <typename WT, bool TOP2, bool VEC>
__global__ void __launch_bounds__(DENSE_WARPS * 32, DENSE_BLOCKS)
screen_dense_kernel(const VerifyArgs a)
{
    constexpr int V16 = 16 / (int)sizeof(WT);                // weights in sixteen bytes
    constexpr int NL = VEC ? 8 / V16 : 4, STEP = VEC ? V16 : 1;      // loads per row, units per load
    constexpr int V = NL * STEP, ROWS = VEC ? 8 : 4;         // units per lane, rows in flight
    using Load = typename std::conditional<VEC, ulonglong2, float>::type;
    __shared__ uint4 s_ids[DENSE_WARPS][16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *mine = reinterpret_cast<uint32_t *>(s_ids[warp]);
    const uint32_t stride = (uint32_t)a.M * (uint32_t)sizeof(WT);        // (M < 2^30)
    asm volatile("griddepcontrol.wait;" ::: "memory");       // for the verify stage, under whose end it is launched
    if (__shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(a.status), 0)) return;
    const bool whole = screen_whole(a.scalars);              // all documents, in the planned order
    const int64_t docs = whole ? a.N : (int64_t)*a.dense_count, warps = (int64_t)gridDim.x * DENSE_WARPS;
    if (docs == 0) return;
    const int64_t pieces = (a.M + 32 * V - 1) / (32 * V);
    for (int64_t item = (int64_t)blockIdx.x * DENSE_WARPS + warp; item < docs * pieces; item += warps) {
        const int64_t at = item % docs, p = whole ? at : (int64_t)a.dense[at];
        const int64_t j0 = item / docs * (32 * V);
        const int32_t orig = a.perm[p];
        const int beg = __ldg(a.rowptr + orig), end = __ldg(a.rowptr + orig + 1);
        Best<TOP2> best;
        best.init();
        // where the lane's loads start; beyond the last unit they repeat it (and count for nothing)
        const WT *col[NL];
#pragma unroll
        for (int l = 0; l < NL; ++l)
            col[l] = static_cast<const WT *>(a.W) + min(j0 + (32 * l + lane) * STEP, a.M - STEP);
        u64 acc[(V + 1) / 2];
        float one[V];
#pragma unroll
        for (int v = 0; v < V; ++v) { acc[v / 2] = 0ull; one[v] = 0.f; }
        // rows q .. of the ids at hand: ROWS of them if full, else those below c
        auto rows = [&](int q, int c, auto full) {
            uint4 f4[ROWS / 4];
#pragma unroll
            for (int k = 0; k < ROWS / 4; ++k) f4[k] = s_ids[warp][q / 4 + k];
            Load w[ROWS][NL];
#pragma unroll
            for (int u = 0; u < ROWS; ++u)
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    w[u][l] = Load();
                    if (decltype(full)::value || q + u < c) {
                        const uint4 t = f4[u / 4];
                        const uint32_t f = u % 4 == 0 ? t.x : u % 4 == 1 ? t.y : u % 4 == 2 ? t.z : t.w;
                        const char *from = reinterpret_cast<const char *>(col[l]) + (u64)f * stride;
                        if constexpr (VEC) w[u][l] = __ldg(reinterpret_cast<const ulonglong2 *>(from));
                        else w[u][l] = dense_ld(reinterpret_cast<const WT *>(from));
                    }
                }
#pragma unroll
            for (int u = 0; u < ROWS; ++u)
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    if constexpr (VEC) dense_add16(acc + l * STEP / 2, w[u][l], WT());
                    else one[l] += w[u][l];
                }
        };
        for (int eb = beg; eb < end; eb += 64) {
            const int c = min(64, end - eb);
            __syncwarp();                                // the ids before these have been used
#pragma unroll
            for (int k = 0; k < 2; ++k)
                mine[32 * k + lane] = 32 * k + lane < c ? BMU_IDX((uint32_t)__ldg(a.colidx + eb + 32 * k + lane), a.D, a.status) : 0u;
            __syncwarp();
            int q = 0;
            for (; q + ROWS <= c; q += ROWS) rows(q, c, std::true_type());
            if (q < c) rows(q, c, std::false_type());
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int64_t j = j0 + (32 * (v / STEP) + lane) * STEP + v % STEP;
            const float sum = !VEC ? one[v] : v % 2 ? hi_f(acc[v / 2]) : lo_f(acc[v / 2]);
            if (j < a.M) best.push(fmaf(-2.f, sum, __ldg(a.norms + j)), (int)j);
        }
        u64 k1, k2;
        best.warp_keys(k1, k2);
        if (lane == 0) {
            // whatever is not the smallest key so far goes on to the second-best one
            const u64 old = atomicMin(a.state + orig, k1);
            if (TOP2) {
                const u64 loser = old > k1 ? old : k1;
                atomicMin(a.state2 + orig, loser < k2 ? loser : k2);
            }
            __threadfence();
            if (atomicAdd(a.lcount + p, 1u) == (uint32_t)pieces - 1) {
                __threadfence();
                const float nx = (float)(end - beg);
                k1 = __ldcg(a.state + orig);
                a.out_bmu[orig] = (int32_t)(uint32_t)k1;
                a.out_dist[orig] = nx + ordered_to_float((uint32_t)(k1 >> 32));
                if (TOP2) {
                    k2 = __ldcg(a.state2 + orig);
                    const bool none = (uint32_t)k2 >= 0x7fffffffu;       // a map of one unit
                    a.out_bmu2[orig] = none ? -1 : (int32_t)(uint32_t)k2;
                    a.out_dist2[orig] = none ? CUDART_INF_F : nx + ordered_to_float((uint32_t)(k2 >> 32));
                }
            }
        }
        __syncwarp();
    }
}

// Launched under the end of the verify stage, which rarely leaves it anything, as that is under the end of
// the last collection: with ordinary launches of both a search took 5-7 us more than without this one.
template <typename WT>
static cudaError_t launch_dense(const VerifyArgs &a, bool top2, const cudaLaunchConfig_t &c)
{
    if (screen_vec(a))
        return top2 ? cudaLaunchKernelEx(&c, screen_dense_kernel<WT, true, true>, a)
                    : cudaLaunchKernelEx(&c, screen_dense_kernel<WT, false, true>, a);
    return top2 ? cudaLaunchKernelEx(&c, screen_dense_kernel<WT, true, false>, a)
                : cudaLaunchKernelEx(&c, screen_dense_kernel<WT, false, false>, a);
}

int launch_screen_dense(const VerifyArgs &a, bool top2, int sms, cudaStream_t s)
{
    ScreenLaunch l((unsigned)(sms * DENSE_BLOCKS), DENSE_WARPS * 32, s, true);
    BMU_CUDA(a.f16 ? launch_dense<__half>(a, top2, l.c) : launch_dense<float>(a, top2, l.c));
    BMU_LAUNCHED();
    return BMU_OK;
}

}  // namespace bmu
