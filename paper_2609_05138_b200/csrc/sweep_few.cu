// The search of few documents (a service that maps what has just come in, a held-out handful):
// too few to fill the chip with a warp per document, and too few to repay a tiling pass.
//
// The grid is documents x pieces of the neuron axis.  A warp takes one document and one piece,
// 32 * V neurons at a time: every lane owns V of them and adds its piece of each listed row of W
// straight from the CSR, eight or sixteen rows in flight, fp32 sums in the row's order as in the generic
// kernel.  It leaves its best (and second-best) key in a slot of its own; the warp that arrives
// last at a document (a ticket per document) merges the slots and writes the outputs, so the whole
// search behind the norms is one clearing of the tickets and one launch.
//
// What bounds it: the L2 -> SM path once the pieces fill the SMs, the latency of one pass over a
// row's ids before that.  256 documents on a 128 x 128 map: 2074 -> 118 us per call (22
// launches of 16 blocks before); 48 documents on 32 x 32: 87 -> 19 us,
// half of them the norms.
#include "common.cuh"

#include <math_constants.h>

#include <type_traits>

namespace bmu {

static const int FEW_WARPS = 4;

// VEC: H 128-bit loads per lane and row (whole, aligned 16-byte pieces); else four 32-bit loads
// per lane, 32 neurons apart.
template <bool VEC, int H, bool TOP2>
__global__ void __launch_bounds__(FEW_WARPS * 32, H == 2 ? 5 : 4)
sweep_few_kernel(const FewArgs a)
{
    constexpr int V = VEC ? 4 * H : 4;               // neurons per lane and slab
    constexpr int ROWS = 64 / V;                     // rows in flight: 64 registers of weights
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * FEW_WARPS + (threadIdx.x >> 5);
    if (i >= a.N) return;
    const int beg = __ldg(a.rowptr + i), end = __ldg(a.rowptr + i + 1);
    const int64_t j_lo = (int64_t)blockIdx.y * a.piece, j_hi = min(j_lo + a.piece, a.M);
    Best<TOP2> best;
    best.init();
    for (int64_t j0 = j_lo; j0 < j_hi; j0 += 32 * V) {
        float acc[V];
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = 0.f;
        // where the lane's loads start; beyond the last neuron they repeat it (and count for nothing)
        constexpr int NL = VEC ? H : V;              // loads per row
        const float *col[NL];
#pragma unroll
        for (int l = 0; l < NL; ++l)
            col[l] = a.W + min(j0 + (VEC ? 128 * l + 4 * lane : 32 * l + lane), a.M - (VEC ? 4 : 1));
        auto rows = [&](int mine, int q, auto count) {
            constexpr int R = decltype(count)::value;
            float w[R][V];
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const uint32_t f = (uint32_t)__shfl_sync(0xffffffffu, mine, q + u);
                const int64_t off = (int64_t)BMU_IDX(f, a.D, a.status) * a.M;
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    if constexpr (VEC) {
                        const float4 t = __ldg(reinterpret_cast<const float4 *>(col[l] + off));
                        w[u][4 * l] = t.x; w[u][4 * l + 1] = t.y; w[u][4 * l + 2] = t.z; w[u][4 * l + 3] = t.w;
                    } else {
                        w[u][l] = __ldg(col[l] + off);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < R; ++u)
#pragma unroll
                for (int v = 0; v < V; ++v) acc[v] += w[u][v];
        };
        for (int eb = beg; eb < end; eb += 32) {
            const int mine = eb + lane < end ? __ldg(a.colidx + eb + lane) : 0;
            const int c = min(32, end - eb);
            int q = 0;
            for (; q + ROWS <= c; q += ROWS) rows(mine, q, std::integral_constant<int, ROWS>());
            if (ROWS > 8 && q + 8 <= c) { rows(mine, q, std::integral_constant<int, 8>()); q += 8; }
            if (ROWS > 4 && q + 4 <= c) { rows(mine, q, std::integral_constant<int, 4>()); q += 4; }
            for (; q < c; ++q) rows(mine, q, std::integral_constant<int, 1>());
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int64_t j = j0 + (VEC ? 128 * (v / 4) + 4 * lane + v % 4 : 32 * v + lane);
            if (j < j_hi) best.push(fmaf(-2.f, acc[v], __ldg(a.norms + j)), (int)j);
        }
    }
    u64 k1, k2;
    best.warp_keys(k1, k2);
    const int pieces = gridDim.y;
    if (pieces > 1) {
        u64 *slot = a.slots + (size_t)i * pieces * (TOP2 ? 2 : 1);
        bool last = false;
        if (lane == 0) {
            slot[(size_t)blockIdx.y * (TOP2 ? 2 : 1)] = k1;
            if (TOP2) slot[(size_t)blockIdx.y * 2 + 1] = k2;
            __threadfence();
            last = atomicAdd(a.tickets + i, 1u) == (uint32_t)pieces - 1;
        }
        if (!__shfl_sync(0xffffffffu, last, 0)) return;
        __threadfence();
        k1 = k2 = KEY_WORST;
        for (int s = lane; s < pieces; s += 32) {
            const u64 b1 = __ldcg(slot + (size_t)s * (TOP2 ? 2 : 1));
            if (TOP2) Best<true>::merge(k1, k2, b1, __ldcg(slot + (size_t)s * 2 + 1));
            else k1 = b1 < k1 ? b1 : k1;
        }
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) {
            const u64 o1 = __shfl_xor_sync(0xffffffffu, k1, m);
            if (TOP2) {
                const u64 o2 = __shfl_xor_sync(0xffffffffu, k2, m);
                Best<true>::merge(k1, k2, o1, o2);
            } else {
                k1 = o1 < k1 ? o1 : k1;
            }
        }
    }
    if (lane == 0) {
        const float nx = (float)(end - beg);
        a.out_bmu[i] = (int32_t)(uint32_t)k1;
        a.out_dist[i] = nx + ordered_to_float((uint32_t)(k1 >> 32));
        if (TOP2) {
            const bool none = (uint32_t)k2 >= 0x7fffffffu;       // a map of one unit
            a.out_bmu2[i] = none ? -1 : (int32_t)(uint32_t)k2;
            a.out_dist2[i] = none ? CUDART_INF_F : nx + ordered_to_float((uint32_t)(k2 >> 32));
        }
    }
}

// How a search is cut: H = 2 (slabs of 256 neurons) once that still gives every SM sixteen warps,
// else slabs of 128; pieces of one slab until there are four hundred warps per SM, longer ones
// beyond (a warp's own set-up and merge are paid once per piece).  1000 documents on 65,536 units:
// 1609 us with slabs of 128 and 64 warps per SM, 1087 so.  Never more than FEW_SLOTS keys beside one per
// document (millions of units, or tens of thousands of nearly empty documents).
static const int64_t FEW_SLOTS = 1 << 20;

static void few_cut(int64_t M, int64_t N, bool vec, int sms, int &h, int64_t &piece)
{
    h = vec && (M + 255) / 256 * N >= (int64_t)sms * 16 ? 2 : 1;
    const int64_t slab = 128 * h, slabs = (M + slab - 1) / slab;
    int64_t per = slabs * N / ((int64_t)sms * 400);
    if (per < 1) per = 1;
    if (per > 16) per = 16;
    if ((slabs + per - 1) / per > 65535) per = (slabs + 65534) / 65535;
    if ((slabs + per - 1) / per * N > FEW_SLOTS + N) per = (slabs * N + FEW_SLOTS - 1) / FEW_SLOTS;
    piece = per * slab;
}

// Room for any of its cuts: a bound that grows with the documents, unlike the cuts, so that a workspace
// for many serves fewer.
size_t few_slots_bytes(int64_t M, int64_t N, bool top2)
{
    const int64_t all = (M + 127) / 128 * N, most = FEW_SLOTS + N;
    return (size_t)(all < most ? all : most) * sizeof(u64) * (top2 ? 2 : 1);
}

template <bool VEC, int H>
static void launch_few(const FewArgs &a, bool top2, const dim3 &grid, cudaStream_t s)
{
    if (top2) { sweep_few_kernel<VEC, H, true><<<grid, FEW_WARPS * 32, 0, s>>>(a); BMU_LAUNCHED(); }
    else { sweep_few_kernel<VEC, H, false><<<grid, FEW_WARPS * 32, 0, s>>>(a); BMU_LAUNCHED(); }
}

int launch_sweep_few(FewArgs a, bool top2, int sms, cudaStream_t s)
{
    const bool vec = a.M % 4 == 0 && (reinterpret_cast<uintptr_t>(a.W) & 15) == 0;
    int h;
    few_cut(a.M, a.N, vec, sms, h, a.piece);
    const dim3 grid((unsigned)((a.N + FEW_WARPS - 1) / FEW_WARPS), (unsigned)((a.M + a.piece - 1) / a.piece));
    if (!vec) launch_few<false, 1>(a, top2, grid, s);
    else if (h == 1) launch_few<true, 1>(a, top2, grid, s);
    else launch_few<true, 2>(a, top2, grid, s);
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

}  // namespace bmu
