// Documents the screen cannot help with (screen.cuh): evaluated against all units, exactly, by the whole
// chip.  The verify stage hands over those with more candidate groups than screen_dense_groups -- exact
// or near ties all over the map, as after an epoch with a wide neighbourhood, weights the 8-bit image does
// not resolve, lists too long for its sums -- and those without any candidate (distances that are not
// finite).  Where most of a sample of the documents would come here, all do, and nothing is screened.
//
// A unit's weights are added in the order of the verify stage (ScreenSums: sixteen fp32 partial sums, each over
// every sixteenth id, added in pairs), so that a unit has the same distance, bit for bit, whichever way it came
// here: which documents come depends on the others in the call, and on when a bound was lowered.
//
// A warp takes a document and a piece of 512 units, 64 of them at a time (128 where rows are not whole 16-byte
// pieces).  Two halves of the warp take every other id (fp16: four quarters every fourth), a lane carries the
// partial sums of its ids for the four (eight) units of a 16-byte load; the next row of a partial sum is asked for
// as soon as the one before has been added, also across the 64s, ids through shared memory.  Pieces outside, documents
// inside, so that all warps in flight share one piece or two: rows of W in L2, those of frequent features in L1.
// Keys meet in the per-document state; the warp that arrives last at a document (a ticket each) writes its outputs.
//
// Bound by the latency of its loads: 64 KB in flight per SM, which the sums' registers bound.  All of 50,000
// documents of 80 ids on 4,096 units take 3.3 ms, 20,000 on 16,384 units 5.4, 50,000 on 4,096 units of fp16 3.4,
// 20,000 on 4,099 units 1.9.  (One sum per unit over all ids, eight units to a lane, twice the warps: 3.0, 5.8, 2.8
// and 2.2, with distances of its own.)  The sixteen sums one after the other, those that wait for their pair in
// registers or shared memory: 3.8, 6.4, 4.6, 2.6.  Pieces of 64, 128, 256 and 1,024 units: 4.8, 4.0, 3.6 and 3.8 for
// the first; twelve warps in two blocks 4.5.
#include "screen.cuh"

#include <cuda_fp16.h>
#include <math_constants.h>

#include <type_traits>

namespace bmu {

// adds a lane's weights of a row: sixteen bytes of it, or four fp32 values
template <typename WT, bool VEC>
__device__ __forceinline__ void dense_add(u64 *acc, const u64 w[2])
{
    if constexpr (sizeof(WT) == 4 || !VEC) {
        add2(acc[0], w[0]);
        add2(acc[1], w[1]);
    } else {
        const uint32_t x[4] = {(uint32_t)w[0], (uint32_t)(w[0] >> 32), (uint32_t)w[1], (uint32_t)(w[1] >> 32)};
#pragma unroll
        for (int i = 0; i < 4; ++i) {                        // (a fp16 value is an fp32 one: one rounding)
            float lo = lo_f(acc[i]), hi = hi_f(acc[i]);
            asm("add.rn.f32.f16 %0, %1, %0;" : "+f"(lo) : "h"((uint16_t)x[i]));
            asm("add.rn.f32.f16 %0, %1, %0;" : "+f"(hi) : "h"((uint16_t)(x[i] >> 16)));
            acc[i] = (u64)__float_as_uint(hi) << 32 | __float_as_uint(lo);
        }
    }
}
__device__ __forceinline__ float dense_ld(const float *p) { return __ldg(p); }
__device__ __forceinline__ float dense_ld(const __half *p) { return __half2float(__ldg(p)); }

// A list's partial sums are shared out to GROUPS groups of lanes, SUMS to a lane; a lane owns V units of a stretch of
// UNITS, VEC: with one load per row.
template <typename WT, bool VEC> struct Dense {
    using Sums = ScreenSums<WT, VEC>;
    static constexpr int V = VEC ? 16 / (int)sizeof(WT) : 4, GROUPS = !VEC ? 1 : V == 4 ? 2 : 4;
    static constexpr int LANES = 32 / GROUPS, UNITS = LANES * V, SUMS = Sums::N / GROUPS;
    static constexpr int WARPS = VEC ? 16 : 24;              // of the one block per SM
};
static const int DENSE_PIECE = 512, DENSE_IDS = 128;

template <typename WT, bool TOP2, bool VEC>
__global__ void __launch_bounds__(Dense<WT, VEC>::WARPS * 32, 1)
screen_dense_kernel(const VerifyArgs a)
{
    using X = Dense<WT, VEC>;
    constexpr int P = X::Sums::N, C = X::SUMS, V = X::V, H = V / 2, GROUPS = X::GROUPS;
    __shared__ uint4 s_ids[X::WARPS][DENSE_IDS / 4];         // the ids of a group of lanes one after the other
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = lane / X::LANES;
    uint32_t *mine = reinterpret_cast<uint32_t *>(s_ids[warp]);
    const uint4 *ids = s_ids[warp] + group * (DENSE_IDS / GROUPS / 4);
    const uint32_t stride = (uint32_t)a.M * (uint32_t)sizeof(WT);        // (M < 2^30)
    asm volatile("griddepcontrol.wait;" ::: "memory");       // for the verify stage, under whose end it is launched
    if (__shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(a.status), 0)) return;
    const bool whole = screen_whole(a.scalars);              // all documents, in the planned order
    const int64_t docs = whole ? a.N : (int64_t)*a.dense_count, warps = (int64_t)gridDim.x * X::WARPS;
    if (docs == 0) return;
    const int64_t pieces = (a.M + DENSE_PIECE - 1) / DENSE_PIECE;
    int64_t at = (int64_t)blockIdx.x * X::WARPS + warp, j0 = 0;      // the item: a document and the first unit of a piece
    auto in_turn = [&]() { for (; at >= docs; at -= docs) j0 += DENSE_PIECE; return j0 < a.M; };
    bool more = in_turn();
    int64_t p_next = 0;
    int32_t orig_next = 0;
    auto ask = [&]() { if (more) { p_next = whole ? at : (int64_t)a.dense[at]; orig_next = a.perm[p_next]; } };
    ask();
    while (more) {
        const int64_t p = p_next, jp = j0;
        const int32_t orig = orig_next;
        const int beg = __ldg(a.rowptr + orig), n = __ldg(a.rowptr + orig + 1) - beg;
        at += warps;
        more = in_turn();
        ask();
        Best<TOP2> best;
        best.init();
        // where the lane's loads start; beyond the last unit they repeat it (and count for nothing)
        auto column = [&](int64_t j) { return static_cast<const WT *>(a.W) + (VEC ? min(j, a.M - V) : (int64_t)0); };
        int64_t j = jp + (VEC ? lane % X::LANES * V : lane);
        const WT *col = column(j);
        u64 w[C][VEC ? 2 : H];
        bool ahead = false;                                  // the first rows of this stretch are on their way
        for (int x = 0; x < DENSE_PIECE && jp + x < a.M; x += X::UNITS, j += X::UNITS) {
            const bool last = x + X::UNITS >= DENSE_PIECE || jp + x + X::UNITS >= a.M;
            const WT *next = column(j + X::UNITS);
            u64 acc[C][H];
#pragma unroll
            for (int c = 0; c < C; ++c)
#pragma unroll
                for (int v = 0; v < H; ++v) acc[c][v] = 0ull;
            // the weights of P ids from place q on, one for every partial sum: all of them, or those below `most`;
            // each is asked for as soon as the one before it has been added
            auto rows = [&](const WT *from, int64_t at, int q, int most, auto full, auto add) {
                uint4 f4[C / 4];
#pragma unroll
                for (int c = 0; c < C / 4; ++c) f4[c] = ids[q / GROUPS / 4 + c];
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    if (decltype(add)::value) dense_add<WT, VEC>(acc[c], w[c]);
                    const uint4 t = f4[c / 4];
                    const uint32_t f = c % 4 == 0 ? t.x : c % 4 == 1 ? t.y : c % 4 == 2 ? t.z : t.w;
                    const bool there = decltype(full)::value || q + c * GROUPS + group < most;
                    const WT *row = reinterpret_cast<const WT *>(reinterpret_cast<const char *>(from) + (u64)f * stride);
                    if constexpr (VEC) {
                        ulonglong2 t2 = make_ulonglong2(0ull, 0ull);
                        if (there) t2 = __ldg(reinterpret_cast<const ulonglong2 *>(row));
                        w[c][0] = t2.x; w[c][1] = t2.y;
                    } else {
#pragma unroll
                        for (int v = 0; v < H; ++v) {
                            const float lo = there ? dense_ld(row + min(at + 64 * v, a.M - 1)) : 0.f;
                            const float hi = there ? dense_ld(row + min(at + 64 * v + 32, a.M - 1)) : 0.f;
                            w[c][v] = (u64)__float_as_uint(hi) << 32 | __float_as_uint(lo);
                        }
                    }
                }
            };
            auto step = [&](const WT *from, int64_t at, int q, int most, auto add) {
                if (q + P <= most) rows(from, at, q, most, std::true_type(), add);
                else rows(from, at, q, most, std::false_type(), add);
            };
            for (int eb = 0; eb < n; eb += DENSE_IDS) {
                const int most = min(DENSE_IDS, n - eb);
                if (x == 0 || n > DENSE_IDS) {
                    __syncwarp();                            // the ids before these have been used
#pragma unroll
                    for (int k = 0; k < DENSE_IDS / 32; ++k) {
                        const int e = 32 * k + lane;
                        mine[e % GROUPS * (DENSE_IDS / GROUPS) + e / GROUPS] =
                            e < most ? BMU_IDX((uint32_t)__ldg(a.colidx + beg + eb + e), a.D, a.status) : 0u;
                    }
                    __syncwarp();
                }
                if (!ahead) step(col, j, 0, most, std::false_type());
                for (int q = P; q < most; q += P) step(col, j, q, most, std::true_type());
                ahead = n <= DENSE_IDS && !last;
                if (ahead) {
                    step(next, j + X::UNITS, 0, most, std::true_type());
                } else {
#pragma unroll
                    for (int c = 0; c < C; ++c) dense_add<WT, VEC>(acc[c], w[c]);
                }
            }
            col = next;
            // the lane's partial sums, in the order of the verify stage
            if constexpr (VEC) {
#pragma unroll
                for (int c = C / 2; c >= 1; c /= 2)
#pragma unroll
                    for (int i = 0; i < c; ++i)
#pragma unroll
                        for (int v = 0; v < H; ++v) add2(acc[i][v], acc[i + c][v]);
            } else {
#pragma unroll
                for (int c = 1; c < C; c *= 2)
#pragma unroll
                    for (int i = 0; i < C; i += 2 * c)
#pragma unroll
                        for (int v = 0; v < H; ++v) add2(acc[i][v], acc[i + c][v]);
            }
            float s[V];
#pragma unroll
            for (int v = 0; v < V; ++v) s[v] = v % 2 ? hi_f(acc[0][v / 2]) : lo_f(acc[0][v / 2]);
            // ... and the groups': of every pair of lanes, one keeps the first half of the units
            int64_t at_j = j;
            int k = V;
#pragma unroll
            for (int m = 16; m >= X::LANES; m /= 2) {
                k /= 2;
                const bool up = (lane & m) != 0;
#pragma unroll
                for (int i = 0; i < V / 2; ++i) {
                    if (i >= k) continue;
                    const float give = up ? s[i] : s[i + k], keep = up ? s[i + k] : s[i];
                    s[i] = keep + __shfl_xor_sync(0xffffffffu, give, m);
                }
                if (up) at_j += k;
            }
#pragma unroll
            for (int i = 0; i < V / GROUPS; ++i) {
                const int64_t ji = at_j + (VEC ? i : 32 * i);
                if (ji < a.M) best.push(fmaf(-2.f, s[i], __ldg(a.norms + ji)), (int)ji);
            }
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
                const float nx = (float)n;
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
template <typename WT, bool TOP2, bool VEC>
static int launch_dense(const VerifyArgs &a, int sms, cudaStream_t s)
{
    using X = Dense<WT, VEC>;
    ScreenLaunch l((unsigned)sms, X::WARPS * 32, s, true);
    BMU_CUDA(cudaLaunchKernelEx(&l.c, screen_dense_kernel<WT, TOP2, VEC>, a));
    BMU_LAUNCHED();
    return BMU_OK;
}

int launch_screen_dense(const VerifyArgs &a, bool top2, int sms, cudaStream_t s)
{
    const bool vec = screen_vec(a);
    if (a.f16) {
        if (vec) return top2 ? launch_dense<__half, true, true>(a, sms, s) : launch_dense<__half, false, true>(a, sms, s);
        return top2 ? launch_dense<__half, true, false>(a, sms, s) : launch_dense<__half, false, false>(a, sms, s);
    }
    if (vec) return top2 ? launch_dense<float, true, true>(a, sms, s) : launch_dense<float, false, true>(a, sms, s);
    return top2 ? launch_dense<float, true, false>(a, sms, s) : launch_dense<float, false, false>(a, sms, s);
}

}  // namespace bmu
