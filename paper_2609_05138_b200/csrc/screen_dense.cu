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
// A warp takes a document and a piece of up to 384 units (fp16: 1,024), 128 of them at a time, in two passes: the partial
// sums of the even places of the list, then those of the odd ones.  A lane carries the partial sums of four (fp16: eight,
// where half of the warp takes every other id of a pass) units, 32 (64) registers, and asks for the next row of each as
// soon as the one before has been added, also across passes and stretches; ids through shared memory.  Pieces outside,
// documents inside, so that all warps in flight share one piece or two: rows of W in L2, those of frequent features
// in L1.  Keys meet in the per-document state; the warp that arrives last at a document (a ticket each) writes its
// outputs.
//
// Bound by the latency of its loads, 64 KB in flight per SM, which the sums' registers bound, and by L1 hits.  All of
// 50,000 documents of 80 ids on 4,096 units take 3.1 ms, 20,000 on 16,384 units 5.3, 50,000 on 4,096 units of fp16 3.1,
// 20,000 on 4,099 units 1.9.  (One sum per unit over all ids, eight units to a lane, twice the warps: 3.0, 5.6, 2.8
// and 2.2, with distances of its own.)  Pieces of 256, 512 and 768 units: 3.3 / 5.4, 3.0 / 6.4, 3.3 / 6.6 for the first two.
// One pass over 64 units, half of the warp for each half of the list: 3.3, 5.4, 3.4; the sixteen sums one after the
// other, those that wait for their pair in registers or shared memory: 3.8, 6.4, 4.6, 2.6; rows asked for sixteen at a time
// and then added: 3.6, 5.9, 4.0; touching a piece's rows ahead in L2: 3.4, 5.5, 3.5, and 5 % more for 100,000 documents
// on 512 x 512.
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

// A list's partial sums are shared out to PASSES over a stretch of UNITS and, in each, GROUPS groups of lanes: SUMS to a
// lane, which owns V units of the stretch, VEC: with one load per row.
template <typename WT, bool VEC> struct Dense {
    using Sums = ScreenSums<WT, VEC>;
    static constexpr int V = VEC ? 16 / (int)sizeof(WT) : 4, PASSES = VEC ? 2 : 1, GROUPS = VEC && V == 8 ? 2 : 1;
    static constexpr int LANES = 32 / GROUPS, UNITS = LANES * V, SHARES = PASSES * GROUPS, SUMS = Sums::N / SHARES;
    static constexpr int WARPS = VEC ? 16 : 24, MOST = V == 8 ? 8 : 3;      // of the one block per SM; stretches of an item
};
static const int DENSE_IDS = 128;

template <typename WT, bool TOP2, bool VEC>
__global__ void __launch_bounds__(Dense<WT, VEC>::WARPS * 32, 1)
screen_dense_kernel(const VerifyArgs a)
{
    using X = Dense<WT, VEC>;
    constexpr int P = X::Sums::N, C = X::SUMS, V = X::V, H = V / 2, SHARES = X::SHARES, OWN = V / X::GROUPS;
    __shared__ uint4 s_ids[X::WARPS][DENSE_IDS / 4];         // the ids of a share one after the other
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = lane / X::LANES;
    uint32_t *mine = reinterpret_cast<uint32_t *>(s_ids[warp]);
    const uint32_t stride = (uint32_t)a.M * (uint32_t)sizeof(WT);        // (M < 2^30)
    asm volatile("griddepcontrol.wait;" ::: "memory");       // for the verify stage, under whose end it is launched
    if (__shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(a.status), 0)) return;
    const bool whole = screen_whole(a.scalars);              // all documents, in the planned order
    const int64_t docs = whole ? a.N : (int64_t)*a.dense_count, warps = (int64_t)gridDim.x * X::WARPS;
    if (docs == 0) return;
    // Few documents: pieces of fewer stretches, so that every warp has four or more (two, eight, sixteen: 60,000 documents
    // on fp16 256 x 256, 91 of them whole, 2,965, 2,957 and 2,984 us instead of 2,948).
    const int64_t stretches = docs * ((a.M + X::UNITS - 1) / X::UNITS) / (4 * warps);
    const int piece = X::UNITS * (int)max((int64_t)1, min((int64_t)X::MOST, stretches));
    const int64_t pieces = (a.M + piece - 1) / piece;
    // the item: a document and the first unit of a piece; and so many of either to the next one
    const int64_t first = (int64_t)blockIdx.x * X::WARPS + warp, step_at = warps % docs, step_j = warps / docs * piece;
    int64_t at = first % docs, j0 = first / docs * piece;
    bool more = j0 < a.M;
    int64_t p_next = 0;
    int32_t orig_next = 0;
    auto ask = [&]() { if (more) { p_next = whole ? at : (int64_t)a.dense[at]; orig_next = a.perm[p_next]; } };
    ask();
    while (more) {
        const int64_t p = p_next, jp = j0;
        const int32_t orig = orig_next;
        const int beg = __ldg(a.rowptr + orig), n = __ldg(a.rowptr + orig + 1) - beg;
        at += step_at;
        j0 += step_j;
        if (at >= docs) { at -= docs; j0 += piece; }
        more = j0 < a.M;
        ask();
        Best<TOP2> best;
        best.init();
        // where the lane's loads start; beyond the last unit they repeat it (and count for nothing)
        auto column = [&](int64_t j) { return static_cast<const WT *>(a.W) + (VEC ? min(j, a.M - V) : (int64_t)0); };
        int64_t j = jp + (VEC ? lane % X::LANES * V : lane);
        const WT *col = column(j);
        u64 w[C][VEC ? 2 : H];
        bool ahead = false;                                  // the first rows of a pass are on their way
        for (int x = 0; x < piece && jp + x < a.M; x += X::UNITS, j += X::UNITS) {
            const bool last = x + X::UNITS >= piece || jp + x + X::UNITS >= a.M;
            const WT *next = column(j + X::UNITS);
            float sum[OWN];
            int64_t own = j;
#pragma unroll
            for (int pass = 0; pass < X::PASSES; ++pass) {
                u64 acc[C][H];
#pragma unroll
                for (int c = 0; c < C; ++c)
#pragma unroll
                    for (int v = 0; v < H; ++v) acc[c][v] = 0ull;
                // the weights of the next C ids of each share of pass `of`, from place q on: all of them, or those below
                // `most`; each is asked for as soon as the one before it has been added
                auto rows = [&](const WT *from, int64_t at, int of, int q, int most, auto full, auto add) {
                    const uint4 *ids = s_ids[warp] + ((group * X::PASSES + of) * (DENSE_IDS / SHARES) + q) / 4;
                    uint4 f4[C / 4];
#pragma unroll
                    for (int c = 0; c < C / 4; ++c) f4[c] = ids[c];
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        if (decltype(add)::value) dense_add<WT, VEC>(acc[c], w[c]);
                        const uint4 t = f4[c / 4];
                        const uint32_t f = c % 4 == 0 ? t.x : c % 4 == 1 ? t.y : c % 4 == 2 ? t.z : t.w;
                        const bool there = decltype(full)::value || (q + c) * SHARES + group * X::PASSES + of < most;
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
                auto step = [&](const WT *from, int64_t at, int of, int q, int most, auto add) {
                    if (q * SHARES + P <= most) rows(from, at, of, q, most, std::true_type(), add);
                    else rows(from, at, of, q, most, std::false_type(), add);
                };
                for (int eb = 0; eb < n; eb += DENSE_IDS) {
                    const int most = min(DENSE_IDS, n - eb);
                    if ((x == 0 && pass == 0) || n > DENSE_IDS) {
                        __syncwarp();                        // the ids before these have been used
#pragma unroll
                        for (int k = 0; k < DENSE_IDS / 32; ++k) {
                            const int e = 32 * k + lane;
                            mine[e % SHARES * (DENSE_IDS / SHARES) + e / SHARES] =
                                e < most ? BMU_IDX((uint32_t)__ldg(a.colidx + beg + eb + e), a.D, a.status) : 0u;
                        }
                        __syncwarp();
                    }
                    if (!ahead) step(col, j, pass, 0, most, std::false_type());
                    for (int q = C; q * SHARES + pass < most; q += C) step(col, j, pass, q, most, std::true_type());
                    ahead = n <= DENSE_IDS && !(last && pass + 1 == X::PASSES);
                    if (ahead && pass + 1 < X::PASSES) {
                        step(col, j, pass + 1, 0, most, std::true_type());
                    } else if (ahead) {
                        step(next, j + X::UNITS, 0, 0, most, std::true_type());
                    } else {
#pragma unroll
                        for (int c = 0; c < C; ++c) dense_add<WT, VEC>(acc[c], w[c]);
                    }
                }
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
                // ... the groups', of every pair of lanes one keeps the first half of the units, and the passes'
                if (X::GROUPS == 2) {
                    const bool up = group != 0;
#pragma unroll
                    for (int i = 0; i < V / 2; ++i) {
                        const float give = up ? s[i] : s[i + V / 2], keep = up ? s[i + V / 2] : s[i];
                        s[i] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
                    }
                    own = j + (up ? V / 2 : 0);
                }
#pragma unroll
                for (int i = 0; i < OWN; ++i) sum[i] = pass ? sum[i] + s[i] : s[i];
            }
            col = next;
#pragma unroll
            for (int i = 0; i < OWN; ++i) {
                const int64_t ji = own + (VEC ? i : 32 * i);
                if (ji < a.M) best.push(fmaf(-2.f, sum[i], __ldg(a.norms + ji)), (int)ji);
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
