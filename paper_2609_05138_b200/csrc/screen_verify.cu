// The verify stage of the screened search (screen.cuh).
//
// collect  after every screening launch: four lanes per document look at the document's stripes (the
//          groups one lane of the sweep carried) in every split of the launch; stripes
//          whose smallest approximate distance lies within the document's window of the smallest seen
//          so far join the document's list.  A full list drops what the shrunken minimum has ruled
//          out; what still does not fit is evaluated at once, up to screen_early_groups.
// verify   after the last launch: the groups still within the window are evaluated exactly -- a 32-byte
//          sector per row (16 bytes of fp16), sixteen (32) rows per instruction and four instructions
//          in flight, as many fp32 sums per unit added in a fixed order -- and the outputs written.
//          Exact keys are merged by their minimum, so the order never changes a result.  Documents
//          with more groups than screen_dense_groups, with none, or with an infinite window are handed on.
//
// Waiting for the last launch matters on trained maps: far from a document's own region the
// distances lie close together, and evaluating every launch's local minimum took 11.4 ms of a
// 25.7 ms search (128 x 128 map, 200,000 documents) where the final window holds 1.8 groups of 32.
// Bound by scattered DRAM sectors (28 million for 50,000 documents with the second-best unit on a
// trained 128 x 128 map, 1.3 TB/s; half of the sectors hit L2): groups of 32 (128 bytes a row) took 788
// us for them and 272 for 120,000 documents on 64 x 64, groups of 8 with eight lanes per row 670 and
// 127, with two lanes per row, a third of the instructions, forty warps per SM and the ids read once per
// document 645 and 94.  More
// loads in flight per warp (eight) with fewer warps: 680 and 110.
#include "screen.cuh"

#include <cuda_fp16.h>
#include <math_constants.h>
#include <type_traits>

namespace bmu {

// sixteen bytes of a row: four fp32 or eight fp16 weights
__device__ __forceinline__ void verify_add16(float s[4], const float4 v)
{
    s[0] += v.x; s[1] += v.y; s[2] += v.z; s[3] += v.w;
}
__device__ __forceinline__ void verify_add16(float s[8], const uint4 v)
{
    const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 t = __half22float2(*reinterpret_cast<const __half2 *>(&x[i]));
        s[2 * i] += t.x; s[2 * i + 1] += t.y;
    }
}
__device__ __forceinline__ float verify_ld(const float *p) { return __ldg(p); }
__device__ __forceinline__ float verify_ld(const __half *p) { return __half2float(__ldg(p)); }

// One group, rows that are whole 16-byte pieces: two lanes per fp32 row (one per fp16 row), so that an
// instruction brings sixteen (32) rows' sectors.  `ids` are the first 128 of the document, a lane each
// four.  The sums of the row lanes are added by a reduction that scatters: afterwards the lanes without
// a bit of REST hold a neuron each, returned as j.
template <typename WT>
struct VerifyVec {
    static constexpr int V = 16 / (int)sizeof(WT), LPR = SC_GROUP / V, RS = 32 / LPR;
    static constexpr int REST = V == 4 ? 6 : 3;              // lane bits left over
    static_assert(RS == ScreenSums<WT, true>::N, "a partial sum per row lane");
    using Vec = typename std::conditional<V == 4, float4, uint4>::type;

    static __device__ __forceinline__ void ids_of(const VerifyArgs &a, int e, int end, uint32_t ids[4])
    {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            ids[i] = e + 32 * i + lane < end ? BMU_IDX((uint32_t)__ldg(a.colidx + e + 32 * i + lane), a.D, a.status) : 0u;
    }
    static __device__ __forceinline__ float sum(const VerifyArgs &a, int64_t j0, int beg, int end, uint32_t ids[4], int64_t &j)
    {
        const int lane = threadIdx.x & 31, row = lane / LPR;
        const int64_t at = j0 + (lane % LPR) * V;
        const char *col = static_cast<const char *>(a.W) + (at < a.M ? at : 0) * sizeof(WT);
        const uint32_t stride = (uint32_t)a.M * (uint32_t)sizeof(WT);
        float s[V];
#pragma unroll
        for (int i = 0; i < V; ++i) s[i] = 0.f;
        for (int e = beg; e < end; e += 128) {
            if (e > beg) ids_of(a, e, end, ids);
            const int n = end - e < 128 ? end - e : 128;
            constexpr int U = 4;                             // rows in flight per lane
#pragma unroll
            for (int t = 0; t < 128 / (RS * U); ++t) {
                if (t * RS * U >= n) break;
                Vec w[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int c = (t * U + u) * RS;          // first of the rows of this instruction
                    const uint32_t f = RS == 32 ? ids[c / 32] : __shfl_sync(0xffffffffu, ids[c / 32], c % 32 + row);
                    w[u] = Vec();
                    if (c + row < n) w[u] = __ldg(reinterpret_cast<const Vec *>(col + (size_t)f * stride));
                }
#pragma unroll
                for (int u = 0; u < U; ++u) verify_add16(s, w[u]);
            }
        }
        if (end - beg > 128) ids_of(a, beg, end, ids);
        int m = 16;
#pragma unroll
        for (int k = V / 2; k >= 1; k >>= 1, m >>= 1) {
            const bool up = (lane & m) != 0;
#pragma unroll
            for (int i = 0; i < k; ++i) {
                const float give = up ? s[i] : s[i + k], keep = up ? s[i + k] : s[i];
                s[i] = keep + __shfl_xor_sync(0xffffffffu, give, m);
            }
        }
#pragma unroll
        for (; m >= LPR; m >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], m);
        j = at + (V == 4 ? 2 * (lane >> 4) + ((lane >> 3) & 1)
                         : 4 * (lane >> 4) + 2 * ((lane >> 3) & 1) + ((lane >> 2) & 1));
        return s[0];
    }
};

// The whole warp evaluates the groups of `mask` (bit 4 s + c: neurons 8c .. 8c + 7 of the stripe in
// slab s) of one stripe for the document whose ids are colidx[beg .. end): the stripe's neurons in slab
// s start at ((base / 4) + launches * s) * 128 + 32 (base % 4).  A lane adds the keys it has to its best
// (and second-best) one.  Rows that are not whole 16-byte pieces: eight lanes per row.
template <typename WT, bool TOP2, bool VEC>
__device__ __forceinline__ void verify_groups(const VerifyArgs &a, const uint4 mask, uint32_t base, int beg,
                                              int end, uint32_t ids[4], u64 &best, u64 &best2)
{
    const int lane = threadIdx.x & 31, r = lane >> 3;
    const WT *W = static_cast<const WT *>(a.W);
    for (int word = 0; word < 4; ++word) {
        uint32_t bits = word == 0 ? mask.x : word == 1 ? mask.y : word == 2 ? mask.z : mask.w;
        while (bits) {
            const int bit = __ffs(bits) - 1;
            bits &= bits - 1;
            const int64_t j0 = ((int64_t)(base >> 2) + a.launches * (8 * word + (bit >> 2))) * SC_SLAB +
                               (base & 3u) * 32 + (bit & 3) * SC_GROUP;
            int64_t j;
            float sum;
            bool mine;
            if (VEC) {
                sum = VerifyVec<WT>::sum(a, j0, beg, end, ids, j);
                mine = (lane & VerifyVec<WT>::REST) == 0;
            } else {
                j = j0 + (lane & 7);
                mine = r == 0;
                const WT *col = W + (j < a.M ? j : a.M - 1);
                sum = 0.f;
                for (int e = beg; e < end; e += 64) {
                    const int mine0 = e + lane < end ? __ldg(a.colidx + e + lane) : 0;
                    const int mine1 = e + 32 + lane < end ? __ldg(a.colidx + e + 32 + lane) : 0;
                    float w[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u) {
                        const uint32_t f = (uint32_t)__shfl_sync(0xffffffffu, u < 8 ? mine0 : mine1, 4 * (u & 7) + r);
                        w[u] = 0.f;
                        if (e + 4 * u + r < end) w[u] = verify_ld(col + (int64_t)BMU_IDX(f, a.D, a.status) * a.M);
                    }
#pragma unroll
                    for (int u = 0; u < 16; ++u) sum += w[u];
                }
                sum += __shfl_xor_sync(0xffffffffu, sum, 8);
                sum += __shfl_xor_sync(0xffffffffu, sum, 16);
            }
            const u64 k = mine && j < a.M ? make_key(fmaf(-2.f, sum, __ldg(a.norms + j)), (int32_t)j) : KEY_WORST;
            if (TOP2) Best<true>::merge(best, best2, k, KEY_WORST);
            else best = k < best ? k : best;
        }
    }
}

// the warp's best (and second-best) key, on every lane
template <bool TOP2>
__device__ __forceinline__ void verify_merge(u64 &best, u64 &best2)
{
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
        const u64 o1 = __shfl_xor_sync(0xffffffffu, best, m);
        if (TOP2) {
            const u64 o2 = __shfl_xor_sync(0xffffffffu, best2, m);
            Best<true>::merge(best, best2, o1, o2);
        } else {
            best = o1 < best ? o1 : best;
        }
    }
}

__device__ __forceinline__ uint32_t popc4(const uint4 v) { return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w); }
__device__ __forceinline__ uint4 shfl4(const uint4 v, int src)
{
    return make_uint4(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src),
                      __shfl_sync(0xffffffffu, v.z, src), __shfl_sync(0xffffffffu, v.w, src));
}

// Eight documents per warp, a lane per stripe.
template <typename WT, bool TOP2, bool VEC>
__global__ void __launch_bounds__(256, 4)
screen_collect_kernel(const VerifyArgs a)
{
    const int lane = threadIdx.x & 31, k = lane & 3;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // (one lane reads the status word for its warp: the lanes must stay together)
    if (__shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(a.status), 0) || screen_whole(a.scalars) ||
        screen_natural(a.scalars) == 0u) return;
    // (in the order of the norms the sweep keeps the lists and the bounds itself; eight documents are of one set)
    const int64_t p = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 8 + (lane >> 2);
    if (screen_by_norm(a.scalars, a.set_reach, p)) return;
    const uint32_t seg = 15u << (lane & ~3), most = screen_early_groups(a.M);
    const int splits = screen_parts(a.scalars, a.splits, a.most_splits);
    const bool there = p < a.N;
    const float win = there ? a.window[p] : 0.f;
    // pass 1: the document's smallest (and second smallest) approximate value so far.  The stripes of
    // a split bring the same second smallest, over all their groups and the earlier launches;
    // whatever a merge of such pairs leaves out only makes it larger, which keeps more.
    float v1 = CUDART_INF_F, v2 = CUDART_INF_F;
    if (there && !a.first) {
        v1 = a.amin[p];
        if (TOP2) v2 = a.amin2[p];
    }
    for (int c = 0; c < splits; ++c) {
        const size_t at = ((size_t)c * a.n_pad + p) * 4 + k;
        float o1 = there ? a.cval[at].x : CUDART_INF_F, o2 = CUDART_INF_F;
        if (TOP2 && there) o2 = a.cval2[at];
#pragma unroll
        for (int m = 2; m > 0; m >>= 1) {
            const float x1 = __shfl_xor_sync(0xffffffffu, o1, m);
            if (TOP2) o2 = fminf(fminf(o2, __shfl_xor_sync(0xffffffffu, o2, m)), fmaxf(o1, x1));
            o1 = fminf(o1, x1);
        }
        if (TOP2) v2 = fminf(fminf(v2, o2), fmaxf(v1, o1));
        v1 = fminf(v1, o1);
    }
    const float limit = (TOP2 ? v2 : v1) + win;
    uint32_t count = there && !a.first ? a.lcount[p] : 0u, n = count & 15u, done = count >> 4 & 0x3ffffffu;
    bool touched = a.first, dense = (count & SC_DENSE) != 0u || win == CUDART_INF_F;
    uint4 *lm = reinterpret_cast<uint4 *>(a.lists + (size_t)p * SC_LIST_BYTES);
    float *lv = reinterpret_cast<float *>(lm + SC_LIST);
    uint32_t *lb = reinterpret_cast<uint32_t *>(lv + SC_LIST);
    // pass 2: what is within the window joins the list
    for (int c = 0; c < splits; ++c) {
        const size_t at = ((size_t)c * a.n_pad + p) * 4 + k;
        const float2 cv = there ? a.cval[at] : make_float2(CUDART_INF_F, 0.f);
        const float own = cv.x;
        uint4 mask = make_uint4(0u, 0u, 0u, 0u);
        if (there && !dense && own <= limit) {
            // words the block has written, slabs its minimum counts from
            const int from = __float_as_int(cv.y) & 255, to = __float_as_int(cv.y) >> 8;
            const uint32_t *words = reinterpret_cast<const uint32_t *>(a.cmask + at);
            uint32_t w[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                w[x] = 8 * x + 8 > from && 8 * x < to ? words[x] : 0u;
                if (from > 8 * x && from < 8 * x + 8) w[x] &= 0xffffffffu << (4 * (from - 8 * x));
            }
            mask = make_uint4(w[0], w[1], w[2], w[3]);
        }
        const bool join = (mask.x | mask.y | mask.z | mask.w) != 0u;
        const uint32_t joining = __ballot_sync(0xffffffffu, join) & seg;
        const int n_new = __popc(joining);
        touched |= joining != 0u;
        // a list that would overflow: drop what is out of the window by now
        const bool full = joining && n + n_new > (uint32_t)SC_LIST;
        if (__any_sync(0xffffffffu, full)) {
            // (the entries change lanes through global memory: what other lanes appended before, what they read below)
            __syncwarp();
            uint32_t kept = 0;
            for (int r = 0; r < (SC_LIST + 3) / 4; ++r) {
                const uint32_t e = r * 4 + k;
                const bool mine = full && e < n;
                const float v = mine ? lv[e] : 0.f;
                const uint4 mk = mine ? lm[e] : make_uint4(0u, 0u, 0u, 0u);
                const uint32_t bs = mine ? lb[e] : 0u;
                const bool keep = mine && v <= limit;
                const uint32_t who = __ballot_sync(0xffffffffu, keep) & seg;
                __syncwarp();                                // read by all before any of them is overwritten
                if (keep) {                                  // entries move towards the front only
                    const uint32_t to = kept + __popc(who & ((1u << lane) - 1u));
                    lv[to] = v; lm[to] = mk; lb[to] = bs;
                }
                kept += __popc(who);
                __syncwarp();
            }
            if (full) n = kept;
        }
        const uint32_t to = n + __popc(joining & ((1u << lane) - 1u));
        const uint32_t base = (uint32_t)(a.launch * 4 + k);
        if (join && to < (uint32_t)SC_LIST) { lv[to] = own; lm[to] = mask; lb[to] = base; }
        n = min(n + (uint32_t)n_new, (uint32_t)SC_LIST);
        const uint32_t left_over = __ballot_sync(0xffffffffu, join && to >= (uint32_t)SC_LIST);
        if (left_over) {                                     // no room: evaluated here and now
            int32_t orig = 0, beg = 0, end = 0;
            if (there) {
                orig = a.perm[p];
                beg = __ldg(a.rowptr + orig);
                end = __ldg(a.rowptr + orig + 1);
            }
            u64 best = KEY_WORST, best2 = KEY_WORST;
            for (uint32_t lanes = left_over; lanes; lanes &= lanes - 1) {
                const int src = __ffs(lanes) - 1;
                const uint4 groups = shfl4(mask, src);
                const uint32_t more = popc4(groups) + __shfl_sync(0xffffffffu, done, src);
                if (__shfl_sync(0xffffffffu, dense, src)) continue;
                if (lane >> 2 == src >> 2) { dense = more > most; done = more; }
                if (more > most) continue;
                u64 k1 = KEY_WORST, k2 = KEY_WORST;
                const int b0 = __shfl_sync(0xffffffffu, beg, src), e0 = __shfl_sync(0xffffffffu, end, src);
                uint32_t ids[4];
                if (VEC) VerifyVec<WT>::ids_of(a, b0, e0, ids);
                verify_groups<WT, TOP2, VEC>(a, groups, __shfl_sync(0xffffffffu, base, src), b0, e0, ids, k1, k2);
                verify_merge<TOP2>(k1, k2);
                if (lane >> 2 == src >> 2) {
                    if (TOP2) Best<true>::merge(best, best2, k1, k2);
                    else best = k1 < best ? k1 : best;
                }
            }
            if (there && (left_over & seg)) {
                if (k == 0) {
                    if (count & 0x80000000u) {
                        if (TOP2) Best<true>::merge(best, best2, a.state[orig], a.state2[orig]);
                        else { const u64 old = a.state[orig]; best = old < best ? old : best; }
                    }
                    a.state[orig] = best;
                    if (TOP2) a.state2[orig] = best2;
                }
                count |= 0x80000000u;
                touched = true;
            }
            __syncwarp();
        }
    }
    if (there && k == 0) {
        a.amin[p] = v1;
        if (TOP2) a.amin2[p] = v2;
        if (touched) a.lcount[p] = (count & 0x80000000u) | (dense ? SC_DENSE : done << 4 | n);
    }
}

// Two documents per warp, sixteen lanes each: a lane takes one list entry.
template <typename WT, bool TOP2, bool VEC>
__global__ void __launch_bounds__(256, 5)
screen_verify_kernel(const VerifyArgs a)
{
    static_assert(SC_LIST <= 15, "a lane per entry, four bits of the count");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");      // screen_dense_kernel waits for the rest
    asm volatile("griddepcontrol.wait;" ::: "memory");                   // as this does for the last collection
    const int lane = threadIdx.x & 31, e = lane & 15;
    const int64_t p = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 2 + (lane >> 4);
    if (__shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(a.status), 0)) return;
    const bool there = p < a.N, whole = screen_whole(a.scalars);
    if (!whole && screen_by_norm(a.scalars, a.set_reach, p)) return;     // (sixteen documents are of one set)
    uint32_t count = 0, base = 0;
    uint4 todo = make_uint4(0u, 0u, 0u, 0u);
    int32_t orig = 0, beg = 0, end = 0;
    if (there) {
        count = whole ? SC_DENSE : a.lcount[p];
        orig = a.perm[p];
        beg = __ldg(a.rowptr + orig);
        end = __ldg(a.rowptr + orig + 1);
        if ((uint32_t)e < (count & 15u)) {
            const float limit = (TOP2 ? a.amin2[p] : a.amin[p]) + a.window[p];
            const uint4 *lm = reinterpret_cast<const uint4 *>(a.lists + (size_t)p * SC_LIST_BYTES);
            const float *lv = reinterpret_cast<const float *>(lm + SC_LIST);
            if (lv[e] <= limit) todo = lm[e];
            base = reinterpret_cast<const uint32_t *>(lv + SC_LIST)[e];
        }
    }
    // too many groups, or none (no distance of it is finite), or given up before
    uint32_t groups = popc4(todo);
#pragma unroll
    for (int m = 8; m > 0; m >>= 1) groups += __shfl_xor_sync(0xffffffffu, groups, m);
    const bool dense = (count & SC_DENSE) || groups > screen_dense_groups(a.M) || (groups == 0u && !(count & 0x80000000u));
    if (dense) todo = make_uint4(0u, 0u, 0u, 0u);
    u64 best = KEY_WORST, best2 = KEY_WORST;
    const uint32_t entries = __ballot_sync(0xffffffffu, (todo.x | todo.y | todo.z | todo.w) != 0u);
#pragma unroll 1
    for (int d = 0; d < 2; ++d) {                            // its ids once per document
        uint32_t lanes = entries & (0xffffu << (16 * d));
        if (!lanes) continue;
        const int b0 = __shfl_sync(0xffffffffu, beg, 16 * d), e0 = __shfl_sync(0xffffffffu, end, 16 * d);
        uint32_t ids[4];
        if (VEC) VerifyVec<WT>::ids_of(a, b0, e0, ids);
        u64 k1 = KEY_WORST, k2 = KEY_WORST;
        for (; lanes; lanes &= lanes - 1) {
            const int src = __ffs(lanes) - 1;
            verify_groups<WT, TOP2, VEC>(a, shfl4(todo, src), __shfl_sync(0xffffffffu, base, src), b0, e0, ids, k1, k2);
        }
        verify_merge<TOP2>(k1, k2);
        if (lane >> 4 == d) { best = k1; best2 = k2; }
    }
    if (there && dense) {
        if (e == 0) {
            a.state[orig] = KEY_WORST;
            if (TOP2) a.state2[orig] = KEY_WORST;
            a.lcount[p] = 0u;                                // its ticket from here on
            if (!whole) a.dense[atomicAdd(a.dense_count, 1u)] = (uint32_t)p;
        }
        return;
    }
    if (there && (count & 0x80000000u)) {
        if (TOP2) Best<true>::merge(best, best2, a.state[orig], a.state2[orig]);
        else { const u64 old = a.state[orig]; best = old < best ? old : best; }
    }
    if (there && e == 0) {
        const float nx = (float)(end - beg);
        a.out_bmu[orig] = (int32_t)(uint32_t)best;
        a.out_dist[orig] = nx + ordered_to_float((uint32_t)(best >> 32));
        if (TOP2) {
            const bool none = best2 == KEY_WORST;            // a map of one unit
            a.out_bmu2[orig] = none ? -1 : (int32_t)(uint32_t)best2;
            a.out_dist2[orig] = none ? CUDART_INF_F : nx + ordered_to_float((uint32_t)(best2 >> 32));
        }
    }
}

// The documents whose slabs were in the order of the norms, one per warp, a lane per list entry.  The units of an
// entry are evaluated several at a time: as many lanes for each as rows are summed side by side above, and their
// sums added in the same order, so that a unit has the same distance, bit for bit, whichever way it came here.  A
// 32-byte sector per row.
template <typename WT, bool TOP2, bool VEC>
__global__ void __launch_bounds__(256, 5)
screen_verify_units_kernel(const VerifyArgs a)
{
    constexpr int L = ScreenSums<WT, VEC>::N, AT_ONCE = 32 / L, U = VEC ? 4 : 16;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31, row = lane % L;
    if (__shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(a.status), 0) || screen_whole(a.scalars) ||
        !screen_ordered(a.scalars)) return;
    const WT *W = static_cast<const WT *>(a.W);
    for (int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < a.N; p += (int64_t)gridDim.x * (blockDim.x / 32)) {
        if (!screen_by_norm(a.scalars, a.set_reach, p)) continue;
        const float win = a.window[p];
        const uint32_t n = a.lcount[p];
        const int32_t orig = a.perm[p];
        const int beg = __ldg(a.rowptr + orig), end = __ldg(a.rowptr + orig + 1);
        uint4 t = make_uint4(0u, 0u, 0u, 0u);
        if (lane < SC_OWN_LIST && (uint32_t)lane < n) t = reinterpret_cast<const uint4 *>(a.lists + p * SC_LIST_BYTES)[lane];
        if (!(__uint_as_float(t.x) <= ordered_to_float(a.bound[p]) + win)) t.z = 0u;
        // too many units, or none (no distance of it is finite), or a list that was too short for them
        const uint32_t units = __reduce_add_sync(0xffffffffu, __popc(t.z));
        if (n > (uint32_t)SC_OWN_LIST || units == 0u || a.reach[p].x > a.scalars[SC_DOC_TOP] || units > screen_dense_groups(a.M) || win == CUDART_INF_F) {
            if (lane == 0) {
                a.state[orig] = KEY_WORST;
                if (TOP2) a.state2[orig] = KEY_WORST;
                a.lcount[p] = 0u;                            // its ticket from here on
                a.dense[atomicAdd(a.dense_count, 1u)] = (uint32_t)p;
            }
            continue;
        }
        u64 best = KEY_WORST, best2 = KEY_WORST;
        for (uint32_t entries = __ballot_sync(0xffffffffu, t.z != 0u); entries; entries &= entries - 1) {
            const int src = __ffs(entries) - 1;
            const int64_t first = (int64_t)__shfl_sync(0xffffffffu, t.y, src) * SC_SLAB + __shfl_sync(0xffffffffu, t.w, src) * 32;
            uint32_t bits = __shfl_sync(0xffffffffu, t.z, src);
            while (bits) {
                int32_t j = -1;
#pragma unroll
                for (int i = 0; i < AT_ONCE; ++i) {
                    if (!bits) break;
                    if (i == lane / L) j = a.units[first + __ffs(bits) - 1];     // (-1 beyond the last unit)
                    bits &= bits - 1;
                }
                float s = 0.f;
                for (int e0 = beg; e0 < end; e0 += L * U) {
                    float w[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int e = e0 + u * L + row;
                        w[u] = j >= 0 && e < end ? verify_ld(W + (int64_t)BMU_IDX((uint32_t)__ldg(a.colidx + e), a.D, a.status) * a.M + j) : 0.f;
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) s += w[u];
                }
#pragma unroll
                for (int m = L / 2; m >= 1; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, VEC ? m : L / 2 / m);
                const u64 k = row == 0 && j >= 0 ? make_key(fmaf(-2.f, s, __ldg(a.norms + j)), j) : KEY_WORST;
                if (TOP2) Best<true>::merge(best, best2, k, KEY_WORST);
                else best = k < best ? k : best;
            }
        }
        verify_merge<TOP2>(best, best2);
        if (lane == 0) {
            const float nx = (float)(end - beg);
            a.out_bmu[orig] = (int32_t)(uint32_t)best;
            a.out_dist[orig] = nx + ordered_to_float((uint32_t)(best >> 32));
            if (TOP2) {
                const bool none = best2 == KEY_WORST;
                a.out_bmu2[orig] = none ? -1 : (int32_t)(uint32_t)best2;
                a.out_dist2[orig] = none ? CUDART_INF_F : nx + ordered_to_float((uint32_t)(best2 >> 32));
            }
        }
    }
}

#define BMU_VERIFY(KERNEL, C) \
    (a.f16 ? (top2 ? (screen_vec(a) ? cudaLaunchKernelEx(&C, KERNEL<__half, true, true>, a) : cudaLaunchKernelEx(&C, KERNEL<__half, true, false>, a)) \
                   : (screen_vec(a) ? cudaLaunchKernelEx(&C, KERNEL<__half, false, true>, a) : cudaLaunchKernelEx(&C, KERNEL<__half, false, false>, a))) \
           : (top2 ? (screen_vec(a) ? cudaLaunchKernelEx(&C, KERNEL<float, true, true>, a) : cudaLaunchKernelEx(&C, KERNEL<float, true, false>, a)) \
                   : (screen_vec(a) ? cudaLaunchKernelEx(&C, KERNEL<float, false, true>, a) : cudaLaunchKernelEx(&C, KERNEL<float, false, false>, a))))

int launch_screen_collect(const VerifyArgs &a, bool top2, cudaStream_t s)
{
    ScreenLaunch l((unsigned)((a.N + 63) / 64), 256, s, true);
    BMU_CUDA(BMU_VERIFY(screen_collect_kernel, l.c));
    BMU_LAUNCHED();
    return BMU_OK;
}

int launch_screen_verify(const VerifyArgs &a, bool top2, cudaStream_t s)
{
    ScreenLaunch l((unsigned)((a.N + 15) / 16), 256, s, true);
    BMU_CUDA(BMU_VERIFY(screen_verify_kernel, l.c));
    BMU_LAUNCHED();
    return BMU_OK;
}

int launch_screen_verify_units(const VerifyArgs &a, bool top2, int sms, cudaStream_t s)
{
    const int64_t blocks = (a.N + 7) / 8;
    ScreenLaunch l((unsigned)(blocks < 5 * sms ? blocks : 5 * sms), 256, s, true);
    BMU_CUDA(BMU_VERIFY(screen_verify_units_kernel, l.c));
    BMU_LAUNCHED();
    return BMU_OK;
}

}  // namespace bmu
