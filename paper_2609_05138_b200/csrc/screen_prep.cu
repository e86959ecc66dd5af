// Preparation of the screening sweep (screen.cuh): ranges of the codebook rows, the steps of the
// fixed-point image and its error bounds, the per-document windows, and the images themselves.
#include "screen.cuh"
#include "mma_ptx.cuh"

#include <cuda_fp16.h>
#include <math_constants.h>
#include <type_traits>

namespace bmu {

static inline size_t up256(size_t x) { return (x + 255) / 256 * 256; }

template <typename Take>
static void codebook_layout(int64_t D, int64_t M, int64_t slots, int64_t ord_slots, int sets, Take take, ScreenLayout *l)
{
    const size_t d4 = (size_t)D * 4;
    l->scalars = take((size_t)sets * SC_SCALARS * 4);
    l->rmin = take(d4); l->rmax = take(d4);
    l->table = take(4 * d4);
    l->kpack = take((size_t)l->head_pad); l->khead = take((size_t)l->head_pad * 4);
    l->img8 = take((size_t)slots * (size_t)(D + 1) * SC_SLAB);
    l->head_img = take((size_t)slots * (size_t)l->head_pad * SC_SLAB);
    l->normp = take((size_t)slots * SC_SLAB * 4);
    const size_t m4 = M >= SC_ORDER_MIN ? (size_t)((M + SC_SLAB - 1) / SC_SLAB * SC_SLAB) * 4 : 0;
    l->units = take(m4); l->unit_norm = take(m4); l->unit_tmp = take(2 * m4);
    l->rank_of = take(m4); l->picks = take(2 * m4);
    // (a search on its own sweeps one order after the other)
    l->ord8 = l->img8; l->ord_head = l->head_img; l->ord_normp = l->normp;
    if (ord_slots && m4) {
        l->ord8 = take((size_t)ord_slots * (size_t)(D + 1) * SC_SLAB);
        l->ord_head = take((size_t)ord_slots * (size_t)l->head_pad * SC_SLAB);
        l->ord_normp = take((size_t)ord_slots * SC_SLAB * 4);
    }
}

void screen_layout(int64_t D, int64_t M, int64_t N, int head, int64_t chunk, bool top2, int sms,
                   ScreenLayout *l)
{
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t at = off; off = up256(off + bytes); return at; };
    l->n_pad = (N + SC_DOCS - 1) / SC_DOCS * SC_DOCS;
    l->head_pad = (head + 127) / 128 * 128;
    const int64_t all = (M + SC_SLAB - 1) / SC_SLAB;
    l->chunk_slabs = chunk / SC_SLAB < all ? chunk / SC_SLAB : all;
    const int64_t launches = (all + l->chunk_slabs - 1) / l->chunk_slabs;
    const int64_t blocks = l->n_pad / SC_DOCS, slabs = (all + launches - 1) / launches;
    l->splits = screen_splits(blocks, slabs, sms);
    const size_t n4 = (size_t)l->n_pad * 4;
    const int64_t room = screen_split_blocks(blocks, slabs, sms);
    const size_t stripes = (size_t)room * SC_DOCS * 4;
    // (what they take together is within `room`, as screen_splits has it)
    const int64_t most = blocks > 0 ? room / blocks : 1, cap = slabs < 16 ? slabs : 16;
    l->most_splits = (int)(most < cap ? most : cap);
    if (l->most_splits < l->splits) l->most_splits = l->splits;
    codebook_layout(D, M, l->chunk_slabs, 0, 1, take, l);
    // a quarter of the launches' slabs: far beyond that the order of the map is the better one
    l->ord_launches = launches <= SC_MAX_LAUNCHES ? (launches + 3) / 4 : 0;
    l->sample = take((size_t)SC_SAMPLE * (size_t)((M + SC_GROUP - 1) / SC_GROUP) * 4);
    l->window = take(n4);
    l->amin = take(n4); l->amin2 = top2 ? take(n4) : l->amin;
    l->cval = take(stripes * sizeof(float2)); l->cmask = take(stripes * sizeof(uint4));
    l->cval2 = top2 ? take(stripes * sizeof(float)) : l->cval;
    l->lcount = take(n4);
    l->lists = take((size_t)l->n_pad * SC_LIST_BYTES);
    const bool order = M >= SC_ORDER_MIN;
    l->reach = take(order ? 2 * n4 : 0);
    l->items = take(order ? (size_t)blocks * SC_PARTS * sizeof(uint2) : 0);
    l->tickets = take(order && launches <= SC_MAX_LAUNCHES ? (size_t)launches * (SC_PARTS + 1) * 4 : 0);
    l->nat_list = take(order ? (size_t)blocks * 4 : 0);
    l->total = off;
}

void screen_shared_layout(int64_t D, int64_t M, int head, int64_t chunk, ScreenLayout *l)
{
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t at = off; off = up256(off + bytes); return at; };
    l->head_pad = (head + 127) / 128 * 128;
    const int64_t all = (M + SC_SLAB - 1) / SC_SLAB;
    l->chunk_slabs = chunk / SC_SLAB < all ? chunk / SC_SLAB : all;
    const int64_t launches = (all + l->chunk_slabs - 1) / l->chunk_slabs;
    l->ord_launches = launches <= SC_MAX_LAUNCHES ? (launches + 3) / 4 : 0;
    codebook_layout(D, M, launches * l->chunk_slabs, l->ord_launches * l->chunk_slabs, 2, take, l);
    l->rank = take((size_t)D * 2); l->feat = take((size_t)D * 2);
    l->total = off;
    l->map_total = off - (l->ord8 == l->img8 ? 0 : l->rank - l->ord8);
}

// ---- ranges of the rows -------------------------------------------------------------------
__device__ __forceinline__ float screen_ld(const float *p) { return __ldg(p); }
__device__ __forceinline__ float screen_ld(const __half *p) { return __half2float(__ldg(p)); }
__device__ __forceinline__ void screen_ld16(const float *p, float v[4])
{
    const float4 t = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void screen_ld16(const __half *p, float v[4])
{
    const uint2 t = __ldg(reinterpret_cast<const uint2 *>(p));
    const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&t.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&t.y));
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// A few documents, evenly through the corpus, against all units in fp32: the smallest value of each 8-unit
// group.  From these the windows' kernel sees how much of the map their windows hold.  A block takes a document
// and 128 units, each of its warps an eighth of the list (one warp for all of it: 26 us longer than the rest of
// the kernel where a list of 400 ids is met).  Its blocks run beside those that read the codebook anyway.
__device__ __forceinline__ int64_t screen_sample_doc(int s, int sampled, int64_t N) { return (2 * s + 1) * N / (2 * sampled); }

template <typename WT, bool VEC>
__device__ __forceinline__ void screen_sample(const WT *__restrict__ W, int64_t D, int64_t M, const float *__restrict__ norms,
                                              const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                                              int64_t N, int sampled, int64_t item, float *__restrict__ groups,
                                              [[maybe_unused]] uint32_t *status)
{
    constexpr int R = VEC ? 8 : 2;                   // rows in flight
    __shared__ float4 part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t pieces = (M + 127) / 128;
    const int sd = (int)(item / pieces);
    const int64_t i = screen_sample_doc(sd, sampled, N), j = item % pieces * 128 + 4 * lane;
    const int first = __ldg(rowptr + i), last = __ldg(rowptr + i + 1), share = (last - first + 7) / 8;
    const int beg = min(first + warp * share, last), end = min(beg + share, last);
    const WT *col = W + (VEC && j < M ? j : 0);
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int e0 = beg; e0 < end; e0 += 32) {
        const int mine = e0 + lane < end ? __ldg(colidx + e0 + lane) : 0, c = min(32, end - e0);
        for (int q = 0; q < c; q += R) {
            float v[R][4];
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const uint32_t f = BMU_IDX((uint32_t)__shfl_sync(0xffffffffu, mine, q + u), D, status);
#pragma unroll
                for (int x = 0; x < 4; ++x) v[u][x] = 0.f;
                if (q + u < c) {
                    if (VEC) screen_ld16(col + (int64_t)f * M, v[u]);
                    else {
#pragma unroll
                        for (int x = 0; x < 4; ++x) v[u][x] = screen_ld(W + (int64_t)f * M + (j + x < M ? j + x : 0));
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < R; ++u)
#pragma unroll
                for (int x = 0; x < 4; ++x) s[x] += v[u][x];
        }
    }
    part[warp][lane] = make_float4(s[0], s[1], s[2], s[3]);
    __syncthreads();
    if (warp) return;
#pragma unroll
    for (int w = 1; w < 8; ++w) {
        const float4 t = part[w][lane];
        s[0] += t.x; s[1] += t.y; s[2] += t.z; s[3] += t.w;
    }
    float least = CUDART_INF_F;
#pragma unroll
    for (int x = 0; x < 4; ++x)
        if (j + x < M) least = fminf(least, fmaf(-2.f, s[x], __ldg(norms + j + x)));
    least = fminf(least, __shfl_xor_sync(0xffffffffu, least, 1));
    if (!(lane & 1) && j < M) groups[(int64_t)sd * ((M + SC_GROUP - 1) / SC_GROUP) + j / SC_GROUP] = least;
}

// Smallest and largest weight of each row: one read of the codebook.  BW warps take a row.  Beside
// them the largest range of the head rows (most[0 .. 7]) and of the others (most[8 .. 15]) and the
// largest |norm| (most[16 .. 23]), as bit patterns of non-negative floats; each eight times, a block
// adds to one of them (thousands of atomics on one word: 10 us for 4096 rows of 1024, 4.3 so).
// The first blocks sample documents (above).
template <typename WT, bool VEC, int BW>
__global__ void __launch_bounds__(256, VEC ? 4 : 6)
screen_range_kernel(const WT *__restrict__ W, int64_t D, int64_t M, const float *__restrict__ norms,
                    const uint16_t *__restrict__ rank, int32_t head, float *__restrict__ rmin,
                    float *__restrict__ rmax, uint32_t *__restrict__ most, const int32_t *__restrict__ rowptr,
                    const int32_t *__restrict__ colidx, int64_t N, int sampled, int sample_blocks,
                    float *__restrict__ groups, uint32_t *status)
{
    if ((int)blockIdx.x < sample_blocks) {
        screen_sample<WT, VEC>(W, D, M, norms, rowptr, colidx, N, sampled, blockIdx.x, groups, status);
        return;
    }
    const unsigned block = blockIdx.x - sample_blocks, blocks = gridDim.x - sample_blocks;
    constexpr int ROWS = 8 / BW;
    __shared__ float s_lo[8], s_hi[8];
    __shared__ uint32_t s_most[3];
    if (threadIdx.x < 3) s_most[threadIdx.x] = 0u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t f = (int64_t)block * ROWS + warp / BW;
    const int part = (warp % BW) * 32 + lane;
    float lo = CUDART_INF_F, hi = -CUDART_INF_F;
    if (f < D) {
        const WT *row = W + f * M;
        if (VEC) {
            const int64_t n4 = M / 4;
            int64_t i = part;
            for (; i + 3 * BW * 32 < n4; i += 4 * BW * 32) {
                float v[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) screen_ld16(row + (i + (int64_t)u * BW * 32) * 4, v[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int c = 0; c < 4; ++c) { lo = fminf(lo, v[u][c]); hi = fmaxf(hi, v[u][c]); }
            }
            for (; i < n4; i += BW * 32) {
                float v[4];
                screen_ld16(row + i * 4, v);
#pragma unroll
                for (int c = 0; c < 4; ++c) { lo = fminf(lo, v[c]); hi = fmaxf(hi, v[c]); }
            }
        } else {
            for (int64_t i = part; i < M; i += BW * 32) {
                const float v = screen_ld(row + i);
                lo = fminf(lo, v); hi = fmaxf(hi, v);
            }
        }
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, m));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, m));
    }
    if (lane == 0) { s_lo[warp] = lo; s_hi[warp] = hi; }
    __syncthreads();
    if (threadIdx.x < ROWS && (int64_t)block * ROWS + threadIdx.x < D) {
        for (int w = 0; w < BW; ++w) {
            lo = w ? fminf(lo, s_lo[threadIdx.x * BW + w]) : s_lo[threadIdx.x * BW];
            hi = w ? fmaxf(hi, s_hi[threadIdx.x * BW + w]) : s_hi[threadIdx.x * BW];
        }
        const int64_t row = (int64_t)block * ROWS + threadIdx.x;
        rmin[row] = lo;
        rmax[row] = hi;
        atomicMax(&s_most[(rank ? (int)rank[row] : (int)row) < head ? 0 : 1], __float_as_uint(__fsub_ru(hi, lo)));
    }
    uint32_t nm = 0;
    u64 least = KEY_WORST;                                 // (a thread's units are all even or all odd)
    for (int64_t j = (int64_t)block * 256 + threadIdx.x; j < M; j += (int64_t)blocks * 256)
    {
        // (a unit at infinity is never within a finite window: it widens nobody's)
        const float v = __ldg(norms + j);
        const uint32_t n = __float_as_uint(fabsf(v));
        if (n < 0x7f800000u) { nm = max(nm, n); least = min(least, make_key(v, (int32_t)j)); }
    }
    if (M >= SC_ORDER_MIN && __any_sync(0xffffffffu, least != KEY_WORST)) {
#pragma unroll
        for (int m = 16; m > 1; m >>= 1) least = min(least, __shfl_xor_sync(0xffffffffu, least, m));
        // (kept as complements: the words begin as zeros)
        u64 *to = reinterpret_cast<u64 *>(status + STATUS_REFS) + 8 * (lane & 1) + (block & 7);
        if (lane < 2 && ~least > *reinterpret_cast<volatile u64 *>(to)) atomicMax(to, ~least);
    }
    nm = __reduce_max_sync(0xffffffffu, nm);
    if (lane == 0 && nm > 0) atomicMax(&s_most[2], nm);
    __syncthreads();
    if (threadIdx.x < 3) {
        uint32_t *to = most + 8 * threadIdx.x + (block & 7);
        const uint32_t v = s_most[threadIdx.x];
        if (v > *reinterpret_cast<volatile uint32_t *>(to)) atomicMax(to, v);
    }
}

// ---- steps and error bounds ----------------------------------------------------------------
// The integer gathered sum of a document lives in 16 bits: with lists of up to L gathered ids a
// code may be 65535 / L at most.  255 up to 257 ids; longer lists cost all documents resolution, down to
// 63, documents beyond that (1040 gathered ids) get an infinite window and are evaluated whole.  So are
// a few that are much longer than the rest: one list of 1000 ids among 100,000 documents on a trained
// 64 x 64 map took the search from 1.85 to 2.39 ms (coarser codes, and a tile that the others wait for).
static const int SC_Q_MIN = 63, SC_Q_TOP = 255;

// The longest list that counts for the codes: that of the tile of rank `few` if the longest of all is more
// than half as long again.  (Lengths that taper off keep their longest.)
__device__ __forceinline__ uint32_t screen_longest(const uint32_t *tile_len, int64_t few)
{
    const uint32_t longest = tile_len[0] & 0xffffu, rest = tile_len[few] & 0xffffu;
    return longest > 65535u / SC_Q_TOP && 2u * longest > 3u * rest ? max(rest, 65535u / SC_Q_TOP) : longest;
}

// The gathered rows share one step d_tail = (largest range) / q_max; a head row has the step k d_head
// with an integer k of its own (its entries of X_head are k instead of 1), so that rows of small range
// keep their resolution.  table[f] = error in the head's image (or the gathered one's), error in the
// gathered image (the last bit of the first: whether the row is in the head); and as pairs of 16 bits, rounded to the
// safe side, largest |w| and the range, and by how much the two reference units lie above the smallest weight.
__device__ __forceinline__ uint32_t screen_up16(float x) { return (__float_as_uint(x) + 0xffffu) >> 16; }
__device__ __forceinline__ float screen_lo16(uint32_t x) { return __uint_as_float(x << 16); }
__device__ __forceinline__ float screen_hi16(uint32_t x) { return __uint_as_float(x & 0xffff0000u); }

template <typename WT>
__global__ void __launch_bounds__(256)
screen_table_kernel(const WT *__restrict__ W, int64_t M, const float *__restrict__ norms, const uint32_t *status, const float *rmin, const float *rmax, int32_t D, int32_t head,
                    int32_t head_pad, const uint16_t *__restrict__ feat, const uint16_t *__restrict__ rank,
                    const uint32_t *__restrict__ tile_len, int64_t few, const uint32_t *most,
                    const float *earlier, int sampled, float *__restrict__ scalars, uint4 *__restrict__ table,
                    unsigned char *__restrict__ kpack, float *__restrict__ khead)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    uint32_t m3[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        m3[c] = 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k) m3[c] = max(m3[c], most[8 * c + k]);
    }
    const float rh = earlier ? earlier[8] : __uint_as_float(m3[0]), rt = earlier ? earlier[9] : __uint_as_float(m3[1]);
    const float norm = earlier ? earlier[5] : __uint_as_float(m3[2]);
    int32_t ref[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        u64 k = 0ull;
        if (M >= SC_ORDER_MIN) {
#pragma unroll
            for (int x = 0; x < 8; ++x) k = max(k, reinterpret_cast<const u64 *>(status + STATUS_REFS)[8 * c + x]);
        }
        ref[c] = earlier ? __float_as_int(earlier[SC_REF + c]) : k ? (int32_t)(uint32_t)~k : -1;
    }
    const uint32_t longest = screen_longest(tile_len, few);
    int q_max = longest <= 65535u / SC_Q_TOP ? SC_Q_TOP : max(SC_Q_MIN, min(SC_Q_TOP, (int)(65535u / longest)));
    const bool stand = earlier && (int)earlier[4] <= q_max;      // images of fewer steps do as well
    if (stand) q_max = (int)earlier[4];
    // (not below 1e-35, so that the reciprocals stay finite)
    const float dh = fmaxf(__fdiv_ru(rh, 255.f * SC_K_MAX), 1e-35f);
    const float dt = fmaxf(__fdiv_ru(rt, (float)q_max), 1e-35f);
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i == 0) {
        scalars[0] = -2.f * dh; scalars[1] = -2.f * dt;
        scalars[2] = 1.f / dt; scalars[3] = stand ? 1.f : 0.f; scalars[4] = (float)q_max;
        scalars[5] = norm; scalars[6] = (float)(65535 / q_max);
        scalars[7] = stand && __float_as_uint(earlier[SC_NATMADE]) ? 0.f : 1.f; scalars[8] = rh; scalars[9] = rt;
        scalars[SC_VOTES] = earlier ? earlier[SC_VOTES] : __uint_as_float(0u);
        // (screen_order_kernel decides otherwise)
        scalars[SC_ORDERED] = __uint_as_float(0u);
        scalars[SC_NAT] = __uint_as_float(SC_ALL); scalars[SC_NATMADE] = __uint_as_float(1u);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            scalars[SC_REF + c] = __int_as_float(ref[c]);
            scalars[SC_REFN + c] = ref[c] < 0 ? CUDART_INF_F : __ldg(norms + ref[c]);
        }
        scalars[SC_SAMPLED] = earlier ? earlier[SC_SAMPLED] : __uint_as_float((uint32_t)sampled);
    }
    // errors: half a step, widened by 2^-10 for the roundings of the coding itself
    const float half = 0.5f * (1.f + 1.f / 1024.f);
    auto scale = [&](float range) {
        return rh > 0.f ? fminf(fmaxf(ceilf(range / rh * (float)SC_K_MAX), 1.f), (float)SC_K_MAX) : 1.f;
    };
    if (i < D) {
        const float range = __fsub_ru(rmax[i], rmin[i]);
        const bool in = (rank ? (int)rank[i] : i) < head;
        float tail = half * dt;
        if (range > dt * (float)q_max)                 // codes of this row saturate in the gathered image
            tail += __fsub_ru(range, __fmul_rd(dt, (float)q_max)) * (1.f + 1.f / 1024.f);
        float e = tail;
        if (in) {
            const float k = scale(range);
            e = half * k * dh;
            if (range > 255.f * k * dh) e += __fsub_ru(range, __fmul_rd(255.f * k, dh)) * (1.f + 1.f / 1024.f);
        }
        float above[2];
#pragma unroll
        for (int c = 0; c < 2; ++c)
            above[c] = ref[c] < 0 ? 0.f : __fsub_rd(screen_ld(W + (int64_t)i * M + ref[c]), rmin[i]);
        table[i] = make_uint4(((__float_as_uint(e) + 1u) & ~1u) | (in ? 1u : 0u), __float_as_uint(tail),
                              screen_up16(fmaxf(fabsf(rmin[i]), fabsf(rmax[i]))) | screen_up16(range) << 16,
                              __float_as_uint(above[0]) >> 16 | (__float_as_uint(above[1]) & 0xffff0000u));
    }
    if (i < head_pad) {
        const bool in = i < head && i < D;
        const int f = in && feat ? (int)feat[i] : i;
        const float k = in ? scale(__fsub_ru(rmax[f], rmin[f])) : 1.f;
        kpack[i] = in ? (unsigned char)k : 0;
        khead[i] = 1.f / (k * dh);
    }
}

// ---- windows: half a warp per planned document --------------------------------------------
// 2 B of what the rows of a document's ids bring; and, by `order`, how far it reaches: a bound of its smallest
// (TOP2: second smallest) approximate value from the reference units, which is their own value and B (and B once
// more, so that the bound holds for what the verify stage computes), and 2 R + 2 B.
struct ScreenWindow { float window, bound, reach; };

// ... by LANES lanes, the rest of the warp the same for another document; `there`: or there is none
template <int LANES>
__device__ __forceinline__ ScreenWindow screen_window_of(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                                                         int64_t i, const uint32_t *__restrict__ key,
                                                         const uint4 *table, const float *scalars,
                                                         bool there, bool order, bool top2,
                                                         [[maybe_unused]] int64_t D, [[maybe_unused]] uint32_t *status)
{
    const int lane = threadIdx.x & (LANES - 1);
    const int beg = there ? __ldg(rowptr + i) : 0, end = there ? __ldg(rowptr + i + 1) : 0;
    float en = 0.f, eo = 0.f, aa = 0.f, rr = 0.f, ra = 0.f, rb = 0.f;
    uint32_t in = 0u;
    for (int e0 = beg; e0 < end; e0 += 4 * LANES) {
        int f[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = e0 + LANES * u + lane;
            f[u] = e < end ? (int)BMU_IDX((uint32_t)__ldg(colidx + e), D, status) : -1;
        }
        uint4 t[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) t[u] = f[u] >= 0 ? table[f[u]] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            en += __uint_as_float(t[u].x); eo += __uint_as_float(t[u].y); aa += screen_lo16(t[u].z); in |= t[u].x;
            if (order) { rr += screen_hi16(t[u].z); ra += screen_lo16(t[u].w); rb += screen_hi16(t[u].w); }
        }
    }
    __syncwarp();
    in = __ballot_sync(0xffffffffu, in & 1u) & (LANES == 32 ? 0xffffffffu : threadIdx.x & 16 ? 0xffff0000u : 0xffffu);
#pragma unroll
    for (int m = LANES / 2; m > 0; m >>= 1) {
        en += __shfl_xor_sync(0xffffffffu, en, m);
        eo += __shfl_xor_sync(0xffffffffu, eo, m);
        aa += __shfl_xor_sync(0xffffffffu, aa, m);
        if (order) {
            rr += __shfl_xor_sync(0xffffffffu, rr, m);
            ra += __shfl_xor_sync(0xffffffffu, ra, m);
            rb += __shfl_xor_sync(0xffffffffu, rb, m);
        }
    }
    // a list that repeats a head id is gathered whole
    const float n = (float)(end - beg), gathered = there ? (float)key[i] : 0.f;
    const float E = in && gathered == n ? eo : en;
    float B = 2.f * E + 1.1920929e-7f * (n * aa + 4.f * scalars[5] + 8.f * aa);
    const float wide = 1.f + 1.f / 4096.f + 2.f * n * 1.1920929e-7f;    // the roundings of these sums themselves
    B *= wide;
    ScreenWindow w;
    w.window = (gathered > scalars[6] || !(B < 1e37f)) ? CUDART_INF_F : 2.f * B;
    w.bound = w.reach = CUDART_INF_F;
    if (order) {
        float va = scalars[SC_REFN] - 2.f * (ra * (2.f - wide)) + 2.f * B;
        float vb = scalars[SC_REFN + 1] - 2.f * (rb * (2.f - wide)) + 2.f * B;
        if (!(va < CUDART_INF_F)) va = CUDART_INF_F;               // (not a number either)
        if (!(vb < CUDART_INF_F)) vb = CUDART_INF_F;
        w.bound = top2 ? fmaxf(va, vb) : fminf(va, vb);
        w.reach = 2.f * rr * wide + 2.f * B;
    }
    return w;
}

// The first blocks, one per sampled document: how many of its groups lie within its window.
// Bound by the latency of its dependent loads: 39 us for 120,000 documents of 80 ids.  With a warp per document, whose
// reductions and last steps then serve one only, 57 (41 without the reaches).
__global__ void __launch_bounds__(256, 6)
screen_window_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                     const int32_t *__restrict__ perm, const uint32_t *__restrict__ key, int64_t N, int64_t n_pad,
                     const uint4 *table, float *scalars, int order, int top2,
                     float *__restrict__ window, float2 *__restrict__ reach, uint32_t *__restrict__ bound,
                     uint32_t *__restrict__ count, uint32_t *__restrict__ set_reach, int64_t D,
                     int sampled, const float *groups, int64_t M, uint32_t *__restrict__ status)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if ((int)blockIdx.x < sampled) {
        __shared__ float s_win, s_least[8];
        __shared__ uint32_t s_in[8];
        const int64_t n = (M + SC_GROUP - 1) / SC_GROUP;
        const float *of = groups + blockIdx.x * n;
        if (warp == 0) {
            const ScreenWindow w = screen_window_of<32>(rowptr, colidx, screen_sample_doc(blockIdx.x, sampled, N), key, table,
                                                        scalars, true, false, top2, D, status);
            if (lane == 0) s_win = w.window;
        }
        float least = CUDART_INF_F;
        for (int64_t g = threadIdx.x; g < n; g += 256) least = fminf(least, of[g]);
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) least = fminf(least, __shfl_xor_sync(0xffffffffu, least, m));
        if (lane == 0) s_least[warp] = least;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 8; ++w) least = fminf(least, s_least[w]);
        const float limit = least + s_win;
        uint32_t within = 0;
        for (int64_t g = threadIdx.x; g < n; g += 256) within += of[g] <= limit;
        within = __reduce_add_sync(0xffffffffu, within);
        if (lane == 0) s_in[warp] = within;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w) within += s_in[w];
            if (within > screen_dense_groups(M) || s_win == CUDART_INF_F)
                atomicAdd(reinterpret_cast<uint32_t *>(scalars) + SC_VOTES, 1u);
        }
        return;
    }
    // (n_pad is a multiple of the sixteen documents of a block, and so is a set of them)
    __shared__ uint32_t s_far[16];
    const int64_t p = ((int64_t)(blockIdx.x - sampled) * blockDim.x + threadIdx.x) >> 4;
    const bool there = p < N && !(*status & PLAN_STATUS_OVERFLOW);
    ScreenWindow w = screen_window_of<16>(rowptr, colidx, there ? perm[p] : 0, key, table, scalars, there, order, top2, D, status);
    if (!there) w.window = 0.f;
    if ((lane & 15) == 0) window[p] = w.window;
    if (!order) return;
    if ((lane & 15) == 0) {
        // (documents that are evaluated whole need no slab)
        const bool none = !there || w.window == CUDART_INF_F;
        const float t = none ? -CUDART_INF_F : w.bound + w.window + w.reach;
        reach[p] = make_float2(t == t ? t : CUDART_INF_F, w.reach);
        bound[p] = float_to_ordered(none ? -CUDART_INF_F : w.bound);
        count[p] = 0u;
        s_far[threadIdx.x >> 4] = none ? 0u : float_to_ordered(t == t ? t : CUDART_INF_F);
        const ScreenSteps steps(scalars);
        if (!none && t < steps.top) atomicAdd(status + STATUS_REACH + steps.of(t), 1u);
    }
    __syncthreads();
    if (threadIdx.x < 16) {
        const uint32_t far = __reduce_max_sync(0xffffu, s_far[threadIdx.x]);
        if (threadIdx.x == 0 && far) atomicMax(set_reach + p / SC_DOCS, far);
    }
}

template <typename WT>
static int launch_range(const WT *W, int64_t D, int64_t M, const float *norms, const uint16_t *rank, int head,
                        float *rmin, float *rmax, uint32_t *most, const int32_t *rowptr, const int32_t *colidx,
                        int64_t N, int sampled, float *sample, uint32_t *status, cudaStream_t s)
{
    const bool vec = M % 4 == 0 && (reinterpret_cast<uintptr_t>(W) & (4 * sizeof(WT) - 1)) == 0;
    const int64_t sb = (M + 127) / 128 * sampled;
    const unsigned blocks = (unsigned)sb + (M >= 8192 ? (unsigned)D : (unsigned)((D + 3) / 4));
#define BMU_RANGE(V, B) { screen_range_kernel<WT, V, B><<<blocks, 256, 0, s>>>(W, D, M, norms, rank, head, rmin, rmax, most, rowptr, colidx, N, sampled, (int)sb, sample, status); BMU_LAUNCHED(); }
    if (M >= 8192) { if (vec) BMU_RANGE(true, 8) else BMU_RANGE(false, 8) }
    else { if (vec) BMU_RANGE(true, 2) else BMU_RANGE(false, 2) }
#undef BMU_RANGE
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

int launch_screen_prepare(const void *W, int f16, int64_t D, int64_t M, const float *norms,
                          const int32_t *rowptr, const int32_t *colidx, int64_t N, int head,
                          const uint16_t *feat, const uint16_t *rank, const int32_t *perm,
                          const uint32_t *key, const uint32_t *tile_len, char *cb, const ScreenLayout &cl,
                          float *scalars, const float *earlier, float *sample, float *window, float2 *reach,
                          uint32_t *bound, uint32_t *count, uint32_t *set_reach, int64_t n_pad, bool top2,
                          uint32_t *status, cudaStream_t s)
{
    const int order = screen_order_possible(D, M, N);
    // (an earlier search of the same codebook has decided for this one too)
    const int sampled = earlier ? 0 : (int)(N < SC_SAMPLE ? N : SC_SAMPLE);
    float *rmin = reinterpret_cast<float *>(cb + cl.rmin), *rmax = reinterpret_cast<float *>(cb + cl.rmax);
    uint4 *table = reinterpret_cast<uint4 *>(cb + cl.table);
    uint32_t *most = status + STATUS_MAXIMA;
    if (!earlier) {
        const int rc = f16 ? launch_range(static_cast<const __half *>(W), D, M, norms, rank, head, rmin, rmax, most,
                                          rowptr, colidx, N, sampled, sample, status, s)
                           : launch_range(static_cast<const float *>(W), D, M, norms, rank, head, rmin, rmax, most,
                                          rowptr, colidx, N, sampled, sample, status, s);
        if (rc) return rc;
    }
    const int64_t rows = D > cl.head_pad ? D : cl.head_pad;
    // up to a thousandth of the tiles, or four where they are few (32 documents of 1000 ids: 27 us for 4,096 units)
    const int64_t tiles = (N + 7) / 8, four = tiles / 64 < 4 ? tiles / 64 : 4, few = tiles / 1024 > four ? tiles / 1024 : four;
    const auto tables = [&](auto w) {
        ScreenLaunch l((unsigned)((rows + 255) / 256), 256, s, !earlier);         // (behind the tiling pass: ordinary)
        const cudaError_t e = cudaLaunchKernelEx(
            &l.c, screen_table_kernel<std::remove_const_t<std::remove_pointer_t<decltype(w)>>>, w, M, norms, (const uint32_t *)status,
            (const float *)rmin, (const float *)rmax, (int32_t)D, head, cl.head_pad, feat, rank, tile_len, few,
            (const uint32_t *)most, earlier, sampled, scalars, table, reinterpret_cast<unsigned char *>(cb + cl.kpack),
            reinterpret_cast<float *>(cb + cl.khead));
        BMU_LAUNCHED();
        return e;
    };
    BMU_CUDA(f16 ? tables(static_cast<const __half *>(W)) : tables(static_cast<const float *>(W)));
    ScreenLaunch l((unsigned)(sampled + n_pad / 16), 256, s, true);
    BMU_CUDA(cudaLaunchKernelEx(&l.c, screen_window_kernel, rowptr, colidx, perm, key, N, n_pad, (const uint4 *)table, scalars,
                                order, (int)top2, window, reach, bound, count, set_reach, D, sampled, (const float *)sample,
                                M, status));
    BMU_LAUNCHED();
    return BMU_OK;
}

// ---- the images -------------------------------------------------------------------------
// Where neuron jn of a slab sits.  The sweep's lane i of a document (i = 0 .. 3) owns the group
// of neurons 32i .. 32i + 31: in the MMA tile these are columns 8k + 2i + {0, 1} (what the
// tensor-memory load hands that lane), in a gathered row the 16-byte pieces i and i + 4 (sixteen
// neurons each), four neurons per 32-bit word with the even bytes holding the first two.
__device__ __forceinline__ int screen_col(int jn) { return 8 * ((jn & 31) >> 1) + 2 * (jn >> 5) + (jn & 1); }

// The code of a weight in the low byte: 2^23 + an integer, rounded to nearest by the addition.
__device__ __forceinline__ uint32_t screen_code(float w, float c, float inv, float q_max)
{
    return __float_as_uint(fminf(fmaxf((w - c) * inv, 0.f), q_max) + 8388608.f);
}
// the low bytes of four words
__device__ __forceinline__ uint32_t screen_pack(uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3)
{
    return __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
}

// Gathered image, blocks of IMAGE_ROWS rows and one slab: a lane codes four neurons of a row, or eight of
// an fp16 row (sixteen bytes), a warp takes four such instructions' rows and stores 128 bytes a row.
// (`block` counts from 0.)  16384 x 16384 floats take 242 us, 5.9 TB/s with what is written; 65536 halves
// 755 us with eight bytes a lane, 630 with sixteen.
template <typename WT, bool VEC> constexpr int IMAGE_V = VEC ? 16 / (int)sizeof(WT) : 4;
template <typename WT, bool VEC> constexpr int IMAGE_ROWS = 8 * 4 * IMAGE_V<WT, VEC> / 4;

__device__ __forceinline__ void screen_ld_vec(const float *p, float v[4]) { screen_ld16(p, v); }
__device__ __forceinline__ void screen_ld_vec(const __half *p, float v[8])
{
    const uint4 t = __ldg(reinterpret_cast<const uint4 *>(p));
    const uint32_t x[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&x[i]));
        v[2 * i] = a.x; v[2 * i + 1] = a.y;
    }
}

template <typename WT, bool VEC>
__device__ __forceinline__ void screen_image_block(const WT *__restrict__ W, int64_t D, int64_t M, int64_t slab,
                                                   int64_t j_slab, int block, const float *rmin,
                                                   const float *scalars, const float *__restrict__ norms,
                                                   unsigned char *__restrict__ img8, float *__restrict__ normp)
{
    constexpr int V = IMAGE_V<WT, VEC>, LPR = SC_SLAB / V, RPI = 32 / LPR;     // lanes per row, rows per instruction
    constexpr int R = 4;                                   // instructions per warp, loads issued together
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, l4 = (lane % LPR) * (V / 4);
    const int64_t j = j_slab + 4 * l4;
    const float inv = scalars[2], q_max = scalars[4];
    const int i = l4 >> 3, hb = (l4 >> 2) & 1, wd = l4 & 3;
    unsigned char *out = img8 + (size_t)slab * (D + 1) * SC_SLAB + (hb * 4 + i) * 16 + wd * 4;
    const int64_t f0 = ((int64_t)block * 8 + warp) * R * RPI + lane / LPR;
    float v[R][V], c[R];
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int64_t f = f0 + u * RPI;
        c[u] = f < D ? rmin[f] : 0.f;
#pragma unroll
        for (int e = 0; e < V; ++e) v[u][e] = c[u];
        if (f < D) {
            if constexpr (VEC) { if (j < M) screen_ld_vec(W + f * M + j, v[u]); }
            else {
#pragma unroll
                for (int e = 0; e < V; ++e) if (j + e < M) v[u][e] = screen_ld(W + f * M + j + e);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int64_t f = f0 + u * RPI;
        if (f > D) break;                                  // row D: zeros (all codes of "c" are 0)
        uint32_t q[V / 4];
#pragma unroll
        for (int w = 0; w < V / 4; ++w)
            q[w] = screen_pack(screen_code(v[u][4 * w], c[u], inv, q_max), screen_code(v[u][4 * w + 2], c[u], inv, q_max),
                               screen_code(v[u][4 * w + 1], c[u], inv, q_max), screen_code(v[u][4 * w + 3], c[u], inv, q_max));
        if constexpr (V == 8) *reinterpret_cast<uint2 *>(out + f * SC_SLAB) = make_uint2(q[0], q[1]);
        else *reinterpret_cast<uint32_t *>(out + f * SC_SLAB) = q[0];
    }
    // the norms, in the order the sweep's lanes read them: piece m of lane i = neurons 32i + 4m ..
    if (block == 0 && threadIdx.x < SC_SLAB) {
        const int jn = threadIdx.x;
        const int64_t jj = j_slab + jn;
        normp[slab * SC_SLAB + ((jn & 31) >> 2) * 16 + (jn >> 5) * 4 + (jn & 3)] =
            jj < M ? norms[jj] : CUDART_INF_F;
    }
}

// Head image, blocks of 32 head features and one slab: a thread codes four features of four neighbouring
// neurons, and through shared memory the sixteen bytes of one core-matrix row (sixteen features of a
// neuron) leave at once.  (With a thread per core-matrix row, loading one weight of sixteen rows, the head
// of 1536 took 230 of the 860 us of both fp16 images of 65536 units; 85 so.)
template <typename WT, bool VEC>
__device__ __forceinline__ void screen_head_block(const WT *__restrict__ W, int64_t D, int64_t M, int64_t slab,
                                                  int64_t j_slab, int block, int32_t head, int32_t head_pad,
                                                  const uint16_t *__restrict__ feat, const float *rmin,
                                                  const float *khead, unsigned char *__restrict__ img)
{
    constexpr int P = 9;                                   // words per neuron: eight, odd pitch
    __shared__ uint32_t tile[SC_SLAB * P];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j = j_slab + 4 * lane;
    float v[4][4], c[4], k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int h = block * 32 + 4 * warp + u;
        k[u] = khead[h];
        c[u] = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) v[u][e] = 0.f;
        if (h < head && h < D) {
            const int64_t f = feat ? (int64_t)__ldg(feat + h) : (int64_t)h;
            c[u] = rmin[f];
            if (VEC) { if (j < M) screen_ld16(W + f * M + j, v[u]); }
            else {
#pragma unroll
                for (int e = 0; e < 4; ++e) if (j + e < M) v[u][e] = screen_ld(W + f * M + j + e);
            }
        }
    }
    uint32_t q[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        uint32_t b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) b[u] = screen_code(j + e < M ? v[u][e] : c[u], c[u], k[u], 255.f);
        q[e] = screen_pack(b[0], b[1], b[2], b[3]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {                          // (in an order that hits 32 banks)
        const int e = (i + (lane >> 3)) & 3;
        const uint32_t lo = (e & 1) ? q[1] : q[0], hi = (e & 1) ? q[3] : q[2];
        tile[(4 * lane + e) * P + warp] = (e & 2) ? hi : lo;
    }
    __syncthreads();
    const int jn = threadIdx.x & 127, half = threadIdx.x >> 7, h0 = block * 32 + half * 16;
    const int n = screen_col(jn);
    const uint32_t *from = tile + jn * P + 4 * half;
    unsigned char *dst = img + ((size_t)slab * (head_pad / 128) + (h0 >> 7)) * MMA_STAGE_BYTES +
                         (n >> 3) * 1024 + ((h0 & 127) >> 4) * 128 + (n & 7) * 16;
    *reinterpret_cast<uint4 *>(dst) = make_uint4(from[0], from[1], from[2], from[3]);
    __syncthreads();                                       // (the caller may take another slab)
}

// ---- images of slabs in the order of the norms --------------------------------------------
// A launch's units, in the order of the map (`picks`: unit, place in the order of the norms; no unit beyond the
// last), so that neighbouring lanes read neighbouring weights of a row; the bytes meet in shared memory.  What is
// read are the sectors that hold a unit: some of a row where few units are needed, all of it, once, where many are.
// (A lane per place, its weight wherever it lies: 463 us for 32 slabs of 64 x 64, D = 16,384.)
static const int ORD_ROWS = 4;                             // rows a block takes at a time
static const int ORD_HEAD = 16;                            // head features a block takes at a time

template <typename WT>
__device__ __forceinline__ void ordered_rows(const WT *__restrict__ W, int64_t D, int64_t M, int64_t f0, int slots,
                                             int place0, const int2 *picks, const float *rmin,
                                             float inv, float q_max, unsigned char *__restrict__ img8)
{
    __shared__ __align__(16) unsigned char bytes[ORD_ROWS * SC_MAX_SLABS * SC_SLAB];
    float c[ORD_ROWS];
    const WT *row[ORD_ROWS];
#pragma unroll
    for (int u = 0; u < ORD_ROWS; ++u) {
        const int64_t f = f0 + u < D ? f0 + u : D - 1;
        row[u] = W + f * M;
        c[u] = rmin[f];
    }
    for (int i = threadIdx.x; i < slots; i += 256) {
        const int2 t = picks[i];
        const int at = t.y - place0, jn = at & (SC_SLAB - 1);
        // in the slab's 128 bytes of a row: as screen_image_block has it
        unsigned char *to = bytes + (at - jn) * ORD_ROWS + (((jn >> 4) & 1) * 4 + (jn >> 5)) * 16 + ((jn >> 2) & 3) * 4 +
                            ((jn & 1) << 1) + ((jn >> 1) & 1);
        float v[ORD_ROWS];
#pragma unroll
        for (int u = 0; u < ORD_ROWS; ++u) v[u] = t.x >= 0 && f0 + u < D ? screen_ld(row[u] + t.x) : c[u];
#pragma unroll
        for (int u = 0; u < ORD_ROWS; ++u) to[u * SC_SLAB] = (unsigned char)screen_code(v[u], c[u], inv, q_max);
    }
    __syncthreads();
    for (int v = threadIdx.x; v < slots * ORD_ROWS / 16; v += 256) {
        const int slab = v / (ORD_ROWS * 8), u = v / 8 % ORD_ROWS, piece = v % 8;
        if (f0 + u <= D)                                   // row D: zeros
            *reinterpret_cast<uint4 *>(img8 + ((size_t)slab * (D + 1) + f0 + u) * SC_SLAB + piece * 16) =
                reinterpret_cast<const uint4 *>(bytes)[v];
    }
    __syncthreads();
}

template <typename WT>
__device__ __forceinline__ void ordered_head(const WT *__restrict__ W, int64_t D, int64_t M, int h0, int slots, int place0,
                                             const int2 *picks, int32_t head, int32_t head_pad,
                                             const uint16_t *__restrict__ feat, const float *rmin,
                                             const float *khead, unsigned char *__restrict__ img)
{
    __shared__ float s_c[ORD_HEAD], s_k[ORD_HEAD];
    __shared__ int64_t s_row[ORD_HEAD];
    if (threadIdx.x < ORD_HEAD) {
        const int h = h0 + threadIdx.x;
        const bool in = h < head && h < D;
        const int64_t f = in ? (feat ? (int64_t)__ldg(feat + h) : (int64_t)h) : -1;
        s_row[threadIdx.x] = in ? f * M : -1;
        s_c[threadIdx.x] = in ? rmin[f] : 0.f;
        s_k[threadIdx.x] = khead[h];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < slots; i += 256) {
        asm volatile("" ::: "memory");                     // (or the sixteen rows' addresses are kept and spill)
        const int2 t = picks[i];
        const int at = t.y - place0, n = screen_col(at & (SC_SLAB - 1));
        uint32_t q[4];
#pragma unroll
        for (int w = 0; w < 4; w += 2) {                   // eight rows in flight
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int64_t r = s_row[4 * w + u];
                v[u] = t.x >= 0 && r >= 0 ? screen_ld(W + r + t.x) : s_c[4 * w + u];
            }
            uint32_t b[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) b[u] = screen_code(v[u], s_c[4 * w + u], s_k[4 * w + u], 255.f);
            q[w] = screen_pack(b[0], b[1], b[2], b[3]);
            q[w + 1] = screen_pack(b[4], b[5], b[6], b[7]);
        }
        unsigned char *dst = img + ((size_t)(at / SC_SLAB) * (head_pad / 128) + (h0 >> 7)) * MMA_STAGE_BYTES +
                             (n >> 3) * 1024 + ((h0 & 127) >> 4) * 128 + (n & 7) * 16;
        *reinterpret_cast<uint4 *>(dst) = make_uint4(q[0], q[1], q[2], q[3]);
    }
    __syncthreads();
}

// A warp per set of 128 documents: which of the launch's slabs any of them reaches, as items of up to SC_PART.
__device__ __forceinline__ void ordered_items(const OrderedImages &g, int set, int slabs, const float *unit_norm,
                                              const float *scalars)
{
    const int lane = threadIdx.x & 31;
    if (!(ordered_to_float(g.set_reach[set]) <= scalars[SC_TOP])) return;    // in the order of the map
    const float top = scalars[SC_DOC_TOP];
    float far = -CUDART_INF_F;
#pragma unroll
    for (int u = 0; u < SC_DOCS / 32; ++u) {
        const int64_t p = (int64_t)set * SC_DOCS + 32 * u + lane;
        const float2 r = g.reach[p];
        if (r.x > top) continue;                           // evaluated whole
        // (less what the launches before have found)
        far = fmaxf(far, g.first ? r.x : fminf(r.x, ordered_to_float(__ldcg(g.bound + p)) + g.window[p] + r.y));
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) far = fmaxf(far, __shfl_xor_sync(0xffffffffu, far, m));
    const bool in = lane < slabs && unit_norm[lane * SC_SLAB] <= far;
    const int n = __popc(__ballot_sync(0xffffffffu, in));  // (ascending: the first ones)
    if (lane < (n + SC_PART - 1) / SC_PART)
        g.items[(size_t)lane * g.sets + atomicAdd(g.tickets + lane, 1u)] =
            make_uint2((uint32_t)set, (uint32_t)(lane * SC_PART) | (uint32_t)min(n, (lane + 1) * SC_PART) << 16);
}

template <typename WT>
__global__ void __launch_bounds__(256, 6)
screen_ordered_image_kernel(const WT *__restrict__ W, int64_t D, int64_t M, const OrderedImages g,
                            const int2 *picks, const float *unit_norm, int32_t head_pad,
                            const uint16_t *__restrict__ feat, const float *rmin,
                            const float *khead, const float *scalars,
                            unsigned char *__restrict__ img8, unsigned char *__restrict__ head_img, float *__restrict__ normp)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!screen_ordered(scalars) || screen_whole(scalars)) return;
    const uint32_t *sc = reinterpret_cast<const uint32_t *>(scalars);
    const int slabs = (int)min((int64_t)g.n_slabs, (int64_t)sc[SC_NEEDED] - g.slab0);
    if (slabs <= 0) return;
    const int place0 = (int)g.slab0 * SC_SLAB, slots = slabs * SC_SLAB;
    const bool stand = sc[SC_STAND] != 0u;         // the images of an earlier search
    const int lists = (g.sets + 7) / 8, rows = (int)((D + ORD_ROWS) / ORD_ROWS), heads = head_pad / ORD_HEAD;
    const int all = stand ? lists : lists + heads + rows;
    for (int item = blockIdx.x; item < all; item += gridDim.x) {
        if (item < lists) {
            const int set = item * 8 + (threadIdx.x >> 5);
            if (set < g.sets) ordered_items(g, set, slabs, unit_norm + place0, scalars);
        } else if (item < lists + heads) {
            ordered_head(W, D, M, (item - lists) * ORD_HEAD, slots, place0, picks + place0, g.head, head_pad, feat, rmin, khead, head_img);
            if (item == lists)
                for (int x = threadIdx.x; x < slots; x += 256) {
                    const int jn = x & (SC_SLAB - 1);
                    normp[x - jn + ((jn & 31) >> 2) * 16 + (jn >> 5) * 4 + (jn & 3)] = unit_norm[place0 + x];
                }
        } else {
            ordered_rows(W, D, M, (int64_t)(item - lists - heads) * ORD_ROWS, slots, place0, picks + place0, rmin,
                         scalars[2], scalars[4], img8);
        }
    }
}

int launch_screen_ordered_images(const void *W, int f16, int64_t D, int64_t M, const OrderedImages &g,
                                 const uint16_t *feat, char *cb, const ScreenLayout &l, const float *scalars, int sms,
                                 cudaStream_t s)
{
    const auto go = [&](auto w) {
        ScreenLaunch p((unsigned)(6 * sms), 256, s, true);
        const cudaError_t e = cudaLaunchKernelEx(
            &p.c, screen_ordered_image_kernel<std::remove_const_t<std::remove_pointer_t<decltype(w)>>>, w, D, M, g,
            reinterpret_cast<const int2 *>(cb + l.picks), reinterpret_cast<const float *>(cb + l.unit_norm),
            (int32_t)l.head_pad, feat, reinterpret_cast<const float *>(cb + l.rmin), reinterpret_cast<const float *>(cb + l.khead),
            scalars, reinterpret_cast<unsigned char *>(cb + l.ord8) + (size_t)g.slot * (D + 1) * SC_SLAB,
            reinterpret_cast<unsigned char *>(cb + l.ord_head) + (size_t)g.slot * l.head_pad * SC_SLAB,
            reinterpret_cast<float *>(cb + l.ord_normp) + g.slot * SC_SLAB);
        BMU_LAUNCHED();
        return e;
    };
    BMU_CUDA(f16 ? go(static_cast<const __half *>(W)) : go(static_cast<const float *>(W)));
    return BMU_OK;
}

// Both images of a slab in one grid, the head's blocks in front.  LOOP: a block takes every gridDim.y-th
// slab -- slower where there is work (a shared codebook's images usually stand), 9 -> 3 us where not.
template <typename WT, bool VEC, bool LOOP>
__global__ void __launch_bounds__(256)
screen_image_kernel(const WT *__restrict__ W, int64_t D, int64_t M, int64_t k, int64_t launches, int64_t n_slabs,
                    int32_t head,
                    int32_t head_pad, const uint16_t *__restrict__ feat, const float *rmin,
                    const float *khead, const float *scalars,
                    const float *__restrict__ norms, unsigned char *__restrict__ img8,
                    unsigned char *__restrict__ head_img, float *__restrict__ normp)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // the images of an earlier search stand; or nothing is swept in this order
    if (scalars[7] == 0.f || screen_whole(scalars) || screen_natural(scalars) == 0u) return;
    const int heads = head_pad / 32;
    auto one = [&](const int64_t slab) {
        const int64_t j_slab = (k + launches * slab) * SC_SLAB;
        if ((int)blockIdx.x < heads)
            screen_head_block<WT, VEC>(W, D, M, slab, j_slab, (int)blockIdx.x, head, head_pad, feat, rmin, khead, head_img);
        else
            screen_image_block<WT, VEC>(W, D, M, slab, j_slab, (int)blockIdx.x - heads, rmin, scalars, norms, img8, normp);
    };
    if constexpr (LOOP)
        for (int64_t slab = blockIdx.y; slab < n_slabs; slab += gridDim.y) one(slab);
    else
        one(blockIdx.y);
}

template <typename WT>
static int launch_images(const WT *W, int64_t D, int64_t M, const float *norms, int64_t k,
                         int64_t launches, int64_t n_slabs, int64_t slot, int head, const uint16_t *feat, char *base,
                         const ScreenLayout &l, const float *scalars, bool expected, cudaStream_t s)
{
    const float *rmin = reinterpret_cast<const float *>(base + l.rmin);
    const float *khead = reinterpret_cast<const float *>(base + l.khead);
    unsigned char *img8 = reinterpret_cast<unsigned char *>(base + l.img8) + (size_t)slot * (D + 1) * SC_SLAB;
    unsigned char *head_img = reinterpret_cast<unsigned char *>(base + l.head_img) + (size_t)slot * l.head_pad * SC_SLAB;
    float *normp = reinterpret_cast<float *>(base + l.normp) + slot * SC_SLAB;
    const bool vec = M % (16 / sizeof(WT)) == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0;
    const int rows = vec ? IMAGE_ROWS<WT, true> : IMAGE_ROWS<WT, false>;
    const dim3 grid((unsigned)(l.head_pad / 32 + (D + 1 + rows - 1) / rows),
                    expected ? 1u : (unsigned)n_slabs);       // few blocks where there is likely nothing to do
    ScreenLaunch p(grid, 256, s, true);
#define BMU_IMG(V, L) { BMU_CUDA(cudaLaunchKernelEx(&p.c, screen_image_kernel<WT, V, L>, W, D, M, k, launches, n_slabs, (int32_t)head, (int32_t)l.head_pad, feat, rmin, khead, scalars, norms, img8, head_img, normp)); BMU_LAUNCHED(); }
    if (expected) { if (vec) BMU_IMG(true, true) else BMU_IMG(false, true) }
    else if (vec) BMU_IMG(true, false) else BMU_IMG(false, false)
#undef BMU_IMG
    return BMU_OK;
}

int launch_screen_quantize(const void *W, int f16, int64_t D, int64_t M, const float *norms,
                           int64_t k, int64_t launches, int64_t n_slabs, int64_t slot, int head,
                           const uint16_t *feat, char *cb, const ScreenLayout &cl, const float *scalars,
                           bool expected, cudaStream_t s)
{
    if (f16)
        return launch_images(static_cast<const __half *>(W), D, M, norms, k, launches, n_slabs, slot, head, feat, cb, cl, scalars, expected, s);
    return launch_images(static_cast<const float *>(W), D, M, norms, k, launches, n_slabs, slot, head, feat, cb, cl, scalars, expected, s);
}

}  // namespace bmu
