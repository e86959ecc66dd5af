// The screening sweep (screen.cuh): approximate distances of 128 documents x all neurons of a
// launch, from the 8-bit image of the codebook.
//
//   head   the sum over the H most frequent features is an integer matrix product on the tensor
//          cores (tcgen05.mma kind::i8, 128 documents x 128 neurons x 32 features, exact 32-bit
//          sums).  X_head -- a byte per document and feature: 0, or the feature's integer row
//          scale -- is the A operand and stays in TENSOR MEMORY for the whole launch (a lane per
//          document, a column per four features), so shared memory holds nothing but the ring of
//          W stages and L1 keeps its size for the gather.
//   tail   the other features are gathered: a warp carries 8 documents x 128 neurons, eight
//          lanes read the 128-byte piece of one document's row (16 neurons per lane), four
//          documents per instruction; bytes are summed in pairs of 16-bit fields, exactly.
//   end    of a slab: the two lanes that hold halves of the same document swap, so that a lane
//          has 32 consecutive neurons of one document -- the very elements the 16x256b
//          tensor-memory load hands it -- forms the distances, and keeps the smallest value, the
//          document's smallest over its four lanes, and a bit mask of the 8-neuron groups that came
//          within the window.  No index arithmetic: the verify stage finds the unit.
//
// The MMAs of the next slab run under the gather.  Waits are bounded and report through the
// status word.
//
// What bounds it (75,776 documents x 3,072 neurons, Zipf 1.1, 24 slabs in 477 us, and in 475 with a block per set of
// documents, of which the parts are): the latency of the gathered loads, 64 KB in flight per SM, which the registers of the tail warps bound; no unit is full
// (L1 data path 66 %, integer ALU 64, L2 55, tensor pipe 36).  The gather alone takes 373 us, the
// epilogue 85, and the head's MMAs (194 us alone) run underneath.  Six instead of the four instructions
// per two words of sc_add took 511 us where these took 507 at the time, three and two multiply-adds 513.  Nor did
// deeper rings, 7-bit codes, pairs of blocks that share the head's stages (524) or touching the next
// rows into L1 (525) help.  A head of 1024 with two accumulators is level with 1536 and one.
//
// The fp32 gather of sweep_mma2.cu, which it replaces for large sweeps, sits at the L2 -> SM path's
// ceiling with 4 bytes per update.  Whole searches before / after: 100,000 documents on a 512 x 512
// map 206.7 / 69.5 ms, 200,000 on a trained 128 x 128 map 32.8 / 10.9 ms, 120,000 on 64 x 64 4.76 /
// 1.71 ms, 60,000 against an fp16 256 x 256 map 22.7 / 11.3 ms.
//
// The blocks stay, one per SM, and take sets of 128 documents and stretches of slabs one after the other; barriers and
// accumulators go on from item to item: 200,000 documents on a trained 128 x 128 map 9.81 -> 9.49 ms, 30,011 on 75 x 75
// 686 -> 671 us; 120,000 on 64 x 64, D = 4,096, where slabs are short, 875 -> 885.
//
// ORDERED: slabs in the order of the norms (screen.cuh, screen_order.cu).  What differs:
//   items      a set of documents reaches a few slabs of a launch, another set many: (set, up to SC_PART slabs),
//              from the lists that screen_ordered_image_kernel makes, the first parts of all sets before the second ones.
//   stopping   a warp leaves an item at the first slab that no document of its tile reaches any more.
//   candidates the bound of a document's smallest value is good from the start and slabs with the smallest
//              norms come first, so that little is ever within a window: what is, is looked up once more, unit by
//              unit, and joins the document's one list.  Parts of the same set share list and bound by atomics.
//   head first once a slab has brought the warp no candidate, the next ones are looked at with the head's sums and the
//              most that the gathered rows could add; where that rules a slab out its rows are not gathered (for
//              120,000 documents on 64 x 64 the search 970 -> 885 us).
// The same documents take 1,255 us with all slabs in the order of the map; 100,000 on 512 x 512 57,000 and 1,500.  Bound by
// the latency of the gathered loads, and by meeting at an item's ends (a quarter of the stalls).

#include "screen.cuh"
#include "mma_ptx.cuh"

#include <math_constants.h>

#include <type_traits>

namespace bmu {

static const int SC_TAIL_WARPS = 16;
static const int SC_THREADS = (SC_TAIL_WARPS + 4) * 32;
static const int SC_TAIL_REGS = 112, SC_CTRL_REGS = 32;      // registers after the hand-over
// W ring: two stages of four blocks of 128 features (64 KB each).  The issuing warp spends some 300
// cycles per stage on its barriers that do not hide under the MMAs of a stage: stages of 16, 32,
// 48 and 64 KB took 515, 497, 491 and 483 us on the launch below.
static const int SC_KS = 4, SC_NS = 2;
// Tensor memory: the accumulators from column 0 -- two that alternate between slabs if X_head
// leaves room (up to 1024 features), else one --, X_head in the last head_pad / 4 columns.
static const size_t SC_SMEM = SC_NS * SC_KS * MMA_STAGE_BYTES + (2 * SC_NS + 5) * 8 + 8 + 2 * 16;

// Adds the sixteen bytes of two rows to a lane's sums.  acc[w] holds the sum of words w modulo 2^32,
// acc[4 + w] the 16-bit sums of their bytes 1 and 3; sc_even takes those out of the former.
__device__ __forceinline__ void sc_add(uint32_t acc[8], const uint4 a, const uint4 b)
{
    const uint32_t x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        acc[w] += x[w] + y[w];
        acc[4 + w] += __byte_perm(x[w], 0u, 0x4341) + __byte_perm(y[w], 0u, 0x4341);
    }
}
// the 16-bit sums of bytes 0 and 2 of word w
__device__ __forceinline__ uint32_t sc_even(uint32_t words, uint32_t odd) { return words - (odd << 8); }

__device__ __forceinline__ u64 sc_pack(float lo, float hi)
{
    return ((u64)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ u64 sc_fma2(u64 a, u64 b, u64 c)
{
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 sc_add2(u64 a, u64 b)
{
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// two distances: norms n2, integer head sums h0 and h1, two 16-bit gathered sums in t
__device__ __forceinline__ u64 sc_dist2(u64 n2, uint32_t h0, uint32_t h1, uint32_t t, u64 sh, u64 st, u64 minus_2p23)
{
    const u64 hf = sc_pack(__uint2float_rn(h0), __uint2float_rn(h1));
    // 2^23 + a 16-bit integer, assembled from bytes; the subtraction is exact
    const u64 tf = sc_add2(((u64)__byte_perm(t, 0x4b000000u, 0x7432) << 32) |
                           __byte_perm(t, 0x4b000000u, 0x7410), minus_2p23);
    return sc_fma2(tf, st, sc_fma2(hf, sh, n2));
}

// (all warps, from two places of the code)
__device__ __forceinline__ void block_sync() { asm volatile("barrier.sync 0, %0;" ::"n"(SC_THREADS) : "memory"); }

template <bool TOP2, bool ORDERED>
__global__ void __launch_bounds__(SC_THREADS, 1)
sweep_screen_kernel(const ScreenArgs a, const OrderedArgs o)
{
    constexpr int NS = SC_NS, KS = SC_KS, NTW = SC_TAIL_WARPS;
    extern __shared__ __align__(128) unsigned char smem[];
    u64 *bars = reinterpret_cast<u64 *>(smem + NS * KS * MMA_STAGE_BYTES);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * NS + 5);
    volatile uint32_t *abort_flag = tmem_slot + 1, *item_slot = tmem_slot + 2;       // (two items, four words each)
    const uint32_t wfull0 = mm_smem(bars), wempty0 = mm_smem(bars + NS);
    const uint32_t tfull0 = mm_smem(bars + 2 * NS), tempty0 = tfull0 + 16, drain = tfull0 + 32;
    const int two = a.head_pad <= 1024, x_col = 512 - a.head_pad / 4;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t natural = screen_natural(a.scalars);
    if (screen_whole(a.scalars) || (ORDERED ? !screen_ordered(a.scalars) : natural == 0u)) return;
    if (ORDERED && o.slab0 >= (int64_t)reinterpret_cast<const uint32_t *>(a.scalars)[SC_NEEDED]) return;

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int KB = a.head_pad / 128;
    if (threadIdx.x == 0) {
        for (int i = 0; i < NS; ++i) { mm_bar_init(wfull0 + 8 * i, 1); mm_bar_init(wempty0 + 8 * i, 1); }
        for (int i = 0; i < 2; ++i) { mm_bar_init(tfull0 + 8 * i, 1); mm_bar_init(tempty0 + 8 * i, NTW); }
        mm_bar_init(drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *abort_flag = 0u;
    }
    __syncthreads();
    if (warp == NTW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(mm_smem(tmem_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    mm_fence_before();
    __syncthreads();
    mm_fence_after();
    const uint32_t tmem = *tmem_slot;
    // The control warpgroup hands registers to the four tail warpgroups, whose loads in flight are bounded by theirs: the
    // block is launched with 96 per thread (640 x 96 = 61440 = 128 x 32 + 512 x 112), so the increase never waits for
    // registers that nobody releases (the launcher checks the build).
    // The loops over the items meet twice an item: X_head is in place; X_head has been read, for every accumulator has
    // been waited for, and the next item is known.
    int done = 0, turn = 0;                               // slabs before this item: which accumulator, which phase; items
    if (warp >= NTW) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(SC_CTRL_REGS));
    int slot = 0, issued = 0;                             // ring of W stages: the producer's and the issuer's
    uint32_t phase = warp == NTW ? 1u : 0u;               // (a fresh ring counts as empty)
    bool ok = true;
    // Item t into the place of the `to`-th one: set of documents (none: there are no more; a block that gave up: let the
    // grid drain), slabs, part.
    auto decode = [&](uint32_t t, int to) {
        uint32_t set = ~0u, range = 0u, part = 0u;
        if (*abort_flag || *reinterpret_cast<volatile uint32_t *>(a.status)) {
        } else if (!ORDERED) {
            const uint32_t n = screen_natural(a.scalars), sets = n == SC_ALL ? (uint32_t)a.blocks : n;
            const uint32_t splits = (uint32_t)screen_parts(a.scalars, a.splits, a.most_splits);
            if (t < sets * splits) {
                set = t % sets;
                part = t / sets;
                if (n != SC_ALL) set = a.nat_list[set];
                range = (uint32_t)a.n_slabs * part / splits | (uint32_t)a.n_slabs * (part + 1) / splits << 16;
            }
        } else {
            for (int c = 0; c < SC_PARTS; ++c) {          // the lists one after the other
                const uint32_t n = __ldcg(o.tickets + c);
                if (t < n) {
                    const uint2 item = o.items[(size_t)c * a.blocks + t];
                    set = item.x; range = item.y;
                    break;
                }
                t -= n;
            }
        }
        volatile uint32_t *d = item_slot + 4 * (to & 1);
        d[0] = set; d[1] = range; d[2] = part;
    };
    if (warp == NTW + 1 && lane == 0) decode(blockIdx.x, 0);
    block_sync();
    for (;; ++turn) {
        const uint32_t range = item_slot[4 * (turn & 1) + 1];
        const int s_lo = (int)(range & 0xffffu), slabs = (int)(range >> 16) - s_lo;
        if (item_slot[4 * (turn & 1)] == ~0u) break;
        mm_fence_before();
        block_sync();
        mm_fence_after();
        if (warp == NTW) {
            // ---------------- producer: the W stages of every slab, in order, through the ring
            if (lane == 0 && ok) {
                const unsigned char *src = a.head_img + (size_t)s_lo * KB * MMA_STAGE_BYTES;
                for (int n = 0; n < slabs && ok; ++n)
                    for (int kb = 0; kb < KB; kb += KS) {
                        if (!mm_wait(wempty0 + 8 * slot, phase, abort_flag, a.status, 1u)) { ok = false; break; }
                        const uint32_t bytes = (uint32_t)(min(KS, KB - kb) * (int)MMA_STAGE_BYTES);
                        mm_bar_expect_tx(wfull0 + 8 * slot, bytes);
                        mm_bulk_load(mm_smem(smem + (size_t)slot * KS * MMA_STAGE_BYTES), src, bytes, wfull0 + 8 * slot);
                        src += bytes;
                        ++issued;
                        if (++slot == NS) { slot = 0; phase ^= 1; }
                    }
            }
            __syncwarp();
        } else if (warp == NTW + 1) {
            // ---------------- one elected thread issues every MMA: 32-bit sums, unsigned bytes, 128 x 128
            const uint32_t idesc = (2u << 4) | (16u << 17) | (8u << 24);
            const uint32_t ring = mm_smem(smem);
            for (int n = done; n < done + slabs && ok; ++n) {
                const int buf = n & two;
                if (n > two)
                    ok = __all_sync(0xffffffffu, mm_wait(tempty0 + 8 * buf, ((n >> two) - 1) & 1, abort_flag, a.status, 2u));
                mm_fence_after();
                for (int kb = 0; kb < KB && ok; kb += KS) {
                    ok = __all_sync(0xffffffffu, mm_wait(wfull0 + 8 * slot, phase, abort_flag, a.status, 4u));
                    if (!ok) break;
                    const uint32_t stage = ring + slot * (uint32_t)(KS * MMA_STAGE_BYTES);
#pragma unroll
                    for (int x = 0; x < KS; ++x)
                        if (kb + x < KB) {
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                mm_mma_i8_ts(tmem + buf * 128, tmem + x_col + (kb + x) * 32 + u * 8,
                                             mm_desc(stage + x * (uint32_t)MMA_STAGE_BYTES + u * 256, 128, 1024),
                                             idesc, (kb | x | u) != 0);
                        }
                    mm_commit_warp(wempty0 + 8 * slot);
                    if (++slot == NS) { slot = 0; phase ^= 1; }
                }
                if (ok) mm_commit_warp(tfull0 + 8 * buf);
            }
            // The next item, now that the last slab is all that is left to gather (two slabs with two accumulators; not at
            // the item's beginning: whoever waits for a long one must not hold another).  By this warp, which has nothing
            // else to do: a tail warp that drew it waited for the counter in front of its last slab, and all others for the
            // item to be looked up (120,000 documents on 64 x 64, D = 4,096, 1,251 -> 1,223 us; 200,000 on a trained 128 x
            // 128 map, planned, 10.65 -> 10.60 ms).  As many tickets as items are taken, if any: then the counter is
            // zero again.
            if (lane == 0) {
                uint32_t t;
                if (ORDERED) {
                    t = atomicAdd(o.tickets + SC_PARTS, 1u);
                } else {
                    const uint32_t sets = screen_natural(a.scalars);
                    const uint32_t items = (sets == SC_ALL ? (uint32_t)a.blocks : sets) * (uint32_t)screen_parts(a.scalars, a.splits, a.most_splits);
                    t = items > gridDim.x ? atomicInc(a.ticket, items - 1u) : items;
                }
                decode(gridDim.x + t, turn + 1);
            }
        }
        __syncwarp();
        done += slabs;
        mm_fence_before();
        block_sync();
        mm_fence_after();
    }
    if (warp == NTW && lane == 0 && !ok) {
        // gave up: let the copies in flight land before leaving
        for (int c = issued > NS ? issued - NS : 0; c < issued; ++c)
            for (uint32_t spin = 0; spin < MMA_WAIT_LIMIT; ++spin)
                if (mm_bar_try(wfull0 + 8 * (c % NS), (c / NS) & 1)) break;
    }
    if (warp == NTW + 1) {
        mm_commit_warp(drain);
        for (uint32_t spin = 0; spin < MMA_WAIT_LIMIT; ++spin)
            if (mm_bar_try(drain, 0)) break;
    }
    __syncwarp();
    } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(SC_TAIL_REGS));
    const int q = warp & 3, e = warp >> 2;
    block_sync();
    for (;; ++turn) {
        const volatile uint32_t *item = item_slot + 4 * (turn & 1);
        if (item[0] == ~0u) break;
        const int group = (int)item[0];
        const int s_lo = (int)(item[1] & 0xffffu), s_hi = (int)(item[1] >> 16);
        const int shift = done - s_lo;                    // from a slab of the launch to its number among the block's
        {
            // X_head into tensor memory: lane 32q + l = document, a column = four features
            const int words = a.head / 32;
            const int64_t p = (int64_t)group * SC_DOCS + 32 * q + lane;
            const bool there = p < a.n_tiles * 8;
            for (int wd = e; wd < a.head_pad / 32; wd += 4) {
                const uint32_t m = there && wd < words ? __ldg(a.tile_head + (size_t)p * words + wd) : 0u;
                const uint4 k0 = reinterpret_cast<const uint4 *>(a.kpack)[2 * wd];
                const uint4 k1 = reinterpret_cast<const uint4 *>(a.kpack)[2 * wd + 1];
                const uint32_t k[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
                uint32_t v[8];
#pragma unroll
                for (int c = 0; c < 8; ++c)          // four mask bits -> four byte masks
                    v[c] = ((((m >> (4 * c)) & 15u) * 0x00204081u) & 0x01010101u) * 255u & k[c];
                mm_tmem_st8(tmem + ((uint32_t)(q * 32) << 16) + x_col + wd * 8, v);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        }
        mm_fence_before();
        block_sync();
        mm_fence_after();
        // ---------------- tail: documents 32q + 8e .. + 7 of a block, one tile
        const int s = lane >> 3, hb = (lane >> 2) & 1, li = lane & 3;
        const uint32_t sel_own = hb ? 0x4432u : 0x4410u, sel_other = hb ? 0x4410u : 0x4432u;
        const u64 sh = sc_pack(a.scalars[0], a.scalars[0]), st = sc_pack(a.scalars[1], a.scalars[1]);
        const u64 minus_2p23 = sc_pack(-8388608.f, -8388608.f);
        const size_t slab_bytes = (size_t)(a.D + 1) * SC_SLAB;
        const int tile = group * (SC_DOCS / 8) + 4 * q + e;
        uint32_t quads = 0;                                              // groups of four rows
        const uint4 *ids = a.tile_ids;
        [[maybe_unused]] size_t room = a.tile_rows_cap;
        if (tile < a.n_tiles) {
            const uint32_t rows = min(__ldg(a.tile_len + tile) & 0xffffu, (uint32_t)a.scalars[6]);
            quads = (rows + 3) / 4;
            const uint32_t off = BMU_IDX(__ldg(a.tile_off + tile), a.tile_rows_cap, a.status);
            ids += off; room -= off;
        }
        ids += s;
        const uint32_t p = (uint32_t)tile * 8 + (lane >> 2);             // this lane's document
        const float win = a.window[p];
        float m1 = 3.0e38f, m2 = 3.0e38f;                                // smallest (and second) value of the document
        // ORDERED: how far it reaches (evaluated whole: not at all), and what bounds its smallest (second) value
        [[maybe_unused]] float reach = -CUDART_INF_F, known = 0.f;
        // otherwise the stripe's smallest value, and the mask: eight slabs a word, stored when full; what lies before
        // slab `valid` does not count
        [[maybe_unused]] float own = 3.0e38f;
        [[maybe_unused]] uint32_t mask = 0u;
        [[maybe_unused]] int valid = s_lo;
        auto stripe = [&]() { return ((size_t)item[2] * a.n_pad + p) * 4 + li; };
        if constexpr (ORDERED) {
            const float2 r = o.reach[p];
            if (r.x <= a.scalars[SC_DOC_TOP]) reach = r.y;
            known = ordered_to_float(__ldcg(o.bound + p));
            if (TOP2) m2 = known; else m1 = known;
        } else if (!a.first) {
            m1 = a.amin[p];
            if (TOP2) m2 = a.amin2[p];
        }
        const unsigned char *base = a.img8 + (size_t)s_lo * slab_bytes + (lane & 7) * 16;
        const float *np = a.normp + (size_t)s_lo * SC_SLAB + li * 4;

        uint4 w[8], ix = make_uint4(0u, 0u, 0u, 0u);
        auto quad = [&](uint32_t h) { return __ldg(ids + BMU_IDX(4 * h, room - s, a.status)); };
        auto load = [&](const unsigned char *from, uint4 *d, uint32_t x0, uint32_t x1) {
            auto piece = [&](uint32_t word, uint32_t sel) {
                const uint32_t f = __byte_perm(word, 0, sel);
                return *reinterpret_cast<const uint4 *>(from + (size_t)(BMU_IDX(f, a.D + 1, a.status) * (uint32_t)SC_SLAB));
            };
            d[0] = piece(x0, sel_own);   d[1] = piece(x1, sel_own);
            d[2] = piece(x0, sel_other); d[3] = piece(x1, sel_other);
        };
        auto begin = [&]() {                                             // the first quad of the slab at `base`
            const uint4 i0 = quad(0);
            ix = quad(quads > 1 ? 1 : 0);
            load(base, w, i0.x, i0.y);
            load(base, w + 4, i0.z, i0.w);
        };
        // ORDERED: whether the head alone is looked at first, and whether a slab's first quad is on its way
        [[maybe_unused]] bool head_first = ORDERED && o.slab0 + s_lo > 0, begun = !head_first;
        [[maybe_unused]] const u64 tail_most = sc_pack((float)(4u * quads) * a.scalars[4], (float)(4u * quads) * a.scalars[4]);
        if (quads && begun) begin();
        for (int sl = s_lo; sl < s_hi; ++sl, np += SC_SLAB) {
            const int n = sl + shift;
            // no document of the tile reaches this slab, nor any behind it: the accumulators still change hands
            if (ORDERED && !__any_sync(0xffffffffu, o.unit_norm[sl * SC_SLAB] <= (TOP2 ? m2 : m1) + win + reach)) {
                for (int r = n; r < shift + s_hi; ++r) {
                    mm_wait(tfull0 + 8 * (r & two), (r >> two) & 1, abort_flag, a.status, 8u);
                    __syncwarp();
                    if (lane == 0) mm_bar_arrive(tempty0 + 8 * (r & two));
                }
                break;
            }
            const uint32_t taddr = tmem + ((uint32_t)(q * 32 + (e >> 1) * 16) << 16) + (uint32_t)((n & two) * 128);
            // integer head sums of eight neurons of the lane's 32 (the load covers two tiles of documents), and their norms
            [[maybe_unused]] auto head8 = [&](int c, uint32_t hs[8], u64 nm[4]) {
                uint32_t v[16];
                mm_tmem_ld_16x256b_x4(taddr + c * 32, v);
                const ulonglong2 n0 = *reinterpret_cast<const ulonglong2 *>(np + (2 * c) * 16);
                const ulonglong2 n1 = *reinterpret_cast<const ulonglong2 *>(np + (2 * c + 1) * 16);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    hs[2 * k] = (e & 1) ? v[4 * k + 2] : v[4 * k];
                    hs[2 * k + 1] = (e & 1) ? v[4 * k + 3] : v[4 * k + 1];
                }
                nm[0] = n0.x; nm[1] = n0.y; nm[2] = n1.x; nm[3] = n1.y;
            };
            if constexpr (ORDERED) {
                if (head_first) {
                    // what the gathered rows can add at most: if that rules the slab out, they are not gathered
                    mm_wait(tfull0 + 8 * (n & two), (n >> two) & 1, abort_flag, a.status, 8u);
                    mm_fence_after();
                    float least = CUDART_INF_F;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint32_t hs[8];
                        u64 nm[4];
                        head8(c, hs, nm);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const u64 x = sc_fma2(sc_pack(__uint2float_rn(hs[2 * k]), __uint2float_rn(hs[2 * k + 1])), sh, nm[k]);
                            least = fminf(least, fminf(lo_f(x), hi_f(x)));
                        }
                    }
                    // (the same operation as sc_dist2's last, with the largest sum there can be: never above what that gives)
                    least = lo_f(sc_fma2(tail_most, st, sc_pack(least, least)));
                    if (!__any_sync(0xffffffffu, least <= (TOP2 ? m2 : m1) + win)) {
                        mm_fence_before();
                        __syncwarp();
                        if (lane == 0) mm_bar_arrive(tempty0 + 8 * (n & two));
                        begun = false;
                        continue;
                    }
                }
                if (!begun) {
                    base = a.img8 + (size_t)sl * slab_bytes + (lane & 7) * 16;
                    if (quads) begin();
                    begun = true;
                }
            }
            uint32_t acc[2][8];                       // own, other document
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int x = 0; x < 8; ++x) acc[t][x] = 0u;
            for (uint32_t h = 0; h < quads; ++h) {
                if (h + 1 == quads && sl + 1 < s_hi) base += slab_bytes;
                sc_add(acc[0], w[0], w[1]);
                sc_add(acc[1], w[2], w[3]);
                load(base, w, ix.x, ix.y);
                sc_add(acc[0], w[4], w[5]);
                sc_add(acc[1], w[6], w[7]);
                load(base, w + 4, ix.z, ix.w);
                ix = quad(h + 2 < quads ? h + 2 : quads > 1 ? h + 2 - quads : 0);
            }
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int x = 0; x < 4; ++x) acc[t][x] = sc_even(acc[t][x], acc[t][4 + x]);
            // swap halves with the lane that holds the other sixteen neurons of this document
            uint32_t lo[8], hi[8];                    // neurons 32i .. + 15 and 32i + 16 .. + 31
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const uint32_t got = __shfl_xor_sync(0xffffffffu, acc[1][x], 4);
                lo[x] = hb ? got : acc[0][x];
                hi[x] = hb ? acc[0][x] : got;
            }
            mm_wait(tfull0 + 8 * (n & two), (n >> two) & 1, abort_flag, a.status, 8u);
            mm_fence_after();
            [[maybe_unused]] auto dist8 = [&](int c, u64 x[4]) {
                uint32_t hs[8];
                u64 nm[4];
                head8(c, hs, nm);
                const uint32_t *t = c < 2 ? lo : hi;
                const int w0 = 2 * (c & 1);
                x[0] = sc_dist2(nm[0], hs[0], hs[1], t[w0], sh, st, minus_2p23);
                x[1] = sc_dist2(nm[1], hs[2], hs[3], t[4 + w0], sh, st, minus_2p23);
                x[2] = sc_dist2(nm[2], hs[4], hs[5], t[w0 + 1], sh, st, minus_2p23);
                x[3] = sc_dist2(nm[3], hs[6], hs[7], t[5 + w0], sh, st, minus_2p23);
            };
            // (twice the same eight neurons at a time, on purpose: by dist8 the map's order, which frees the accumulator in
            // front of the last eight's arithmetic, took 2-8 % more)
            float mc[4];
            if constexpr (ORDERED) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    u64 x[4];
                    dist8(c, x);
                    mc[c] = fminf(fminf(fminf(lo_f(x[0]), hi_f(x[0])), fminf(lo_f(x[1]), hi_f(x[1]))),
                                  fminf(fminf(lo_f(x[2]), hi_f(x[2])), fminf(lo_f(x[3]), hi_f(x[3]))));
                }
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c) {             // eight neurons of the lane's 32 at a time
                    uint32_t v[16];
                    mm_tmem_ld_16x256b_x4(taddr + c * 32, v);
                    const ulonglong2 n0 = *reinterpret_cast<const ulonglong2 *>(np + (2 * c) * 16);
                    const ulonglong2 n1 = *reinterpret_cast<const ulonglong2 *>(np + (2 * c + 1) * 16);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (c == 3) {                         // the accumulator is free
                        mm_fence_before();
                        __syncwarp();
                        if (lane == 0) mm_bar_arrive(tempty0 + 8 * (n & two));
                    }
                    uint32_t hs[8];                       // (the load covers two tiles of documents)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        hs[2 * k] = (e & 1) ? v[4 * k + 2] : v[4 * k];
                        hs[2 * k + 1] = (e & 1) ? v[4 * k + 3] : v[4 * k + 1];
                    }
                    const uint32_t *t = c < 2 ? lo : hi;
                    const int w0 = 2 * (c & 1);
                    const u64 x0 = sc_dist2(n0.x, hs[0], hs[1], t[w0], sh, st, minus_2p23);
                    const u64 x1 = sc_dist2(n0.y, hs[2], hs[3], t[4 + w0], sh, st, minus_2p23);
                    const u64 x2 = sc_dist2(n1.x, hs[4], hs[5], t[w0 + 1], sh, st, minus_2p23);
                    const u64 x3 = sc_dist2(n1.y, hs[6], hs[7], t[5 + w0], sh, st, minus_2p23);
                    mc[c] = fminf(fminf(fminf(lo_f(x0), hi_f(x0)), fminf(lo_f(x1), hi_f(x1))),
                                  fminf(fminf(lo_f(x2), hi_f(x2)), fminf(lo_f(x3), hi_f(x3))));
                }
            }
            // the document's smallest (and second smallest) value over its four lanes
            const float m = fminf(fminf(mc[0], mc[1]), fminf(mc[2], mc[3]));
            if (!ORDERED) own = fminf(own, m);
            float g1 = m, g2 = CUDART_INF_F;
#pragma unroll
            for (int x = 1; x < 4; x <<= 1) {
                const float o1 = __shfl_xor_sync(0xffffffffu, g1, x);
                if (TOP2) {
                    const float o2 = __shfl_xor_sync(0xffffffffu, g2, x);
                    g2 = fminf(fminf(g2, o2), fmaxf(g1, o1));
                }
                g1 = fminf(g1, o1);
            }
            [[maybe_unused]] const float before = m1;
            if (TOP2) m2 = fminf(fminf(m2, g2), fmaxf(m1, g1));
            m1 = fminf(m1, g1);
            const float limit = (TOP2 ? m2 : m1) + win;
            if constexpr (!ORDERED) {
                if (before > limit) { mask = 0u; valid = sl; own = m; }      // nothing before this slab can win
                if (m <= limit)
                    mask |= ((mc[0] <= limit ? 1u : 0u) | (mc[1] <= limit ? 2u : 0u) | (mc[2] <= limit ? 4u : 0u) |
                             (mc[3] <= limit ? 8u : 0u)) << (4 * (sl & 7));
                if ((sl & 7) == 7 || sl + 1 == s_hi) {
                    reinterpret_cast<uint32_t *>(a.cmask + stripe())[sl >> 3] = mask;
                    mask = 0u;
                }
                continue;
            }
            // some unit of the warp's is within a window: which ones, from the sums once more
            head_first = !__any_sync(0xffffffffu, m <= limit);
            if (!head_first) {
                uint32_t bits = 0u;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    u64 x[4];
                    dist8(c, x);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        bits |= ((lo_f(x[i]) <= limit ? 1u : 0u) | (hi_f(x[i]) <= limit ? 2u : 0u)) << (8 * c + 2 * i);
                }
                if (bits) {
                    const uint32_t n_at = atomicAdd(o.count + p, 1u);
                    if (n_at < (uint32_t)SC_OWN_LIST)
                        reinterpret_cast<uint4 *>(o.lists + (size_t)p * SC_LIST_BYTES)[n_at] = make_uint4(__float_as_uint(m), (uint32_t)(o.slab0 + sl), bits, (uint32_t)li);
                }
            }
            mm_fence_before();                        // the accumulator is free
            __syncwarp();
            if (lane == 0) mm_bar_arrive(tempty0 + 8 * (n & two));
        }
        if constexpr (ORDERED) {
            const float found = TOP2 ? m2 : m1;
            if (li == 0 && found < known) atomicMin(o.bound + p, float_to_ordered(found));
        } else {
            a.cval[stripe()] = make_float2(own, __int_as_float(valid | (s_hi << 8)));
            if (TOP2) a.cval2[stripe()] = m2;
        }
        done = shift + s_hi;
        mm_fence_before();
        block_sync();
        mm_fence_after();
    }
    }
    mm_fence_before();
    __syncthreads();
    mm_fence_after();
    if (warp == NTW)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

int64_t screen_split_blocks(int64_t blocks, int64_t n_slabs, int sms)
{
    // what screen_splits takes beyond one block per set, at most (where it takes two: up to about
    // 3/4 n_slabs * sms sets)
    const int64_t most = (n_slabs < 16 ? n_slabs : 16) - 1, extra = 3 * (n_slabs + 4) * sms / 4;
    return blocks + (most * blocks < extra ? most * blocks : extra);
}

// How many blocks share a launch's slabs for one set of documents, in units of a slab's time.  Each
// block costs about half a slab to set up.  A few blocks per SM run in waves; with many, the longest
// lists first and all blocks of a split in front of the next, the scheduler evens them out but for about
// one block's time at the end.  (Stretches of equal estimated cost per SM leave less idle, but their
// blocks stand at different slabs and the whole image competes for L2 instead of a few slabs: 59.7 ms
// with four stretches per SM and 64.8 with one, against 56.9, on 512 x 512.)
int screen_splits(int64_t blocks, int64_t n_slabs, int sms)
{
    const int64_t room = screen_split_blocks(blocks, n_slabs, sms);
    int best = 1;
    double least = 1e300;
    for (int sp = 1; sp <= 16 && sp <= n_slabs && blocks * sp <= room; ++sp) {
        const int64_t waves = (blocks * sp + sms - 1) / sms;
        const double t = waves <= 4 ? (double)waves * ((double)((n_slabs + sp - 1) / sp) + 0.5)
                                    : (double)blocks * ((double)n_slabs + 0.5 * sp) / sms + (double)n_slabs / sp;
        if (t < least * 0.995) { least = t; best = sp; }
    }
    return best;
}

template <bool TOP2, bool ORDERED>
static int launch_sweep(const ScreenArgs &a, const OrderedArgs &o, int sms, cudaStream_t s)
{
    static bool configured[64];
    int dev = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && !configured[dev]) {
        // refuse a build whose launch registers do not cover the hand-over inside the kernel
        cudaFuncAttributes f;
        BMU_CUDA(cudaFuncGetAttributes(&f, sweep_screen_kernel<TOP2, ORDERED>));
        if (SC_THREADS * f.numRegs < 128 * SC_CTRL_REGS + 32 * SC_TAIL_WARPS * SC_TAIL_REGS) {
            set_error("screening sweep: built with %d registers per thread, too few for the hand-over", f.numRegs);
            return BMU_ERR_UNSUPPORTED;
        }
        BMU_CUDA(cudaFuncSetAttribute(sweep_screen_kernel<TOP2, ORDERED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SC_SMEM));
        configured[dev] = true;
    }
    const int64_t items = (int64_t)a.blocks * (ORDERED ? SC_PARTS : a.most_splits);
    ScreenLaunch l((unsigned)(items < sms ? items : sms), SC_THREADS, s, true, SC_SMEM);
    BMU_CUDA(cudaLaunchKernelEx(&l.c, sweep_screen_kernel<TOP2, ORDERED>, a, o));
    BMU_LAUNCHED();
    return BMU_OK;
}

int launch_sweep_screen(const ScreenArgs &a, const OrderedArgs &o, bool top2, bool ordered, int sms, cudaStream_t s)
{
    if (a.n_slabs <= 0 || a.blocks <= 0) return BMU_OK;
    if (a.n_slabs > SC_MAX_SLABS || a.head_pad > SC_MAX_HEAD) {
        set_error("screening sweep: at most %d slabs per launch and %d head rows", SC_MAX_SLABS, SC_MAX_HEAD);
        return BMU_ERR_INVALID_ARG;
    }
    if (ordered) return top2 ? launch_sweep<true, true>(a, o, sms, s) : launch_sweep<false, true>(a, o, sms, s);
    return top2 ? launch_sweep<true, false>(a, o, sms, s) : launch_sweep<false, false>(a, o, sms, s);
}

}  // namespace bmu
