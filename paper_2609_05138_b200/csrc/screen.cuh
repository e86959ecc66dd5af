// Screen and verify: the search of large sweeps in two stages that give the results of one.
//
//   screen   every (document, neuron) pair gets an APPROXIMATE distance from an 8-bit
//            fixed-point image of the codebook -- a quarter of the fp32 bytes, summed exactly
//            in integers -- together with a rigorous per-document bound on how far an
//            approximate distance can be from the distance the verify stage computes.  What
//            leaves the stage is, per document, the set of 8-neuron groups that hold a neuron
//            within twice that bound of the smallest approximate distance.  Every neuron that
//            could be the best (or second-best) unit is in one of these groups.
//   verify   the groups are evaluated exactly as the gathered kernels do it: fp32 sums over
//            the fp32 (or widened fp16) weights of the caller's codebook, fp32 distances,
//            lowest index on ties.  Only these numbers are ever returned.  Documents that
//            keep too many groups, or none, are evaluated whole (screen_dense.cu).
//
// The bound (screen_table_kernel and screen_window_kernel in screen_prep.cu compute it).  A
// weight w of feature f is stored as q = round((w - c_f) / step_f), c_f the row's minimum, so
// |w - (c_f + step_f q)| <= e_f; the sum of c_f over a document is the same for every neuron
// and plays no part.  With E = sum of e_f over the document's ids, A = sum of the rows' largest
// |w|, n the finite norms and |x| ids, the approximate distance differs from the exact real value of
// n_j - 2 s_ij (minus that constant) by at most 2 E + rounding, and the verify stage's fp32
// value by at most 2^-23 |x| A + rounding; together B = 2 E + 2^-23 (|x| A + 4 max|n| + 8 A).
// If j* wins the exact comparison then, for every j, approx(j*) <= approx(j) + 2 B: a neuron
// further than 2 B above the smallest approximate distance cannot win, whatever the weights.
//
// Units by norm (screen_order.cu).  Relative to the same constant no unit comes below n_j - 2 R, R = sum of
// (largest - smallest weight) over the rows of the document's ids, and some unit with a small norm gives an upper
// bound of the document's smallest value before anything has been summed.  So a unit whose norm lies more than
// 2 R + 2 B above what is still within the window cannot be in it.  Where the norms of the units spread further
// than that -- a codebook as it is first filled: 16,384 iid U[0,1) weights have norms of 5461 +- 38, a document of 80
// ids a 2 R of 160, of which the winner's own sum uses up half -- the slabs are made of units in the order of
// their norms, every document stops at the first slab beyond its reach, and most of the map is never summed (all
// but 12 % on 64 x 64, all but 4 % on 128 x 128).  Otherwise the slabs follow the map.  Both may be swept, one for
// the sets of 128 documents that reach a little, the other for those that reach far.
#pragma once

#include "common.cuh"

namespace bmu {

static const int SC_SLAB = 128;          // neurons per slab (one MMA tile, one 128-byte row piece)
static const int SC_GROUP = 8;           // neurons per group: what the verify stage evaluates at once
static const int SC_DOCS = 128;          // documents per block
static const int SC_MAX_HEAD = 1536;     // X_head in tensor memory: one column per four features
static const int SC_MAX_SLABS = 32;      // per launch: four bits each in a stripe's group mask
static const int SC_K_MAX = 32;          // largest integer row scale of a head feature
// -2 d_head, -2 d_tail, 1 / d_tail, whether the codes are an earlier search's, q_max, max |norm|, 65535 / q_max (the longest list that is
// screened), whether the images have to be made, largest range of the head rows and of the others
// ... and, as integers, how many of the sampled documents are to be evaluated whole, and how many were sampled;
// whether slabs are swept in the order of the norms, how many of them have an image, up to which norm units are in
// order, and how far a set of documents may reach to be swept so; the two units whose distances bound a document's
// smallest value (the smallest norms at even and at odd indices); whether the images of the slabs in that order
// stand from an earlier search, and how many units are in order; the two units' norms; how many sets of documents
// are swept in the order of the map (SC_ALL: each of them), and whether the images in that order are or will be made;
// how far a document may reach not to be evaluated whole
static const int SC_VOTES = 10, SC_SAMPLED = 11, SC_ORDERED = 12, SC_NEEDED = 13, SC_SORTED = 14, SC_TOP = 15,
                 SC_REF = 16, SC_STAND = 18, SC_KEPT = 19, SC_REFN = 20, SC_NAT = 22, SC_NATMADE = 23, SC_DOC_TOP = 24, SC_SAMPLE = 16,
                 SC_SCALARS = 32;
static const uint32_t SC_ALL = ~0u;
// Below this many units slabs always follow the map: too few for an order to spare many
static const int64_t SC_ORDER_MIN = 1024;
// Candidates wait in a list per document until every unit has been screened: a launch's local
// minimum says little before the document's own region of the map has been seen.
static const int SC_LIST = 12;           // entries: smallest value, group mask, first group
// ... where slabs are in the order of the norms, in the same room: smallest value, slab, which of the 32 units of a
// lane, the lane
static const int SC_OWN_LIST = 16;
static const size_t SC_LIST_BYTES = (size_t)SC_LIST * 24;                 // masks, values, groups
static_assert(SC_OWN_LIST * 16 <= SC_LIST * 24 && SC_LIST * 24 % 16 == 0, "one list per document");
// A block of that sweep takes up to this many slabs of a launch for a set of documents; sets and parts wait in lists
static const int SC_PART = 8, SC_PARTS = SC_MAX_SLABS / SC_PART;
// Documents and units are counted by how far they reach, in this many steps
static const int SC_BINS = 4096;
static const int SC_MAX_LAUNCHES = 1024;                     // ... with slabs in the order of the norms
static const uint32_t SC_DENSE = 1u << 30;           // in a document's count: to be evaluated whole

// Device arrays of one search: offsets into the workspace, relative to its screen part.
struct ScreenLayout {
    size_t scalars, rmin, rmax, table, kpack, khead, sample, window, amin, amin2;
    size_t cval, cval2, cmask, lcount, lists, img8, head_img, normp, total;
    // of slabs in the order of the norms
    size_t units, unit_norm, unit_tmp, rank_of, picks, ord8, ord_head, ord_normp, reach, items, tickets, nat_list;
    int64_t ord_launches;                // how many launches may sweep them
    int64_t n_pad;                       // documents rounded up to whole blocks
    int head_pad;                        // head rows rounded up to a stage (128)
    int64_t chunk_slabs;                 // slabs of the largest launch
    int splits, most_splits;             // blocks that share a launch's slabs for a set of documents; room for so many
    size_t rank, feat, map_total;        // only in a ScreenShared; without the images in the order of the norms
};

// What the searches of one call share that read the same codebook: the head they agree on, the row
// ranges and the images of all slabs.  Each search checks on the device that the images resolve its own
// longest list and makes them anew if not.
struct ScreenShared {
    char *base;
    ScreenLayout lay;                    // codebook arrays, two sets of scalars, a slab slot per launch and slab
    int used;                            // searches so far
};

struct ScreenArgs {
    const unsigned char *img8;           // [slab][D + 1][128]: row D is zero
    const unsigned char *head_img;       // [slab][head_pad / 128][16 KB]
    const float *normp;                  // [slab][128], in the order the lanes read it
    const uint32_t *kpack;               // head_pad / 4 words: four row scales each
    const float *scalars;
    const float *window;                 // 2 B per planned document
    const uint32_t *tile_len, *tile_off;
    const uint4 *tile_ids;               // quad layout: four rows of a tile, two documents a word
    const uint32_t *tile_head;           // head / 32 mask words per planned document
    const float *amin, *amin2;           // smallest (second) value of the earlier launches
    float2 *cval;                        // [split][n_pad][4]: a stripe's (the neurons one lane carries)
                                         // smallest value, and the first slab its mask counts from
    float *cval2;                        // second smallest value of the document
    uint4 *cmask;                        // the stripe's 8-neuron groups within the window: bit 4 s + c
    uint32_t *status, *ticket;           // of the next item, zero
    const uint32_t *nat_list;            // sets of documents, if not all
    int64_t D, n_tiles, n_pad;
    size_t tile_rows_cap;
    int32_t head, head_pad, n_slabs, splits, most_splits, blocks, first;
};

// The same search with slabs in the order of the norms
struct OrderedArgs {
    const float2 *reach;                 // per planned document: the largest norm it may need, and 2 R + 2 B
    uint32_t *bound;                     // of its smallest (second smallest) value, as float_to_ordered
    const float *unit_norm;              // norms in ascending order, from the launch's first slab on
    const uint2 *items;                  // [SC_PARTS][blocks]: set of documents, first slab | last << 16
    uint32_t *tickets;                   // SC_PARTS lengths of these lists, and the next to be taken
    char *lists;                         // a document's SC_OWN_LIST entries, SC_LIST_BYTES apart
    uint32_t *count;
    int64_t slab0;                       // the launch's first slab in that order
};

struct VerifyArgs {
    const void *W;
    int64_t D, M, N, n_pad;
    const float *norms;
    const int32_t *rowptr, *colidx, *perm;
    const float *window;
    const float2 *cval;
    const float *cval2;
    const uint4 *cmask;
    float *amin, *amin2;                 // smallest (second) approximate value so far
    uint32_t *lcount;                    // bits 0 .. 3: entries of the list; 4 .. 29: groups evaluated already;
                                         // 30: to be evaluated whole; 31: state[] holds exact keys
    char *lists;
    const uint32_t *set_reach;           // how far each set of documents reaches, as float_to_ordered
    const float2 *reach;
    const uint32_t *bound;
    const int32_t *units;
    u64 *state, *state2;                 // exact keys of what did not fit a list
    uint32_t *dense, *dense_count;       // planned documents to be evaluated whole
    const float *scalars;
    int32_t *out_bmu, *out_bmu2;
    float *out_dist, *out_dist2;
    uint32_t *status;
    int64_t launch, launches;            // slab s of the launch is launch + s * launches of the map
    int32_t splits, most_splits, first, f16;
};

// In which order the fp32 weights of a unit are added wherever it is evaluated: N partial sums, the i-th over ids i,
// i + N, ... of the list, then i and i + N / 2 of them, and so on (rows that are not whole 16-byte pieces, VEC false:
// 0 and 1, 2 and 3, then those two).  As many as rows are loaded side by side in the verify stage.
template <typename WT, bool VEC> struct ScreenSums {
    static constexpr int N = !VEC ? 4 : sizeof(WT) == 4 ? 16 : 32;
};

#ifdef __CUDACC__
// Most of the sampled documents are better evaluated whole: nothing is screened, all documents are.
__device__ __forceinline__ bool screen_whole(const float *scalars)
{
    const uint32_t *s = reinterpret_cast<const uint32_t *>(scalars);
    return 2u * s[SC_VOTES] > s[SC_SAMPLED];
}
__device__ __forceinline__ bool screen_ordered(const float *scalars)         // some sets are
{
    return reinterpret_cast<const uint32_t *>(scalars)[SC_ORDERED] != 0u;
}
__device__ __forceinline__ uint32_t screen_natural(const float *scalars)      // how many sets are not
{
    return reinterpret_cast<const uint32_t *>(scalars)[SC_NAT];
}
// ... and how many parts a launch's slabs are cut into for each: more than `splits` where they are few
__device__ __forceinline__ int screen_parts(const float *scalars, int splits, int most)
{
    const uint32_t n = screen_natural(scalars);
    return n == SC_ALL || n == 0u ? splits : (int)min((uint32_t)most, max((uint32_t)splits, 512u / n));
}
__device__ __forceinline__ bool screen_by_norm(const float *scalars, const uint32_t *set_reach, int64_t p)
{
    return screen_ordered(scalars) && ordered_to_float(set_reach[p / SC_DOCS]) <= scalars[SC_TOP];
}
// Steps between the smallest norm and the largest
struct ScreenSteps {
    float lo, top, scale;
    __device__ __forceinline__ ScreenSteps(float least, float most) : lo(least), top(most)
    {
        scale = top > lo ? (float)SC_BINS / (top - lo) : 0.f;
    }
    __device__ __forceinline__ ScreenSteps(const float *scalars)
        : ScreenSteps(fminf(scalars[SC_REFN], scalars[SC_REFN + 1]), scalars[5]) {}
    __device__ __forceinline__ int of(float n) const { return max(0, min((int)((n - lo) * scale), SC_BINS - 1)); }
};
#endif

// Rows are whole 16-byte pieces
inline bool screen_vec(const VerifyArgs &a)
{
    return (reinterpret_cast<uintptr_t>(a.W) & 15) == 0 && a.M % (a.f16 ? 8 : 4) == 0;
}

// A document with more candidate groups than this, an eighth of the map, is evaluated whole: scattered
// 32-byte sectors bring an update at an eighth to a quarter of the rate of whole rows (all of a map of
// 4,096 units for 20,000 documents: 5.5 ms, 1.3).  Those that find no place in a list are evaluated before
// it is known how many there will be: a quarter of that.
__host__ __device__ __forceinline__ uint32_t screen_dense_groups(int64_t M)
{
    return M / 64 > 8 ? (uint32_t)(M / 64) : 8u;
}
__host__ __device__ __forceinline__ uint32_t screen_early_groups(int64_t M)
{
    return M / 256 > 8 ? (uint32_t)(M / 256) : 8u;
}

void screen_layout(int64_t D, int64_t M, int64_t N, int head, int64_t chunk, bool top2, int sms,
                   ScreenLayout *l);
void screen_shared_layout(int64_t D, int64_t M, int head, int64_t chunk, ScreenLayout *l);
// blocks that share a launch's slabs, and the most that `blocks` or fewer sets of documents take of them in
// all: a bound that grows with the blocks, unlike the splits, so that a workspace for many serves fewer
int screen_splits(int64_t blocks, int64_t n_slabs, int sms);
int64_t screen_split_blocks(int64_t blocks, int64_t n_slabs, int sms);
// row ranges, scales, errors and the per-document windows: once per search (key: a document's gathered
// ids, by its number in the corpus; the maxima behind `status` are zero).  codebook arrays at cb + cl;
// `earlier`: the scalars of an earlier search of the same codebook and head, whose ranges still stand
int launch_screen_prepare(const void *W, int f16, int64_t D, int64_t M, const float *norms,
                          const int32_t *rowptr, const int32_t *colidx, int64_t N, int head,
                          const uint16_t *feat, const uint16_t *rank, const int32_t *perm,
                          const uint32_t *key, const uint32_t *tile_len, char *cb, const ScreenLayout &cl,
                          float *scalars, const float *earlier, float *sample, float *window, float2 *reach,
                          uint32_t *bound, uint32_t *count, uint32_t *set_reach, int64_t n_pad, bool top2,
                          uint32_t *status, cudaStream_t s);
// whether that can be decided in favour of the order of the norms at all, or nothing of it is launched
bool screen_order_possible(int64_t D, int64_t M, int64_t N);
// which sets of documents are swept in the order of the norms, and the units in that order
int launch_screen_order(const float *norms, int64_t D, int64_t M, int64_t N, int64_t launches, char *cb,
                        const ScreenLayout &cl, float *scalars, const float *earlier, const uint32_t *status,
                        const uint32_t *set_reach, int sets, uint32_t *tickets, uint32_t *nat_list, cudaStream_t s);
// the 8-bit images and the norms of the n_slabs slabs of launch k (neurons beyond M: never chosen), into the slots
// from `slot` on; nothing if the scalars say that they stand, as may be `expected`
int launch_screen_quantize(const void *W, int f16, int64_t D, int64_t M, const float *norms,
                           int64_t k, int64_t launches, int64_t n_slabs, int64_t slot, int head,
                           const uint16_t *feat, char *cb, const ScreenLayout &cl, const float *scalars,
                           bool expected, cudaStream_t s);
// ... of slabs in the order of the norms, slab0 and the following, and the lists of the sweep's items
struct OrderedImages {
    int64_t slab0, slot;
    int n_slabs, head, sets, first;
    const uint32_t *set_reach, *bound;
    const float2 *reach;
    const float *window;
    uint2 *items;
    uint32_t *tickets;
};
int launch_screen_ordered_images(const void *W, int f16, int64_t D, int64_t M, const OrderedImages &g,
                                 const uint16_t *feat, char *cb, const ScreenLayout &cl, const float *scalars, int sms,
                                 cudaStream_t s);
// A launch that may begin under the end of the one before it on the stream, if that one's blocks allow it
// (griddepcontrol.launch_dependents).  Every kernel launched so waits for it first of all (griddepcontrol.wait), also
// where it has nothing to do: whoever waits for the end of one kernel has then waited for all before it.
// What a kernel of the chain reads from another of it, screen_range_kernel among them, it reads by ordinary loads: it
// may live before that has been written, and read-only loads (__ldg, const __restrict__) promise that nobody writes while
// it does.  The caller's arrays and those of the tiling pass are complete before the chain begins.
struct ScreenLaunch {
    cudaLaunchAttribute attr;
    cudaLaunchConfig_t c;
    ScreenLaunch(dim3 blocks, unsigned threads, cudaStream_t s, bool early, size_t smem = 0) : c()
    {
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        c.gridDim = blocks; c.blockDim = dim3(threads); c.dynamicSmemBytes = smem;
        c.stream = s; c.attrs = &attr; c.numAttrs = early ? 1 : 0;
    }
    ScreenLaunch(const ScreenLaunch &) = delete;
};
// one launch for either order of the slabs: the one that the scalars do not name returns at once
int launch_sweep_screen(const ScreenArgs &a, const OrderedArgs &o, bool top2, bool ordered, int sms, cudaStream_t s);
// after each launch: what it could not rule out, into the documents' lists
int launch_screen_collect(const VerifyArgs &a, bool top2, cudaStream_t s);
// after the last: the lists evaluated exactly, and the outputs
int launch_screen_verify(const VerifyArgs &a, bool top2, cudaStream_t s);
// the same for slabs in the order of the norms
int launch_screen_verify_units(const VerifyArgs &a, bool top2, int sms, cudaStream_t s);
// directly behind them: the documents they handed over (none, as a rule)
int launch_screen_dense(const VerifyArgs &a, bool top2, int sms, cudaStream_t s);

}  // namespace bmu
