// The document-tiling pass (Section 4.1 "tile size", Section 4.2 "tile
// membership"): turns the caller's CSR into the form the planned, tiled and
// tensor-core sweeps walk.  The pass
//   1. orders documents by length (longest first; by the length of the gathered
//      list when there is a dense head) so that the documents that share a warp,
//      a tile or a block carry similar numbers of features and finish together;
//   2. re-packs every row as ascending 16-bit feature ids in 16-byte groups
//      (8 ids), padded with the sentinel 0xFFFF and closed by one all-sentinel
//      group, so eight ids arrive with one aligned 128-bit load and a list
//      ends by itself;
//   3. (tiled and tensor-core sweeps) cuts the length-ordered documents into tiles
//      of 8 and writes, per tile, an id matrix: row b holds the b-th id of each of
//      the tile's 8 documents (0xFFFF where a document has run out), so one aligned
//      128-bit load hands a warp the next row of all eight documents.
// Integer work only; the order of documents never changes any result because
// every document is reduced on its own.
#include "common.cuh"

#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>

namespace bmu {

static const int PLAN_BINS = 65536;      // one bin per row length: documents end up exactly
                                         // length-ordered (ids are 16-bit, so rows are shorter)

// ---- frequency ranks of the features (Table 8: the paper relabels its vocabulary by
// frequency and keeps that as substrate; here the relabelling is internal to the plan, so the
// dense head is the `head` most frequent features whatever ids the caller uses) -------------
// Listings per feature for the ids in [lo, hi): counted in shared memory first (a frequent
// feature is listed by most documents, and that many atomics on one global counter crawl),
// then flushed.
__global__ void __launch_bounds__(1024)
plan_feat_hist_kernel(const int32_t *__restrict__ colidx, int64_t nnz, int32_t lo, int32_t hi,
                      uint32_t *__restrict__ count)
{
    extern __shared__ uint32_t bins[];
    const int n_bins = hi - lo;
    for (int b = threadIdx.x; b < n_bins; b += blockDim.x) bins[b] = 0u;
    __syncthreads();
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t f = __ldg(colidx + e);
        if (f >= lo && f < hi) atomicAdd(bins + (f - lo), 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < n_bins; b += blockDim.x)
        if (bins[b]) atomicAdd(count + lo + b, bins[b]);
}

__global__ void plan_iota_kernel(int32_t D, uint32_t *__restrict__ v)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < D) v[i] = (uint32_t)i;
}

// Is the vocabulary labelled by frequency already?  If the ids below `head` cover at least 98 %
// of the listings that the `head` most frequent features cover, the ids are kept as ranks (rows
// then stay ascending and need no re-sorting).  One block.
__global__ void __launch_bounds__(1024)
plan_rank_decide_kernel(const uint32_t *__restrict__ count, const uint32_t *__restrict__ count_sorted,
                        int32_t D, int32_t head, int force, uint32_t *__restrict__ keep_ids)
{
    __shared__ unsigned long long s_id[32], s_rk[32];
    unsigned long long by_id = 0, by_rank = 0;
    for (int i = threadIdx.x; i < head && i < D; i += 1024) {
        by_id += count[i];
        by_rank += count_sorted[i];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        by_id += __shfl_xor_sync(0xffffffffu, by_id, off);
        by_rank += __shfl_xor_sync(0xffffffffu, by_rank, off);
    }
    if ((threadIdx.x & 31) == 0) { s_id[threadIdx.x >> 5] = by_id; s_rk[threadIdx.x >> 5] = by_rank; }
    __syncthreads();
    if (threadIdx.x == 0) {
        by_id = by_rank = 0;
        for (int w = 0; w < 32; ++w) { by_id += s_id[w]; by_rank += s_rk[w]; }
        *keep_ids = (!force && by_id * 100ull >= by_rank * 98ull) ? 1u : 0u;
    }
}

// sorted[r] = the feature of rank r (most frequent first, ties by ascending id)
__global__ void plan_rank_tables_kernel(const uint32_t *__restrict__ sorted, int32_t D,
                                        const uint32_t *__restrict__ keep_ids,
                                        uint16_t *__restrict__ rank_of_feat,
                                        uint16_t *__restrict__ feat_of_rank)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= D) return;
    const uint32_t f = *keep_ids ? (uint32_t)r : sorted[r];
    feat_of_rank[r] = (uint16_t)f;
    rank_of_feat[f] = (uint16_t)r;
}

// Sorting key of a document: how many of its ids the gather will visit, i.e. the ids at or
// above `head` (all of them when head == 0) -- or the whole list if it repeats an id below
// `head`: such a list keeps multiset semantics by staying out of the dense head altogether
// (plan_tile_len_kernel below), so all of it is gathered.  The key must be the gathered length exactly:
// the room reserved for the tile id matrices counts on documents ordered by it.  With `ckeys`
// the same pass over the row also forms the 64-bit content key (plan_cluster_key_kernel below
// says what it holds).  One warp per document.
__device__ __forceinline__ void plan_min3(uint32_t &a, uint32_t &b, uint32_t &c, uint32_t v)
{
    if (v < a) { c = b; b = a; a = v; } else if (v < b) { c = b; b = v; } else if (v < c) { c = v; }
}

__global__ void __launch_bounds__(256)
plan_key_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                const uint16_t *__restrict__ rank, int64_t N, int32_t head,
                uint32_t *__restrict__ key, [[maybe_unused]] int64_t D,
                [[maybe_unused]] uint32_t *__restrict__ status, int mode,
                u64 *__restrict__ ckeys, uint32_t *__restrict__ cvals)
{
    __shared__ uint32_t seen[8][HEAD_ROWS_MAX / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= N) return;
    for (int w = lane; w < head / 32; w += 32) seen[warp][w] = 0u;
    __syncwarp();
    const int beg = rowptr[i], end = rowptr[i + 1];
    int cnt = 0, repeat = 0;
    uint32_t m1 = 0, m2 = 0;                             // largest and second largest rank
    uint32_t s1 = 0xffffu, s2 = 0xffffu, s3 = 0xffffu;   // three smallest ranks >= head
    for (int e = beg + lane; e < end; e += 32) {
        const int32_t r = rank ? (int32_t)rank[BMU_IDX((uint32_t)colidx[e], D, status)] : colidx[e];
        if (r >= head) {
            ++cnt;
        } else {
            const uint32_t bit = 1u << (r & 31);
            repeat |= (atomicOr(&seen[warp][r >> 5], bit) & bit) != 0u;
        }
        if (ckeys) {
            const uint32_t rr = min((uint32_t)r, 0xfffeu);
            if (rr > m1) { m2 = m1; m1 = rr; } else if (rr > m2) { m2 = rr; }
            if (r >= head) plan_min3(s1, s2, s3, rr);
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
    repeat = __any_sync(0xffffffffu, repeat);
    const uint32_t len = repeat ? (uint32_t)(end - beg) : (uint32_t)cnt;
    if (lane == 0) key[i] = len;
    if (ckeys) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const uint32_t o1 = __shfl_xor_sync(0xffffffffu, m1, off);
            const uint32_t o2 = __shfl_xor_sync(0xffffffffu, m2, off);
            const uint32_t hi = max(m1, o1), lo = min(m1, o1);
            m2 = max(lo, max(m2, o2));
            m1 = hi;
            const uint32_t t1 = __shfl_xor_sync(0xffffffffu, s1, off);
            const uint32_t t2 = __shfl_xor_sync(0xffffffffu, s2, off);
            const uint32_t t3 = __shfl_xor_sync(0xffffffffu, s3, off);
            plan_min3(s1, s2, s3, t1);
            plan_min3(s1, s2, s3, t2);
            plan_min3(s1, s2, s3, t3);
        }
        if (lane == 0) {
            const u64 top = (u64)(uint32_t)(PLAN_BINS - 1 - min(len, (uint32_t)(PLAN_BINS - 1))) << 48;
            ckeys[i] = mode == 4 ? top | ((u64)s1 << 32) | ((u64)s2 << 16) | (u64)s3
                                 : top | ((u64)m1 << 32) | ((u64)m2 << 16) | (u64)s1;
            cvals[i] = (uint32_t)i;
        }
    }
}

// Lengths below LOCAL_BINS are counted and placed block by block in shared memory first: a hundred
// thousand documents have some sixty lengths, and an atomic per document on sixty counters crawls
// (120,000 documents: 24 us each for the counting and the placing, 3.3 and 3.7 so).
static const int LOCAL_BINS = 1024, LOCAL_DOCS = 1024;

// histogram of the sorting keys, and the largest key (aux[0]) so that the scan below can
// leave out the bins no document falls into
__global__ void __launch_bounds__(256)
plan_hist_kernel(const int32_t *__restrict__ rowptr, const uint32_t *__restrict__ key, int64_t N,
                 uint32_t *__restrict__ hist, uint32_t *__restrict__ aux)
{
    __shared__ uint32_t bins[LOCAL_BINS];
    for (int b = threadIdx.x; b < LOCAL_BINS; b += 256) bins[b] = 0u;
    __syncthreads();
    int most = 0;
#pragma unroll
    for (int k = 0; k < LOCAL_DOCS / 256; ++k) {
        const int64_t i = (int64_t)blockIdx.x * LOCAL_DOCS + 256 * k + threadIdx.x;
        if (i >= N) break;
        const int len = min(key ? (int)key[i] : rowptr[i + 1] - rowptr[i], PLAN_BINS - 1);
        if (len < LOCAL_BINS) atomicAdd(bins + len, 1u);
        else atomicAdd(hist + (PLAN_BINS - 1 - len), 1u);         // longest rows first
        most = max(most, len);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < LOCAL_BINS; b += 256)
        if (bins[b]) atomicAdd(hist + (PLAN_BINS - 1 - b), bins[b]);
    most = __reduce_max_sync(0xffffffffu, most);
    if ((threadIdx.x & 31) == 0 && most > 0) atomicMax(aux, (uint32_t)most);
}

// Exclusive scan of the bin counters from the first bin that can hold a document (the one of
// the largest key, `most`) to the last, by the WARPS warps of a block: a warp owns a contiguous run
// of bins and walks it 32 bins at a time (coalesced loads, shuffle scan); first the runs'
// totals, then the scan proper with each run's offset.
template <int WARPS>
__device__ __forceinline__ void plan_scan_bins(const uint32_t *hist, uint32_t most, uint32_t *cursor)
{
    __shared__ uint32_t s_tot[WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lo = PLAN_BINS - 1 - (int)min(most, (uint32_t)(PLAN_BINS - 1));
    const int per = ((PLAN_BINS - lo + WARPS - 1) / WARPS + 31) / 32 * 32;      // bins per warp, whole steps
    const int beg = lo + warp * per, end = min(beg + per, PLAN_BINS);
    uint32_t tot = 0;
    for (int b = beg + lane; b < end; b += 32) tot += __ldcg(hist + b);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, off);
    if (lane == 0) s_tot[warp] = tot;
    __syncthreads();
    uint32_t run = 0;
    for (int w = 0; w < warp; ++w) run += s_tot[w];
    for (int b0 = beg; b0 < end; b0 += 32) {
        const int b = b0 + lane;
        const uint32_t h = b < end ? __ldcg(hist + b) : 0u;
        uint32_t inc = h;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += v;
        }
        if (b < end) cursor[b] = run + inc - h;
        run += __shfl_sync(0xffffffffu, inc, 31);
    }
}

__global__ void __launch_bounds__(1024)
plan_scan_bins_kernel(const uint32_t *__restrict__ hist, const uint32_t *__restrict__ aux,
                      uint32_t *__restrict__ cursor)
{
    plan_scan_bins<32>(hist, aux[0], cursor);
}

// a document's planned position, and the groups of 8 ids its row needs there (plus its closing
// sentinel group); ngroups[N] = 0 closes the array for the scan
__global__ void __launch_bounds__(256)
plan_scatter_kernel(const int32_t *__restrict__ rowptr, const uint32_t *__restrict__ key, int64_t N,
                    uint32_t *__restrict__ cursor, int32_t *__restrict__ perm,
                    uint32_t *__restrict__ ngroups)
{
    constexpr int K = LOCAL_DOCS / 256;
    __shared__ uint32_t bins[LOCAL_BINS];
    for (int b = threadIdx.x; b < LOCAL_BINS; b += 256) bins[b] = 0u;
    if (ngroups && blockIdx.x == 0 && threadIdx.x == 0) ngroups[N] = 0u;
    __syncthreads();
    int len[K], row[K];
    uint32_t at[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int64_t i = (int64_t)blockIdx.x * LOCAL_DOCS + 256 * k + threadIdx.x;
        len[k] = -1;
        if (i >= N) continue;
        row[k] = rowptr[i + 1] - rowptr[i];
        len[k] = min(key ? (int)key[i] : row[k], PLAN_BINS - 1);
        at[k] = len[k] < LOCAL_BINS ? atomicAdd(bins + len[k], 1u)
                                    : atomicAdd(cursor + (PLAN_BINS - 1 - len[k]), 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < LOCAL_BINS; b += 256)           // room for the block's documents of length b
        if (bins[b]) bins[b] = atomicAdd(cursor + (PLAN_BINS - 1 - b), bins[b]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (len[k] < 0) continue;
        const uint32_t p = at[k] + (len[k] < LOCAL_BINS ? bins[len[k]] : 0u);
        perm[p] = (int32_t)((int64_t)blockIdx.x * LOCAL_DOCS + 256 * k + threadIdx.x);
        if (ngroups) ngroups[p] = (uint32_t)((row[k] + 7) / 8 + 1);
    }
}

// Tile membership by content (Section 4.2: documents that share features are put in the same
// tile).  Sorting key of a document: its length key first -- tiles must stay exactly
// length-ordered -- then a few of its features, so that inside a run of equally long documents
// those with the same features lie next to each other.  Which features (ranks, or ids on a
// vocabulary labelled by frequency):
//   mode 3  the two rarest of the list, then the most frequent one at or above `head`;
//   mode 4  the three most frequent ones at or above `head` (the first three the gather visits).
// Either way the shared features sit at the same step of the lists of a tile (the front, or the
// back of equally long lists), so the loads of one step ask for the same row.  One warp per
// document.
__global__ void __launch_bounds__(256)
plan_cluster_key_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                        const uint16_t *__restrict__ rank, const uint32_t *__restrict__ len_key,
                        int64_t N, int32_t head, int mode, [[maybe_unused]] int64_t D,
                        [[maybe_unused]] uint32_t *status, u64 *__restrict__ keys,
                        uint32_t *__restrict__ vals)
{
    const int lane = threadIdx.x & 31;
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= N) return;
    const int beg = rowptr[i], end = rowptr[i + 1];
    uint32_t m1 = 0, m2 = 0;                         // largest and second largest rank
    uint32_t s1 = 0xffffu, s2 = 0xffffu, s3 = 0xffffu;   // three smallest ranks >= head
    for (int e = beg + lane; e < end; e += 32) {
        const uint32_t f = (uint32_t)colidx[e];
        const uint32_t r = rank ? (uint32_t)rank[BMU_IDX(f, D, status)] : min(f, 0xfffeu);
        if (r > m1) { m2 = m1; m1 = r; } else if (r > m2) { m2 = r; }
        if (r >= (uint32_t)head) plan_min3(s1, s2, s3, r);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const uint32_t o1 = __shfl_xor_sync(0xffffffffu, m1, off);
        const uint32_t o2 = __shfl_xor_sync(0xffffffffu, m2, off);
        const uint32_t hi = max(m1, o1), lo = min(m1, o1);
        m2 = max(lo, max(m2, o2));
        m1 = hi;
        const uint32_t t1 = __shfl_xor_sync(0xffffffffu, s1, off);
        const uint32_t t2 = __shfl_xor_sync(0xffffffffu, s2, off);
        const uint32_t t3 = __shfl_xor_sync(0xffffffffu, s3, off);
        plan_min3(s1, s2, s3, t1);
        plan_min3(s1, s2, s3, t2);
        plan_min3(s1, s2, s3, t3);
    }
    if (lane == 0) {
        const int len = min(len_key ? (int)len_key[i] : end - beg, PLAN_BINS - 1);
        const u64 top = (u64)(uint32_t)(PLAN_BINS - 1 - len) << 48;
        keys[i] = mode == 4 ? top | ((u64)s1 << 32) | ((u64)s2 << 16) | (u64)s3
                            : top | ((u64)m1 << 32) | ((u64)m2 << 16) | (u64)s1;
        vals[i] = (uint32_t)i;
    }
}

// groups of 8 ids the row at planned position p needs (plus its closing sentinel group)
__global__ void plan_groups_kernel(const int32_t *__restrict__ rowptr,
                                   const int32_t *__restrict__ perm, int64_t N,
                                   uint32_t *__restrict__ ngroups)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p == 0) ngroups[N] = 0u;
    if (p >= N) return;
    const int32_t i = perm[p];
    ngroups[p] = (uint32_t)((rowptr[i + 1] - rowptr[i] + 7) / 8 + 1);
}

__global__ void plan_identity_kernel(const int32_t *__restrict__ rowptr, int64_t N,
                                     int32_t *__restrict__ perm, uint32_t *__restrict__ ngroups)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) ngroups[N] = 0u;
    if (i >= N) return;
    perm[i] = (int32_t)i;
    ngroups[i] = (uint32_t)((rowptr[i + 1] - rowptr[i] + 7) / 8 + 1);
}

// Size checks of the pass (one thread): the scanned offsets must fit the room that was
// reserved for what they index.  A failure sets bit 64 of the status word; the kernels that
// would write through those offsets, and every sweep, then do nothing.
__global__ void plan_check_kernel(const uint32_t *__restrict__ last_off, uint64_t room,
                                  uint32_t *__restrict__ status)
{
    if ((uint64_t)*last_off > room) atomicOr(status, PLAN_STATUS_OVERFLOW);
}

// One warp per planned document: writes its ascending 16-bit id list.  Rows that
// are not already in non-decreasing order are ordered by counting, for each id, the ids that
// must precede it (quadratic in the row length, rows are short).
__global__ void __launch_bounds__(256)
plan_fill_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                 const uint16_t *__restrict__ rank, const int32_t *__restrict__ perm,
                 const uint32_t *__restrict__ doc_off, int64_t N, uint16_t *__restrict__ ids16,
                 uint32_t *__restrict__ status, [[maybe_unused]] int64_t D)
{
    if (*status & PLAN_STATUS_OVERFLOW) return;
    // with a rank table the list holds ranks (ascending: most frequent first), not ids
#define BMU_PLAN_ID(e) (rank ? (int32_t)rank[BMU_IDX((uint32_t)row[e], D, status)] : row[e])
    const int lane = threadIdx.x & 31;
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (p >= N) return;
    const int32_t i = perm[p];
    const int beg = rowptr[i], len = rowptr[i + 1] - beg;
    const int32_t *row = colidx + beg;
    uint16_t *dst = ids16 + ((size_t)doc_off[p] + 1) * 8;          // group 0 is the global sentinel
    const int padded = ((len + 7) / 8 + 1) * 8;

    bool sorted = true;
    for (int e = lane; e + 1 < len; e += 32) sorted &= BMU_PLAN_ID(e) <= BMU_PLAN_ID(e + 1);
    sorted = __all_sync(0xffffffffu, sorted);
    if (sorted) {
        for (int e = lane; e < padded; e += 32) dst[e] = e < len ? (uint16_t)BMU_PLAN_ID(e) : 0xFFFFu;
    } else {
        for (int e = lane; e < padded; e += 32)
            if (e >= len) dst[e] = 0xFFFFu;
        for (int e = lane; e < len; e += 32) {
            const int32_t f = BMU_PLAN_ID(e);
            int pos = 0;
            for (int k = 0; k < len; ++k) {
                const int32_t g = BMU_PLAN_ID(k);
                pos += (g < f) || (g == f && k < e);
            }
            dst[pos] = (uint16_t)f;
        }
    }
#undef BMU_PLAN_ID
    if (p == 0 && lane < 8) ids16[lane] = 0xFFFFu;                  // global sentinel group
    if (p == N - 1 && lane < 16) dst[padded + lane] = 0xFFFFu;      // two groups of slack at the end
}

// ---- tiles of 8 documents -------------------------------------------------
// The ids below `head` (a multiple of 32, at most HEAD_ROWS_MAX) at the front of a document's
// ascending list become a bit mask of head / 32 words, and the list the sweep walks starts
// behind them.  A list that repeats one of them keeps multiset semantics by opting out (mask
// 0, nothing skipped): its ids all stay in the list.
// per tile: longest and shortest list behind the head (max | min << 16), and the head masks
// (head / 32 words per document, document-major).  One block per tile, one warp per document:
// the lanes read the front of the document's ascending list 32 ids at a time and set the mask
// bits in shared memory; a list that repeats a head id opts out (mask 0, nothing skipped).
__global__ void __launch_bounds__(256)
plan_tile_len_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ perm,
                     const uint32_t *__restrict__ doc_off, const uint16_t *__restrict__ ids16,
                     int64_t N, int64_t n_tiles, uint32_t head, uint32_t *__restrict__ tile_rows,
                     uint32_t *__restrict__ tile_len, uint32_t *__restrict__ tile_head)
{
    __shared__ uint32_t s_mask[8][HEAD_ROWS_MAX / 32];
    __shared__ uint32_t s_left[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tile = blockIdx.x;
    const int64_t p = tile * 8 + warp;                                    // planned position
    const uint32_t words = head ? head / 32 : 1;
    for (uint32_t w = lane; w < words; w += 32) s_mask[warp][w] = 0u;
    __syncwarp();
    uint32_t len = 0, skip = 0;
    if (p < N) {
        const int32_t i = perm[p];
        len = (uint32_t)min(rowptr[i + 1] - rowptr[i], 65535);
        if (head) {
            const uint16_t *ids = ids16 + ((size_t)doc_off[p] + 1) * 8;
            bool repeat = false;
            for (uint32_t e0 = 0; e0 < len && e0 <= head; e0 += 32) {
                const uint32_t e = e0 + lane;
                const uint32_t f = (e < len && e <= head) ? ids[e] : 0xffffu;
                const bool in = f < head;
                if (in) {
                    const uint32_t bit = 1u << (f & 31u);
                    repeat |= (atomicOr(&s_mask[warp][f >> 5], bit) & bit) != 0u;
                }
                const uint32_t got = __ballot_sync(0xffffffffu, in);
                skip += (uint32_t)__popc(got);
                if (got != 0xffffffffu) break;                            // the list left the head
            }
            if (__any_sync(0xffffffffu, repeat)) {
                __syncwarp();
                for (uint32_t w = lane; w < words; w += 32) s_mask[warp][w] = 0u;
                skip = 0;
            }
        }
    }
    __syncwarp();
    {
        uint32_t *mask = tile_head + (size_t)p * words;
        for (uint32_t w = lane; w < words; w += 32) mask[w] = s_mask[warp][w];
    }
    if (lane == 0) s_left[warp] = len - skip;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t mx = 0, mn = 0xffffffffu;
        for (int t = 0; t < 8; ++t) { mx = max(mx, s_left[t]); mn = min(mn, s_left[t]); }
        tile_rows[tile] = mx;
        tile_len[tile] = mx | (mn << 16);
    }
}

// One warp per tile: row r of the matrix = the r-th id, in visiting order, of each of its
// 8 documents behind the head.  Visiting order: ascending, or (interleave) dealt alternately
// from the frequent and the rare half of the document's own list, so that at any moment a
// warp mixes loads that hit L1 with loads that go to L2.  The order depends on the document
// alone, never on its tile mates, so results do not depend on how tiles were cut.
__global__ void __launch_bounds__(256)
plan_tile_fill_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ perm,
                      const uint32_t *__restrict__ doc_off, const uint16_t *__restrict__ ids16,
                      const uint32_t *__restrict__ tile_len, const uint32_t *__restrict__ tile_off,
                      const uint32_t *__restrict__ tile_head, uint32_t head_words,
                      const uint16_t *__restrict__ feat_of_rank, int64_t N, int64_t n_tiles,
                      int interleave, uint4 *__restrict__ tile_ids,
                      uint32_t *__restrict__ status, [[maybe_unused]] int64_t D)
{
    if (*status & PLAN_STATUS_OVERFLOW) return;
    const int lane = threadIdx.x & 31;
    const int64_t tile = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (tile >= n_tiles) return;
    const uint32_t rows = tile_len[tile] & 0xffffu;
    const uint16_t *src[8];
    uint32_t len[8];
    for (int t = 0; t < 8; ++t) {
        const int64_t p = tile * 8 + t;
        len[t] = 0;
        src[t] = ids16;
        if (p < N) {
            const int32_t i = perm[p];
            uint32_t skip = 0;
            for (uint32_t w = 0; w < head_words; ++w)
                skip += (uint32_t)__popc(tile_head[(tile * 8 + t) * head_words + w]);
            len[t] = (uint32_t)min(rowptr[i + 1] - rowptr[i], 65535) - skip;
            src[t] = ids16 + ((size_t)doc_off[p] + 1) * 8 + skip;
        }
    }
    uint4 *dst = tile_ids + tile_off[tile];
    for (uint32_t r = lane; r < rows; r += 32) {
        uint32_t f[8];
        for (int t = 0; t < 8; ++t) {
            uint32_t e = r;
            if (interleave) e = (r & 1u) ? (len[t] + 1) / 2 + r / 2 : r / 2;
            f[t] = r < len[t] ? src[t][e] : 0xffffu;
            if (feat_of_rank && f[t] != 0xffffu)                              // rank -> row of W
                f[t] = feat_of_rank[BMU_IDX(f[t], D, status)];
        }
        dst[r] = make_uint4(f[0] | (f[1] << 16), f[2] | (f[3] << 16), f[4] | (f[5] << 16),
                            f[6] | (f[7] << 16));
    }
}

size_t plan_bytes(int64_t N, int64_t nnz, int head, int64_t D, int cluster, bool quads, PlanLayout *l)
{
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    size_t off = 0;
    PlanLayout t;
    t.perm_off = off; off = up(off + (size_t)N * 4);
    t.docoff_off = off; off = up(off + (size_t)(N + 1) * 4);
    t.ngroups_off = off; if (!quads) off = up(off + (size_t)(N + 1) * 4);
    t.bins_off = off; off = up(off + (size_t)PLAN_BINS * 4 * 2 + 256);   // counters, cursors, aux
    t.id_groups_cap = (size_t)nnz / 8 + 2 * (size_t)N + 4;
    t.ids_off = off; if (!quads) off = up(off + t.id_groups_cap * 16);
    size_t scan_tmp = 0;
    if (!quads)
        cub::DeviceScan::ExclusiveSum(nullptr, scan_tmp, (uint32_t *)nullptr, (uint32_t *)nullptr,
                                      (int)(N + 1));
    t.scan_off = off; t.scan_bytes = scan_tmp; off = up(off + scan_tmp);
    // tiles: with documents exactly length-ordered, the sum over tiles of the longest row
    // is at most nnz / 8 plus the spread of lengths (< 65536)
    const size_t n_tiles = ((size_t)N + 7) / 8;
    t.tilelen_off = off; off = up(off + (n_tiles + 1) * 4);
    t.tilerows_off = off; if (!quads) off = up(off + (n_tiles + 1) * 4);
    t.tileoff_off = off; off = up(off + (n_tiles + 1) * 4);
    t.tilehead_off = off; off = up(off + n_tiles * 8 * 4 * (size_t)(head > 32 ? head / 32 : 1));
    t.tile_rows_cap = (size_t)nnz / 8 + 65536 + 4 * n_tiles;     // (rounded up to whole groups of four)
    t.tileids_off = off; off = up(off + t.tile_rows_cap * 16);
    // frequency ranks of the features (dense head only): counts, sort buffers, the two tables
    t.rank_off = t.feat_off = t.fsort_off = t.fsort_tmp_off = off;
    t.fsort_tmp_bytes = 0;
    if (head > 0 && D > 0 && D <= 65535) {
        const size_t d4 = up((size_t)D * 4), d2 = up((size_t)D * 2);
        t.rank_off = off; off += d2;
        t.feat_off = off; off += d2;
        t.fsort_off = t.fsort_tmp_off = off;
        if (!quads) {
            off += 4 * d4;                           // counts, sorted counts, ids, sorted ids
            size_t tmp = 0;
            cub::DeviceRadixSort::SortPairsDescending(nullptr, tmp, (uint32_t *)nullptr, (uint32_t *)nullptr,
                                                      (uint32_t *)nullptr, (uint32_t *)nullptr, (int)D);
            t.fsort_tmp_off = off; t.fsort_tmp_bytes = tmp; off = up(off + tmp);
        }
    }
    // ordering by content: 64-bit keys and document numbers, in and out, and the sort's scratch
    t.cluster_off = t.cluster_tmp_off = off;
    t.cluster_tmp_bytes = 0;
    if (cluster >= 3 && N > 0) {
        t.cluster_off = off; off = up(off + (size_t)N * 8 * 2 + (size_t)N * 4);
        size_t tmp = 0;
        cub::DeviceRadixSort::SortPairs(nullptr, tmp, (u64 *)nullptr, (u64 *)nullptr,
                                        (uint32_t *)nullptr, (uint32_t *)nullptr, (int)N);
        t.cluster_tmp_off = off; t.cluster_tmp_bytes = tmp; off = up(off + tmp);
    }
    t.total = off;
    if (l) *l = t;
    return off;
}

static int launch_feat_hist(const int32_t *colidx, int64_t nnz, int64_t D, uint32_t *count, cudaStream_t s)
{
    if (nnz <= 0) return BMU_OK;
    const int32_t span = 32768;                           // 128 KB of shared-memory counters
    static bool configured[64];
    int dev = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && !configured[dev]) {
        BMU_CUDA(cudaFuncSetAttribute(plan_feat_hist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, span * 4));
        configured[dev] = true;
    }
    for (int32_t lo = 0; lo < (int32_t)D; lo += span) {
        const int32_t hi = lo + span < (int32_t)D ? lo + span : (int32_t)D;
        { plan_feat_hist_kernel<<<148, 1024, (size_t)(hi - lo) * 4, s>>>(colidx, nnz, lo, hi, count); BMU_LAUNCHED(); }
    }
    return BMU_OK;
}

int launch_plan(const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz,
                int order_by_length, int head, int relabel, int64_t D, char *ws, const PlanLayout &l,
                uint32_t *status, cudaStream_t s)
{
    // dense head: rank the features by how many documents list them, so that the head is the
    // `head` most frequent features whatever their ids
    const uint16_t *rank = nullptr;
    if (head > 0 && relabel != 2 && l.fsort_tmp_bytes > 0) {
        const size_t d4 = ((size_t)D * 4 + 255) / 256 * 256;
        uint32_t *count = reinterpret_cast<uint32_t *>(ws + l.fsort_off);
        uint32_t *count_sorted = reinterpret_cast<uint32_t *>(ws + l.fsort_off + d4);
        uint32_t *ids = reinterpret_cast<uint32_t *>(ws + l.fsort_off + 2 * d4);
        uint32_t *ids_sorted = reinterpret_cast<uint32_t *>(ws + l.fsort_off + 3 * d4);
        uint16_t *rank_of_feat = reinterpret_cast<uint16_t *>(ws + l.rank_off);
        uint16_t *feat_of_rank = reinterpret_cast<uint16_t *>(ws + l.feat_off);
        BMU_CUDA(cudaMemsetAsync(count, 0, (size_t)D * 4, s));
        const int rc = launch_feat_hist(colidx, nnz, D, count, s);
        if (rc) return rc;
        { plan_iota_kernel<<<(unsigned)((D + 255) / 256), 256, 0, s>>>((int32_t)D, ids); BMU_LAUNCHED(); }
        size_t tmp = l.fsort_tmp_bytes;
        BMU_CUDA(cub::DeviceRadixSort::SortPairsDescending(ws + l.fsort_tmp_off, tmp, count, count_sorted,
                                                           ids, ids_sorted, (int)D, 0, 32, s));
        // the decision word borrows the first counter of the length histogram (cleared below)
        uint32_t *keep_ids = reinterpret_cast<uint32_t *>(ws + l.bins_off);
        { plan_rank_decide_kernel<<<1, 1024, 0, s>>>(count, count_sorted, (int32_t)D, head, relabel == 1,
                                                   keep_ids); BMU_LAUNCHED(); }
        { plan_rank_tables_kernel<<<(unsigned)((D + 255) / 256), 256, 0, s>>>(ids_sorted, (int32_t)D,
                                                                            keep_ids, rank_of_feat,
                                                                            feat_of_rank); BMU_LAUNCHED(); }
        rank = rank_of_feat;
    }
    int32_t *perm = reinterpret_cast<int32_t *>(ws + l.perm_off);
    uint32_t *doc_off = reinterpret_cast<uint32_t *>(ws + l.docoff_off);
    uint32_t *ngroups = reinterpret_cast<uint32_t *>(ws + l.ngroups_off);
    uint32_t *hist = reinterpret_cast<uint32_t *>(ws + l.bins_off);
    uint32_t *cursor = hist + PLAN_BINS;
    uint32_t *aux = cursor + PLAN_BINS;              // [0] the largest sorting key
    uint16_t *ids16 = reinterpret_cast<uint16_t *>(ws + l.ids_off);
    const unsigned blocks = (unsigned)((N + 255) / 256);
    if (order_by_length) {
        // with a dense head the documents are ordered by what is left for the gather, so that
        // the documents of a tile finish their lists together (the key borrows the doc_off
        // array, which is written only by the scan after the scatter)
        const uint32_t *key = nullptr;
        const bool by_content = order_by_length >= 3 && l.cluster_tmp_bytes > 0;
        u64 *keys_in = reinterpret_cast<u64 *>(ws + l.cluster_off);
        u64 *keys_out = keys_in + N;
        uint32_t *vals_in = reinterpret_cast<uint32_t *>(keys_out + N);
        if (head > 0) {
            // length key and, if wanted, the content key in one pass over the rows
            { plan_key_kernel<<<(unsigned)((N * 32 + 255) / 256), 256, 0, s>>>(
                rowptr, colidx, rank, N, head, doc_off, D, status, order_by_length,
                by_content ? keys_in : nullptr, vals_in); BMU_LAUNCHED(); }
            key = doc_off;
        }
        // counters and the largest key in one clearing (the cursors in between are all written
        // or never read)
        BMU_CUDA(cudaMemsetAsync(hist, 0, (size_t)PLAN_BINS * 4 * 2 + 256, s));
        if (by_content) {
            // by length, then by the rarest features: one radix sort of (key, document) pairs
            if (head == 0)
                { plan_cluster_key_kernel<<<(unsigned)((N * 32 + 255) / 256), 256, 0, s>>>(
                    rowptr, colidx, rank, key, N, head, order_by_length, D, status, keys_in, vals_in); BMU_LAUNCHED(); }
            size_t ctmp = l.cluster_tmp_bytes;
            BMU_CUDA(cub::DeviceRadixSort::SortPairs(ws + l.cluster_tmp_off, ctmp, keys_in, keys_out,
                                                     vals_in, reinterpret_cast<uint32_t *>(perm),
                                                     (int)N, 0, 64, s));
            { plan_groups_kernel<<<blocks, 256, 0, s>>>(rowptr, perm, N, ngroups); BMU_LAUNCHED(); }
        } else {
            { plan_hist_kernel<<<(unsigned)((N + LOCAL_DOCS - 1) / LOCAL_DOCS), 256, 0, s>>>(rowptr, key, N, hist, aux); BMU_LAUNCHED(); }
            { plan_scan_bins_kernel<<<1, 1024, 0, s>>>(hist, aux, cursor); BMU_LAUNCHED(); }
            { plan_scatter_kernel<<<(unsigned)((N + LOCAL_DOCS - 1) / LOCAL_DOCS), 256, 0, s>>>(rowptr, key, N, cursor, perm, ngroups); BMU_LAUNCHED(); }
        }
    } else {
        { plan_identity_kernel<<<blocks, 256, 0, s>>>(rowptr, N, perm, ngroups); BMU_LAUNCHED(); }
    }
    size_t tmp = l.scan_bytes;
    BMU_CUDA(cub::DeviceScan::ExclusiveSum(ws + l.scan_off, tmp, ngroups, doc_off, (int)(N + 1), s));
    // group 0 is the global sentinel and two groups of slack close the lists
    { plan_check_kernel<<<1, 1, 0, s>>>(doc_off + N, (uint64_t)l.id_groups_cap - 3, status); BMU_LAUNCHED(); }
    { plan_fill_kernel<<<(unsigned)((N * 32 + 255) / 256), 256, 0, s>>>(rowptr, colidx, rank, perm,
                                                                       doc_off, N, ids16, status, D); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

int launch_plan_tiles(const int32_t *rowptr, int64_t N, int interleave, int head, int relabel,
                      int64_t D, char *ws, const PlanLayout &l, uint32_t *status, cudaStream_t s)
{
    const uint16_t *feat_of_rank = (head > 0 && relabel != 2 && l.fsort_tmp_bytes > 0)
                                       ? reinterpret_cast<const uint16_t *>(ws + l.feat_off) : nullptr;
    const int64_t n_tiles = (N + 7) / 8;
    const int32_t *perm = reinterpret_cast<const int32_t *>(ws + l.perm_off);
    const uint32_t *doc_off = reinterpret_cast<const uint32_t *>(ws + l.docoff_off);
    const uint16_t *ids16 = reinterpret_cast<const uint16_t *>(ws + l.ids_off);
    uint32_t *tile_len = reinterpret_cast<uint32_t *>(ws + l.tilelen_off);
    uint32_t *tile_rows = reinterpret_cast<uint32_t *>(ws + l.tilerows_off);
    uint32_t *tile_off = reinterpret_cast<uint32_t *>(ws + l.tileoff_off);
    uint4 *tile_ids = reinterpret_cast<uint4 *>(ws + l.tileids_off);
    uint32_t *tile_head = reinterpret_cast<uint32_t *>(ws + l.tilehead_off);
    { plan_tile_len_kernel<<<(unsigned)n_tiles, 256, 0, s>>>(
        rowptr, perm, doc_off, ids16, N, n_tiles, (uint32_t)head, tile_rows, tile_len, tile_head); BMU_LAUNCHED(); }
    BMU_CUDA(cudaMemsetAsync(tile_rows + n_tiles, 0, 4, s));
    size_t tmp = l.scan_bytes;
    BMU_CUDA(cub::DeviceScan::ExclusiveSum(ws + l.scan_off, tmp, tile_rows, tile_off,
                                           (int)(n_tiles + 1), s));
    // the sweeps read one row past a tile's last (the next row is fetched ahead)
    { plan_check_kernel<<<1, 1, 0, s>>>(tile_off + n_tiles, (uint64_t)l.tile_rows_cap - 1, status); BMU_LAUNCHED(); }
    { plan_tile_fill_kernel<<<(unsigned)((n_tiles * 32 + 255) / 256), 256, 0, s>>>(
        rowptr, perm, doc_off, ids16, tile_len, tile_off, tile_head,
        (uint32_t)(head ? head / 32 : 1), feat_of_rank, N, n_tiles, interleave, tile_ids, status, D); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

// ---- the pass of the two-stage search (screen.cuh) ---------------------------------------------
// Its sweep sums integers, so the order inside a list is free, and it walks lists laid out as quads
// (plan_quad_fill_kernel): nothing of the 16-bit row lists above is needed.  Counters, head, lengths,
// order, tiles; eight launches where the general pass takes forty.  30,011 documents whose ids are no
// frequency ranks: 420 us of kernels -> 55; 120,000 labelled by frequency: 400 -> 125.

// The `head` features listed by most documents, ties to the lower id: feat[h] ascending, rank[f] = h or
// 0xffff.  The first block: a thread per PER neighbouring ids kept in registers, a binary search for the
// smallest threshold with at most `head` features above it, then one scan.  It is bound by the latency of
// its reductions; counters and ranks move 16 bytes at a time (12 us for 16384 features; two bytes at a
// time, each a sector of its own, 24).  The other blocks clear `zeroed` words for the kernels behind.
template <int PER>
__global__ void __launch_bounds__(1024)
plan_select_kernel(const uint32_t *__restrict__ count, int32_t D, int32_t head, uint16_t *__restrict__ rank,
                   uint16_t *__restrict__ feat, uint4 *__restrict__ zeroed, int32_t n_zeroed)
{
    static_assert(PER % 8 == 0, "whole vectors of ranks");
    __shared__ uint32_t s_warp[2][32];
    if (blockIdx.x > 0) {
        for (int i = (blockIdx.x - 1) * 1024 + threadIdx.x; i < n_zeroed; i += (gridDim.x - 1) * 1024)
            zeroed[i] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, f0 = (int)threadIdx.x * PER;
    uint32_t v[PER], hi = 0;
#pragma unroll
    for (int i = 0; i < PER; i += 4) {
        if (f0 + i + 4 <= D) {
            const uint4 t = __ldg(reinterpret_cast<const uint4 *>(count + f0 + i));
            v[i] = t.x; v[i + 1] = t.y; v[i + 2] = t.z; v[i + 3] = t.w;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[i + e] = f0 + i + e < D ? __ldg(count + f0 + i + e) : 0u;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) hi = max(hi, v[i + e]);
    }
    int turn = 0;                                     // two buffers: one barrier per reduction
    auto block_reduce = [&](uint32_t x, bool sum) {
        x = sum ? __reduce_add_sync(0xffffffffu, x) : __reduce_max_sync(0xffffffffu, x);
        turn ^= 1;
        if (lane == 0) s_warp[turn][warp] = x;
        __syncthreads();
        x = s_warp[turn][lane];
        return sum ? __reduce_add_sync(0xffffffffu, x) : __reduce_max_sync(0xffffffffu, x);
    };
    uint32_t lo = 0, above = 0;
    if (D > head) {
        hi = block_reduce(hi, false);
        while (lo < hi) {
            const uint32_t mid = lo + (hi - lo) / 2;
            uint32_t n = 0;
#pragma unroll
            for (int i = 0; i < PER; ++i) n += v[i] > mid;
            if (block_reduce(n, true) <= (uint32_t)head) hi = mid; else lo = mid + 1;
        }
        uint32_t n = 0;
#pragma unroll
        for (int i = 0; i < PER; ++i) n += v[i] > lo;
        above = block_reduce(n, true);
    }
    // those above the threshold and the first of those at it; low half counts the former, high the latter
    uint32_t mine = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (f0 + i < D) mine += D <= head || v[i] > lo ? 1u : v[i] == lo ? 0x10000u : 0u;
    uint32_t inc = mine;
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, inc, m);
        if (lane >= m) inc += x;
    }
    turn ^= 1;
    if (lane == 31) s_warp[turn][warp] = inc;
    __syncthreads();
    uint32_t before = inc - mine;
    const uint32_t others = __reduce_add_sync(0xffffffffu, lane < warp ? s_warp[turn][lane] : 0u);
    before += others;
    uint32_t over = before & 0xffffu, at = before >> 16;
    const uint32_t room = (uint32_t)head - above;     // how many at the threshold still fit
#pragma unroll
    for (int i = 0; i < PER; i += 8) {
        if (f0 + i >= D) break;
        uint32_t r[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const uint32_t c = v[i + e];
            const bool is_over = D <= head || c > lo, is_at = !is_over && c == lo;
            const uint32_t slot = over + min(at, room);
            const bool in = f0 + i + e < D && (is_over || (is_at && at < room));
            r[e >> 1] |= (in ? slot : 0xffffu) << (16 * (e & 1));
            if (in) feat[slot] = (uint16_t)(f0 + i + e);
            over += is_over;
            at += is_at;
        }
        if (f0 + i + 8 <= D) *reinterpret_cast<uint4 *>(rank + f0 + i) = make_uint4(r[0], r[1], r[2], r[3]);
        else
            for (int e = 0; f0 + i + e < D; ++e) rank[f0 + i + e] = (uint16_t)(r[e >> 1] >> (16 * (e & 1)));
    }
}

// A document's sorting key: how many of its ids are gathered -- the ones outside the head, or all of
// them if it lists a head id twice (plan_key_kernel above) -- and, for an order by content, the ids of
// its two rarest features and of the most frequent gathered one below the length.  One warp each; ids
// that ascend strictly cannot repeat, only the others are looked at again through a bit per head row.
// For an order by length alone (`hist`) a block counts its lengths in shared memory first, and the last
// block to finish turns the counters into positions: two launches less, some 10 us.
static const int KEY_WARPS = 16;

__global__ void __launch_bounds__(KEY_WARPS * 32)
plan_quad_key_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                     const uint16_t *__restrict__ rank, const uint32_t *__restrict__ count, int64_t N,
                     int32_t head, uint32_t *__restrict__ key, int64_t D, uint32_t *__restrict__ status,
                     u64 *__restrict__ ckeys, uint32_t *__restrict__ cvals, uint32_t *__restrict__ hist)
{
    __shared__ uint32_t seen[KEY_WARPS][HEAD_ROWS_MAX / 32], bins[LOCAL_BINS], s_most, s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (hist) {
        for (int b = threadIdx.x; b < LOCAL_BINS; b += KEY_WARPS * 32) bins[b] = 0u;
        if (threadIdx.x == 0) s_most = 0u;
        __syncthreads();
    }
    uint32_t longest = 0;
    for (int64_t i = (int64_t)blockIdx.x * KEY_WARPS + warp; i < N; i += (int64_t)gridDim.x * KEY_WARPS) {
        const int beg = __ldg(rowptr + i), end = __ldg(rowptr + i + 1);
        int in_head = 0, last = -1;
        bool ascending = true;
        // (count << 16 | id): the smallest two name the rarest features, the largest the most frequent
        u64 r1 = ~0ull, r2 = ~0ull, top = 0ull;
        for (int e0 = beg; e0 < end; e0 += 128) {
            int f[4], h[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = e0 + 32 * u + lane;
                f[u] = e < end ? (int)BMU_IDX((uint32_t)__ldg(colidx + e), D, status) : 0x7fffffff;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) h[u] = f[u] == 0x7fffffff ? 0xffff : rank ? (int)__ldg(rank + f[u]) : f[u];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (e0 + 32 * u >= end) break;                       // (the same for the whole warp)
                int before = __shfl_up_sync(0xffffffffu, f[u], 1);
                if (lane == 0) before = last;
                ascending &= f[u] == 0x7fffffff || f[u] > before;
                last = __shfl_sync(0xffffffffu, f[u], 31);
                in_head += h[u] < head;
                if (ckeys && f[u] != 0x7fffffff) {
                    const u64 v = ((u64)__ldg(count + f[u]) << 16) | (uint32_t)f[u];
                    if (v < r1) { r2 = r1; r1 = v; } else if (v < r2) { r2 = v; }
                    if (h[u] >= head && v > top) top = v;
                }
            }
        }
        int repeat = 0;
        if (!__all_sync(0xffffffffu, ascending)) {
            for (int w = lane; w < head / 32; w += 32) seen[warp][w] = 0u;
            __syncwarp();
            for (int e = beg + lane; e < end; e += 32) {
                const int f = (int)BMU_IDX((uint32_t)__ldg(colidx + e), D, status);
                const int h = rank ? (int)__ldg(rank + f) : f;
                if (h < head) {
                    const uint32_t bit = 1u << (h & 31);
                    repeat |= (atomicOr(&seen[warp][h >> 5], bit) & bit) != 0u;
                }
            }
        }
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) in_head += __shfl_xor_sync(0xffffffffu, in_head, m);
        repeat = __any_sync(0xffffffffu, repeat);
        const uint32_t len = (uint32_t)(end - beg - (repeat ? 0 : in_head));
        longest = max(longest, min(len, (uint32_t)(PLAN_BINS - 1)));
        if (lane == 0) {
            key[i] = len;
            if (hist && len < LOCAL_BINS) atomicAdd(bins + len, 1u);
            else if (hist) atomicAdd(hist + (PLAN_BINS - 1 - min(len, (uint32_t)(PLAN_BINS - 1))), 1u);
        }
        if (ckeys) {
#pragma unroll
            for (int m = 16; m > 0; m >>= 1) {
                const u64 o1 = __shfl_xor_sync(0xffffffffu, r1, m), o2 = __shfl_xor_sync(0xffffffffu, r2, m);
                const u64 ot = __shfl_xor_sync(0xffffffffu, top, m);
                r2 = min(min(r2, o2), max(r1, o1));
                r1 = min(r1, o1);
                top = max(top, ot);
            }
            if (lane == 0) {
                ckeys[i] = (u64)(uint32_t)(PLAN_BINS - 1 - min(len, (uint32_t)(PLAN_BINS - 1))) << 48 |
                           (r1 & 0xffffull) << 32 | (r2 & 0xffffull) << 16 | (top & 0xffffull);
                cvals[i] = (uint32_t)i;
            }
        }
        __syncwarp();
    }
    if (!hist) return;
    uint32_t *most = status + STATUS_PLAN_MOST;
    if (lane == 0) atomicMax(&s_most, longest);
    __syncthreads();
    if (threadIdx.x == 0 && s_most > *reinterpret_cast<volatile uint32_t *>(most)) atomicMax(most, s_most);
    for (int b = threadIdx.x; b < LOCAL_BINS; b += KEY_WARPS * 32)
        if (bins[b]) atomicAdd(hist + (PLAN_BINS - 1 - b), bins[b]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(status + STATUS_KEY_TICKET, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    plan_scan_bins<KEY_WARPS>(hist, __ldcg(most), hist + PLAN_BINS);
}

// One block per tile, a warp per document: the head mask, and the gathered ids into quads -- whole
// groups of four rows, stored by pairs of documents: word 4s + r of the sixteen is row r of documents 2s
// and 2s + 1, so that one 128-bit load gives a lane four rows of the pair it gathers.  Absent entries name
// row D, which is all zeros.  Lists of up to QUAD_SMEM ids are put together in shared memory.  A tile has
// as many rows as its first document has ids, and takes its room from a common cursor: where a tile's
// quads lie does not matter to the sweep (in place of a scan over the tiles, four launches).
static const int QUAD_SMEM = 256;

__global__ void __launch_bounds__(256)
plan_quad_fill_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                      const uint16_t *__restrict__ rank, const int32_t *__restrict__ perm,
                      const uint32_t *__restrict__ key, int64_t N, int32_t head,
                      uint32_t *__restrict__ tile_len, uint32_t *__restrict__ tile_off,
                      uint32_t *__restrict__ cursor, uint32_t tile_rows_cap,
                      uint4 *__restrict__ tile_ids, uint32_t *__restrict__ tile_head,
                      uint32_t *__restrict__ status, int64_t D)
{
    __shared__ uint32_t s_mask[8][HEAD_ROWS_MAX / 32];
    __shared__ __align__(4) uint16_t s_ids[QUAD_SMEM][8];
    __shared__ uint32_t s_rows, s_off;
    if (threadIdx.x == 0) {
        uint32_t len = min(key[perm[8 * (int64_t)blockIdx.x]], 65535u);
        const uint32_t room = (len + 3) / 4 * 4, off = atomicAdd(cursor, room);
        const bool fits = off <= tile_rows_cap && room <= tile_rows_cap - off;
        if (!fits) { atomicOr(status, PLAN_STATUS_OVERFLOW); len = 0u; }
        tile_len[blockIdx.x] = len;
        tile_off[blockIdx.x] = s_off = fits ? off : 0u;
        s_rows = fits ? room : 0u;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, words = head / 32;
    const int64_t tile = blockIdx.x, p = tile * 8 + warp;
    const int rows = (int)s_rows;
    uint32_t *dst = reinterpret_cast<uint32_t *>(tile_ids + s_off);
    // entry (row, this warp's document): sixteen bits of a quad's word
    auto put = [&](int row, uint32_t f) {
        if (row < QUAD_SMEM) s_ids[row][warp] = (uint16_t)f;
        else reinterpret_cast<uint16_t *>(dst)[(row >> 2) * 32 + (4 * (warp >> 1) + (row & 3)) * 2 + (warp & 1)] = (uint16_t)f;
    };
    for (int w = lane; w < words; w += 32) s_mask[warp][w] = 0u;
    __syncwarp();
    int n = 0;
    if (p < N) {
        const int32_t i = perm[p];
        const int beg = __ldg(rowptr + i), end = __ldg(rowptr + i + 1);
        const bool whole = key[i] == (uint32_t)(end - beg);      // nothing of it goes to the head
        for (int e0 = beg; e0 < end; e0 += 128) {
            int f[4], h[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = e0 + 32 * u + lane;
                f[u] = e < end ? (int)BMU_IDX((uint32_t)__ldg(colidx + e), D, status) : -1;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) h[u] = f[u] < 0 ? 0 : whole ? 0xffff : rank ? (int)__ldg(rank + f[u]) : f[u];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (e0 + 32 * u >= end) break;
                const bool out = f[u] >= 0 && h[u] >= head;
                if (f[u] >= 0 && !out) atomicOr(&s_mask[warp][h[u] >> 5], 1u << (h[u] & 31));
                const uint32_t who = __ballot_sync(0xffffffffu, out);
                if (out) {
                    const int row = n + __popc(who & ((1u << lane) - 1u));
                    if (row < rows) put(row, (uint32_t)f[u]);
                }
                n += __popc(who);
            }
        }
    }
    for (int row = n + lane; row < rows; row += 32) put(row, (uint32_t)D);
    __syncthreads();
    for (int x = threadIdx.x; x < min(rows, QUAD_SMEM) * 4; x += 256) {      // word x of the tile
        const int row = (x >> 4) * 4 + (x & 3), s = (x >> 2) & 3;
        dst[x] = *reinterpret_cast<const uint32_t *>(&s_ids[row][2 * s]);
    }
    uint32_t *mask = tile_head + (size_t)p * words;
    for (int w = lane; w < words; w += 32) mask[w] = s_mask[warp][w];
}

int launch_plan_screen(const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz, int by_content,
                       int head, int relabel, int64_t D, char *ws, const PlanLayout &l, uint32_t *count,
                       uint16_t *rank_of, uint16_t *feat_of, bool selected, uint32_t *status, cudaStream_t s)
{
    const uint16_t *rank = nullptr;
    by_content = by_content && l.cluster_tmp_bytes > 0;
    const bool select = relabel != 2 && !selected;
    if (select || by_content) {
        const int rc = launch_feat_hist(colidx, nnz, D, count, s);
        if (rc) return rc;
    }
    if (relabel != 2) rank = rank_of;
    if (select) {
        uint4 *bins = reinterpret_cast<uint4 *>(ws + l.bins_off);        // the lengths' counters
        const int32_t n_bins = by_content ? 0 : PLAN_BINS / 4;
        if (D <= 16 * 1024) { plan_select_kernel<16><<<9, 1024, 0, s>>>(count, (int32_t)D, head, rank_of, feat_of, bins, n_bins); BMU_LAUNCHED(); }
        else { plan_select_kernel<64><<<9, 1024, 0, s>>>(count, (int32_t)D, head, rank_of, feat_of, bins, n_bins); BMU_LAUNCHED(); }
    }
    int32_t *perm = reinterpret_cast<int32_t *>(ws + l.perm_off);
    uint32_t *key = reinterpret_cast<uint32_t *>(ws + l.docoff_off);
    uint32_t *hist = reinterpret_cast<uint32_t *>(ws + l.bins_off);
    uint32_t *cursor = hist + PLAN_BINS;
    u64 *keys_in = reinterpret_cast<u64 *>(ws + l.cluster_off), *keys_out = keys_in + N;
    uint32_t *vals_in = reinterpret_cast<uint32_t *>(keys_out + N);
    if (!select && !by_content) BMU_CUDA(cudaMemsetAsync(hist, 0, (size_t)PLAN_BINS * 4, s));
    const int64_t key_blocks = (N + KEY_WARPS - 1) / KEY_WARPS;
    { plan_quad_key_kernel<<<(unsigned)(key_blocks < 592 ? key_blocks : 592), KEY_WARPS * 32, 0, s>>>(
        rowptr, colidx, rank, count, N, head, key, D, status, by_content ? keys_in : nullptr, vals_in,
        by_content ? nullptr : hist); BMU_LAUNCHED(); }
    if (by_content) {
        size_t tmp = l.cluster_tmp_bytes;
        BMU_CUDA(cub::DeviceRadixSort::SortPairs(ws + l.cluster_tmp_off, tmp, keys_in, keys_out, vals_in,
                                                 reinterpret_cast<uint32_t *>(perm), (int)N, 0, 64, s));
    } else {
        { plan_scatter_kernel<<<(unsigned)((N + LOCAL_DOCS - 1) / LOCAL_DOCS), 256, 0, s>>>(rowptr, key, N, cursor, perm, nullptr); BMU_LAUNCHED(); }
    }
    const int64_t n_tiles = (N + 7) / 8;
    uint32_t *tile_len = reinterpret_cast<uint32_t *>(ws + l.tilelen_off);
    uint32_t *tile_off = reinterpret_cast<uint32_t *>(ws + l.tileoff_off);
    const uint32_t rows_cap = (uint32_t)(l.tile_rows_cap < 0xffffffffull ? l.tile_rows_cap : 0xffffffffull);
    { plan_quad_fill_kernel<<<(unsigned)n_tiles, 256, 0, s>>>(
        rowptr, colidx, rank, perm, key, N, head, tile_len, tile_off, status + STATUS_TILE_CURSOR, rows_cap,
        reinterpret_cast<uint4 *>(ws + l.tileids_off), reinterpret_cast<uint32_t *>(ws + l.tilehead_off), status, D); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

}  // namespace bmu
