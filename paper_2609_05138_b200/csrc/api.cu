// Host side of the C ABI: argument checks, workspace layout, neuron-axis
// chunking (Section 4.2) and the order in which the kernels are queued.
#include "screen.cuh"

#include <stdarg.h>
#include <string.h>

#include <mutex>
#include <new>

namespace bmu {

static thread_local char g_err[512] = "";
thread_local unsigned long long g_kernel_launches = 0;

void set_error(const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

int cuda_fail(cudaError_t e, const char *what)
{
    set_error("%s: %s", what, cudaGetErrorString(e));
    return BMU_ERR_CUDA;
}

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static const int64_t MAX_M = (int64_t)1 << 30;   // row pitch M*4 must fit 32 bits
static const int64_t MAX_I32 = 0x7fffffff;

// ---- workspace layout -----------------------------------------------------
struct Layout {
    size_t status_off, count_off, sets_off, tickets_off, slots_off, norms_off, state_off, state2_off, head_off, repack_off, screen_off, plan_off, total;
    PlanLayout plan;
    ScreenLayout screen;
};


static int64_t device_l2()
{
    int dev = 0, l2 = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev) != cudaSuccess || l2 <= 0)
        l2 = 64 << 20;
    return l2;
}

static int device_sms()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
        n = 148;
    return n;
}

// Neurons per launch of the tensor-core sweep: whole 256-neuron slabs whose rows take about
// 0.4 of L2 (768 neurons at D = 16384 on a 126 MB L2).  Measured on config 4: 768 beats 1024 by
// 2 % and 512 by 3 %; at 1024 the chunk (67 MB) no longer stays resident in the two-part L2 and
// its rows are fetched from DRAM five times over.
static int64_t mma_auto_chunk(int64_t D, int64_t M)
{
    int64_t c = (int64_t)((double)device_l2() * 0.42) / (D * 4) / MMA_SLAB * MMA_SLAB;
    if (c < MMA_SLAB) c = MMA_SLAB;
    if (c > M) c = M / MMA_SLAB * MMA_SLAB;
    return c;
}

static int64_t mma_chunk(const bmu_opts &o, int64_t D, int64_t M)
{
    return o.chunk_neurons ? ((int64_t)o.chunk_neurons + MMA_SLAB - 1) / MMA_SLAB * MMA_SLAB
                           : mma_auto_chunk(D, M);
}

// Bytes of the compact chunk copy: unless told otherwise the tensor-core sweeps gather from a
// [D][chunk] copy of the chunk's columns (4 KB row pitch at a chunk of 1024), made before each
// launch, instead of from the codebook itself (row pitch 4 * M bytes), so that the rows of a
// chunk share pages: 2-7 % faster on every benchmark shape for 0.2 % more traffic.
static size_t mma_repack_bytes(const bmu_opts &o, int64_t D, int64_t M, int64_t N, int64_t nnz,
                               bool top2)
{
    if (o.repack == 2 || (o.kernel != 0 && o.kernel != 6)) return 0;
    if (D > LANES_MAX_D || M < MMA_SLAB) return 0;
    const int64_t chunk = mma_chunk(o, D, M);
    if (M <= chunk) return 0;                      // one launch: the codebook is the chunk
    (void)N; (void)nnz;
    return (size_t)D * (size_t)(chunk < M ? chunk : M) * sizeof(float);
}

// one block per codebook row: `width_bytes` (a multiple of 16) from byte `off_bytes` of the row
__global__ void __launch_bounds__(256)
repack_chunk_kernel(const char *__restrict__ W, int64_t pitch_bytes, int64_t off_bytes,
                    int32_t width_bytes, char *__restrict__ out)
{
    const uint4 *src = reinterpret_cast<const uint4 *>(W + (int64_t)blockIdx.x * pitch_bytes + off_bytes);
    uint4 *dst = reinterpret_cast<uint4 *>(out + (int64_t)blockIdx.x * width_bytes);
    for (int i = threadIdx.x; i < width_bytes / 16; i += 256) dst[i] = __ldcs(src + i);
}

// Features summed on the tensor cores: 640 (measured best of 512 .. 1024 on configs 2-5 in
// full-length runs, where the board sits at its power cap: 768 wins short runs at boost clocks
// and loses 1-2 % once the cap binds), less if the vocabulary is smaller.
static int mma_head_rows(const bmu_opts &o, int64_t D)
{
    if (o.head_rows) return o.head_rows;
    const int64_t cap = D / 64 * 64, want = 640;
    return (int)(cap < want ? (cap < 64 ? 64 : cap) : want);
}

// Features the screening sweep sums on the tensor cores: all that tensor memory holds beside the
// accumulator (1536), or the whole vocabulary if it is smaller.
static int screen_head_rows(const bmu_opts &o, int64_t D)
{
    if (o.head_rows) return o.head_rows;
    const int64_t up = (D + 63) / 64 * 64;
    return (int)(up < SC_MAX_HEAD ? up : SC_MAX_HEAD);
}

static Layout layout_for(int64_t D, int64_t M, int64_t N, int64_t nnz, int kernel,
                         bool top2 = false, int head = 640, size_t repack_bytes = 0, int cluster = 0,
                         int64_t screen_chunk = 0, bool few = false)
{
    Layout l;
    size_t off = 0;
    l.status_off = off; off = 256;
    if (screen_chunk) off = align_up((size_t)STATUS_WORDS * 4, 256);
    l.count_off = off;                   // (the features' counters, cleared with the status word)
    if (screen_chunk) off = align_up(off + (size_t)D * sizeof(uint32_t), 256);
    l.sets_off = off;                    // (how far each set of documents reaches, cleared too)
    if (screen_chunk) off = align_up(off + (size_t)((N + SC_DOCS - 1) / SC_DOCS) * sizeof(uint32_t), 256);
    l.tickets_off = l.slots_off = off;
    if (few) {                           // (the tickets behind the status word: cleared with it)
        off = align_up(off + (size_t)N * sizeof(uint32_t), 256);
        l.slots_off = off; off = align_up(off + few_slots_bytes(M, N, top2), 256);
    }
    l.norms_off = off; off = align_up(off + (size_t)M * sizeof(float), 256);
    l.state_off = off; off = align_up(off + (size_t)N * sizeof(u64), 256);
    l.state2_off = off;
    if (top2) off = align_up(off + (size_t)N * sizeof(u64), 256);
    // split image of the frequent rows for the tensor-core sweep (it may be the automatic choice)
    l.head_off = off;
    if (!screen_chunk && (kernel == 0 || kernel == 6) && D >= head && D <= LANES_MAX_D && M >= MMA_SLAB)
        off = align_up(off + head_image2_bytes(M, head), 256);
    l.repack_off = off;                  // compact copy of the codebook chunk being swept
    off = align_up(off + repack_bytes, 256);
    l.screen_off = off;                  // arrays of the screened search
    memset(&l.screen, 0, sizeof(l.screen));
    if (screen_chunk) {
        screen_layout(D, M, N, head, screen_chunk, top2, device_sms(), &l.screen);
        off += l.screen.total;
    }
    l.plan_off = off;
    memset(&l.plan, 0, sizeof(l.plan));
    if (kernel != 1 && D <= LANES_MAX_D) off += plan_bytes(N, nnz, head, D, cluster, screen_chunk != 0, &l.plan);
    l.total = off;
    return l;
}

// How the tiling pass orders the documents: 0 corpus order, 1 by length, 3 / 4 by length and
// content.  The tensor-core sweep takes 3 unless told otherwise (measured on configs 2-4: 0.5,
// 2.8 and 2.5 % faster than by length alone, the extra sort included; 4 gains less).
static int plan_order(const bmu_opts &o, bool tensor_core_sweep)
{
    if (o.cluster == 2) return 0;
    if (o.cluster >= 3) return o.cluster;
    return (o.cluster == 0 && tensor_core_sweep) ? 3 : 1;
}

// ---- which of the automatic ways a search takes ----------------------------------------------
// Three ways compete: straight from the CSR with the neuron axis over the grid (sweep_few.cu; no
// preparation, every update from L2), the planned warp-per-document kernel (a tiling pass, L1 hits)
// and the two-stage search (screen.cuh: two more reads of the codebook, a quarter of the bytes per
// update).  Their times in us for U = nnz * M updates, fitted to searches of 300 .. 30,000 documents of 79
// ids (lognormal) against 1,024 .. 16,384 units, D = 4,096 and 16,384:
//   few       15 + U / 4.5e6 (rows that are not whole 16-byte pieces: U / 1.9e6)
//   planned   0.09 M + U / 1.1e7 (fp16 codebook: U / 1.35e7) for equally long documents, which it likes
//             best; 60 more for these.  It is only left where it loses even so.  On maps below a
//             thousand units its warps are not full: 50 + U' / 6.7e6, the units in whole 128s (400 units,
//             D = 4,096, 30,000 documents of 64 ids: 244, two-stage 160; 256 units: 122 and 148)
//   two-stage 90 + 0.0022 D + 0.009 M + 1.6e-6 D M + 0.002 N + U / 3.3e7
// e.g. D = 4,096, M = 1,024: 4,000 documents 90 / 161 / 144 us, 10,000: 215 / 208 / 174; D = 16,384,
// M = 4,096: 1,000 documents 92 / 454 / 269, 10,000: 761 / 757 / 450 (with slabs by norm and blocks that stay, on an iid
// codebook: 87 / 180 / 120, - / 211 / 155, 99 / 551 / 279, - / 734 / 426; the model has not been fitted again).  Two
// lines beside the model: from
// 1,024 documents and 600,000 listings on it is never the first, and below 1,024 documents never the second
// (its warps would not fill the chip) unless two stages are ruled out and the sweep is large (2e10 updates).
// There the first takes 60 + U / 6.1e6 (3.1e6) for more than a few hundred us, and two stages 0.2 us more
// per id of a list, whose ends nothing hides; they are chosen where they promise a tenth.  First / two
// stages in us, 1,000 documents: 80 ids, 127 x 127, D = 4,096 493 / 367, 400 ids 2091 / 580; 400 ids,
// M = 65,536, D = 16,384 4344 / 3324, M = 16,384 1083 / 916; but 700 ids, M = 4,096 506 / 456 (left),
// 500 of 400 ids on 75 x 75 407 / 440.
static const int64_t FEW_MAX_DOCS = 1024, FEW_MAX_LISTINGS = 600000, ONE_SHOT_READS = (int64_t)1 << 25;

static double few_us(int64_t M, double u) { return 15.0 + u / (M % 4 == 0 ? 4.5e6 : 1.9e6); }
static double planned_us(int64_t M, double nnz, bool f16)
{
    const double wide = 0.09 * (double)M + nnz * (double)M / (f16 ? 1.35e7 : 1.1e7);
    const double narrow = 50.0 + nnz * (double)((M + 127) / 128 * 128) / 6.7e6;
    return f16 || wide > narrow ? wide : narrow;
}
static double two_stage_us(int64_t D, int64_t M, int64_t N, double u)
{
    return 90.0 + 0.0022 * (double)D + 0.009 * (double)M + 1.6e-6 * (double)D * (double)M + 0.002 * (double)N + u / 3.3e7;
}

// options of the warp-per-document kernels: whoever sets one means those kernels (and so, where the
// sweep is not large, does a chunk of their neurons)
static bool rows_opts(const bmu_opts &o) { return o.vec || o.warps || o.docs_per_warp; }

static bool screen_possible(const bmu_opts &o, int64_t D, int64_t M)
{
    return o.cluster != 2 && D >= 1 && D <= LANES_MAX_D && M >= 1 && screen_head_rows(o, D) <= SC_MAX_HEAD;
}

// (a one-shot search that has not read its number of listings back says 0: the first)
static bool few_wanted(const bmu_opts &o, int64_t D, int64_t M, int64_t N, int64_t nnz)
{
    if (o.kernel != 0 || o.two_stage == 1 || o.chunk_neurons || rows_opts(o)) return false;
    const double u = (double)nnz * (double)M;
    const bool screened = o.two_stage != 2 && screen_possible(o, D, M);
    if (N < FEW_MAX_DOCS) {
        if (!screened) return u < 2e10 || D > LANES_MAX_D || M % 4 != 0 || M < 256;
        const double list = (double)nnz / (double)(N > 0 ? N : 1);
        return 60.0 + u / (M % 4 == 0 ? 6.1e6 : 3.1e6) < 1.1 * (two_stage_us(D, M, 0, u) + 0.2 * list);
    }
    return nnz < FEW_MAX_LISTINGS && (!screened || few_us(M, u) < two_stage_us(D, M, N, u));
}

static bool screen_wanted(const bmu_opts &o, int64_t D, int64_t M, int64_t N, int64_t nnz, bool f16 = false)
{
    if (o.two_stage == 2 || !screen_possible(o, D, M)) return false;
    if (o.two_stage == 1) return o.kernel == 0 || o.kernel == 6;
    if (o.kernel != 0 || (!f16 && few_wanted(o, D, M, N, nnz))) return false;
    const double u = (double)nnz * (double)M;
    if (rows_opts(o) || o.chunk_neurons) return u >= 2e10;
    if (N < FEW_MAX_DOCS && !f16) return true;
    const bool planned_ok = f16 || (M % 4 == 0 && M >= 256);
    return !planned_ok || two_stage_us(D, M, N, u) < planned_us(M, (double)nnz, f16);
}

// Does the two-stage search order equally long documents by content (bmu_opts.cluster 3 and 4)?  The
// sweep gains 1-2 % from it, the sort costs 60-110 us: left to itself only where a plan is made to be
// kept or the sweep takes some ten milliseconds.
static int screen_by_content(const bmu_opts &o, int64_t M, int64_t nnz, bool kept)
{
    if (o.cluster) return o.cluster >= 3;
    return kept || (double)nnz * (double)M >= 2e11;
}

// Neurons per launch: the chunk's 8-bit image, (D + 1) * chunk bytes, in about 0.4 of L2
static int64_t screen_chunk(const bmu_opts &o, int64_t D)
{
    int64_t c = o.chunk_neurons ? ((int64_t)o.chunk_neurons + MMA_SLAB - 1) / MMA_SLAB * MMA_SLAB
                                : (int64_t)((double)device_l2() * 0.42) / (D + 1) / MMA_SLAB * MMA_SLAB;
    const int64_t most = (int64_t)SC_MAX_SLABS * SC_SLAB;
    return c < MMA_SLAB ? MMA_SLAB : c > most ? most : c;
}

static Layout screen_layout_of(const bmu_opts &o, int64_t D, int64_t M, int64_t N, int64_t nnz, bool top2)
{
    return layout_for(D, M, N, nnz, 6, top2, screen_head_rows(o, D), 0, plan_order(o, true), screen_chunk(o, D));
}

// the layout search_impl uses for these options (the workspace-size queries must agree with it)
static Layout layout_of(const bmu_opts &o, int64_t D, int64_t M, int64_t N, int64_t nnz, bool top2,
                        bool plan = false)
{
    if (few_wanted(o, D, M, N, nnz))                // (a plan is made for its order only)
        return layout_for(D, M, N, nnz, plan ? 3 : 1, top2, 640, 0, 0, 0, true);
    if (screen_wanted(o, D, M, N, nnz))
        return screen_layout_of(o, D, M, N, nnz, top2);
    return layout_for(D, M, N, nnz, o.kernel, top2, mma_head_rows(o, D),
                      mma_repack_bytes(o, D, M, N, nnz, top2), plan_order(o, true));
}

// Could a search of no more documents and listings take the two-stage form?  Its model grows slower in the
// listings than the others': most likely with all of them.  Below 1,024 documents it gains with the
// documents (shorter lists), above it loses; with a half-precision codebook it only loses.
static bool screen_within(const bmu_opts &o, int64_t D, int64_t M, int64_t N, int64_t nnz, bool f16 = false)
{
    if (N <= 0) return false;
    if (f16) return screen_wanted(o, D, M, 1, nnz, true);
    return screen_wanted(o, D, M, N < FEW_MAX_DOCS ? N : FEW_MAX_DOCS - 1, nnz) ||
           (N >= FEW_MAX_DOCS && screen_wanted(o, D, M, FEW_MAX_DOCS, nnz));
}

// What the workspace queries answer: room for every way that a search of these or smaller sizes may take
// (N and nnz; D, M and the options the same), so that a workspace sized for the largest batch serves all,
// and one sized with default options the same sizes with others.  Each part grows with N and with nnz.
static size_t query_bytes(const bmu_opts &o, int64_t D, int64_t M, int64_t N, int64_t nnz, bool top2, bool plan)
{
    size_t need = layout_of(o, D, M, N, nnz, top2, plan).total;
    auto room = [&](const Layout &l) { if (l.total > need) need = l.total; };
    if (o.kernel == 0) {
        room(layout_for(D, M, N, nnz, 0, top2, mma_head_rows(o, D), mma_repack_bytes(o, D, M, N, nnz, top2),
                        plan_order(o, true)));
        room(layout_for(D, M, N, nnz, plan ? 3 : 1, top2, 640, 0, 0, 0, true));
    }
    if (screen_within(o, D, M, N, nnz)) room(screen_layout_of(o, D, M, N, nnz, top2));
    return need;
}

static int check_sizes(int64_t D, int64_t M, int64_t N, int64_t nnz)
{
    if (D < 0 || M < 0 || N < 0 || nnz < 0) {
        set_error("negative size (D=%lld M=%lld N=%lld nnz=%lld)", (long long)D, (long long)M,
                  (long long)N, (long long)nnz);
        return BMU_ERR_INVALID_ARG;
    }
    if (M >= MAX_M || D > MAX_I32 || N >= MAX_I32 || nnz > MAX_I32) {
        set_error("size beyond the limits (M < 2^30; D, N, nnz < 2^31)");
        return BMU_ERR_UNSUPPORTED;
    }
    return BMU_OK;
}

static int check_opts(const bmu_opts &o)
{
    if (o.tile_order < 0 || o.tile_order > 2) { set_error("bmu_opts.tile_order must be 0, 1 or 2"); return BMU_ERR_INVALID_ARG; }
    if (o.tile_head < 0 || o.tile_head > 1) { set_error("bmu_opts.tile_head must be 0 or 1"); return BMU_ERR_INVALID_ARG; }
    if (o.head_rows < 0 || o.head_rows > HEAD_ROWS_MAX || o.head_rows % 64 != 0) {
        set_error("bmu_opts.head_rows must be 0 or a multiple of 64 up to %d", HEAD_ROWS_MAX);
        return BMU_ERR_INVALID_ARG;
    }
    if (o.repack < 0 || o.repack > 2) { set_error("bmu_opts.repack must be 0, 1 or 2"); return BMU_ERR_INVALID_ARG; }
    if (o.relabel < 0 || o.relabel > 2) { set_error("bmu_opts.relabel must be 0, 1 or 2"); return BMU_ERR_INVALID_ARG; }
    if (o.two_stage < 0 || o.two_stage > 2) { set_error("bmu_opts.two_stage must be 0, 1 or 2"); return BMU_ERR_INVALID_ARG; }
    for (int i = 0; i < 2; ++i)
        if (o.reserved[i] != 0) { set_error("bmu_opts.reserved must be zero"); return BMU_ERR_INVALID_ARG; }
    if (o.kernel != 0 && o.kernel != 1 && o.kernel != 3 && o.kernel != 4 && o.kernel != 6) {
        set_error("bmu_opts.kernel must be 0, 1, 3, 4 or 6");
        return BMU_ERR_INVALID_ARG;
    }
    if (o.stage_rows != 0 || o.stages != 0) {
        set_error("bmu_opts.stage_rows and bmu_opts.stages must be zero");
        return BMU_ERR_INVALID_ARG;
    }
    if (o.cluster < 0 || o.cluster > 4) { set_error("bmu_opts.cluster must be 0 .. 4"); return BMU_ERR_INVALID_ARG; }
    if (o.chunk_neurons < 0) { set_error("bmu_opts.chunk_neurons < 0"); return BMU_ERR_INVALID_ARG; }
    if (o.vec != 0 && o.vec != 4 && o.vec != 8) { set_error("bmu_opts.vec must be 0, 4 or 8"); return BMU_ERR_INVALID_ARG; }
    return BMU_OK;
}

// Neurons per L2-resident chunk: the chunk's share of the codebook,
// D * chunk * 4 bytes, is kept to about half of L2 so that the rows of one
// chunk stay cached while every document passes over them.
static int64_t auto_chunk(int64_t D, int64_t M, int slab)
{
    int64_t c = D > 0 ? (device_l2() / 2) / (D * 4) : M;
    c = c / slab * slab;
    if (c < slab) c = slab;
    if (c > M) c = (M + slab - 1) / slab * slab;
    return c;
}

// Which kernel a search takes and how it is cut into launches.
struct Route {
    int kernel;            // 1 generic, 3 planned, 4 tiled, 6 tensor-core head + gathered tail
    int head;              // features summed on the tensor cores (kernel 6), else 0
    int slab;              // neurons a block (or warp) carries at a time
    int docs_per_block;    // documents that share a block
    int64_t chunk;         // neurons per launch (one L2-resident chunk)
    int64_t m_full;        // neurons covered by whole slabs; the rest takes the generic kernel
    int repack;            // 1: a compact copy of the chunk's columns precedes each launch
    int few;               // few documents: straight from the CSR (sweep_few.cu)
    int two_stage;         // screened, then verified (screen.cuh): the screen's head, else 0
};

static int route_search(const bmu_opts &o, int64_t D, int64_t M, int64_t N, int64_t nnz, uintptr_t w_addr,
                        Route &r)
{
    const int head = mma_head_rows(o, D);
    r.two_stage = 0;
    r.few = few_wanted(o, D, M, N, nnz);
    if (screen_wanted(o, D, M, N, nnz)) {
        r.kernel = 6; r.head = head; r.slab = SC_SLAB; r.docs_per_block = SC_DOCS;
        r.two_stage = screen_head_rows(o, D);
        r.chunk = screen_chunk(o, D);
        r.m_full = M;
        r.repack = 1;                      // the images of the chunk, made before each launch
        return BMU_OK;
    }
    if (o.two_stage == 1) {
        set_error("the two-stage sweep needs kernel 0 or 6, 1 <= D <= %d, length-ordered documents "
                  "(cluster != 2) and head_rows <= %d", LANES_MAX_D, SC_MAX_HEAD);
        return BMU_ERR_UNSUPPORTED;
    }
    // the planned warp-per-document kernel needs 16-bit ids and whole 16-byte row pieces
    const bool planned_ok = D <= LANES_MAX_D && M % 4 == 0 && M >= rows_slab_width(o) &&
                            (w_addr & 15) == 0;
    if (o.kernel == 3 && !planned_ok) {
        set_error("planned kernel needs M %% 4 == 0, M >= 128, D <= %d and W 16-byte aligned",
                  LANES_MAX_D);
        return BMU_ERR_UNSUPPORTED;
    }
    const bool tiled_ok = planned_ok && M >= 128 && o.cluster != 2;
    // tensor-core head: additionally at least one whole 256-neuron slab and `head` features
    const bool mma_ok = tiled_ok && D >= head && M >= MMA_SLAB;
    if (o.kernel == 6 && !mma_ok) {
        set_error("tensor-core sweep needs what the tiled kernel needs, D >= %d and M >= %d",
                  head, MMA_SLAB);
        return BMU_ERR_UNSUPPORTED;
    }
    // automatic choice for large sweeps: the tensor-core sweep where it applies, else the tiled
    // kernel; both repay their extra preparation only when there is enough to sweep
    const bool big = !r.few && (double)nnz * (double)M >= 2e10;
    const bool mma = o.kernel == 6 || (o.kernel == 0 && mma_ok && big);
    const bool tiled = !mma && (o.kernel == 4 || (o.kernel == 0 && tiled_ok && big));
    if (tiled && !tiled_ok) {
        set_error("tiled kernel needs M %% 4 == 0, M >= 128, D <= %d, W 16-byte aligned and "
                  "length-ordered documents (cluster != 2)", LANES_MAX_D);
        return BMU_ERR_UNSUPPORTED;
    }
    const bool planned = !tiled && !mma && (o.kernel == 3 || (o.kernel == 0 && planned_ok));
    r.head = 0; r.repack = 0;
    if (mma) {
        r.kernel = 6; r.head = head; r.slab = 256; r.docs_per_block = MMA_DOCS;
        r.chunk = mma_chunk(o, D, M);
        r.m_full = M / MMA_SLAB * MMA_SLAB;
        r.repack = o.repack != 2 && M > r.chunk;
    } else if (tiled) {
        r.kernel = 4; r.slab = 128; r.docs_per_block = 8 * (o.warps ? o.warps : 4);
        r.chunk = o.chunk_neurons ? (o.chunk_neurons + 127) / 128 * 128 : auto_chunk(D, M, 128);
        r.m_full = M / 128 * 128;
    } else if (planned) {
        r.kernel = 3; r.slab = rows_slab_width(o); r.docs_per_block = o.warps ? o.warps : 16;
        r.chunk = o.chunk_neurons ? (o.chunk_neurons + r.slab - 1) / r.slab * r.slab
                                  : auto_chunk(D, M, r.slab);
        r.m_full = M / r.slab * r.slab;
    } else {
        r.kernel = 1; r.slab = 32 * (o.vec ? o.vec : 4);
        r.docs_per_block = (o.warps ? o.warps : 16) * (o.docs_per_warp ? o.docs_per_warp : 4);
        r.chunk = o.chunk_neurons ? (o.chunk_neurons + r.slab - 1) / r.slab * r.slab
                                  : auto_chunk(D, M, r.slab);
        r.m_full = M;
    }
    return BMU_OK;
}

// Cuts [0, m_full) into the launches of the tensor-core sweep: as many as chunks of `chunk`
// neurons need, the 256-neuron slabs dealt evenly among them (so that the last launch is not a
// single slab whose MMAs nothing overlaps).  Launch k covers [cut(k), cut(k + 1)).
struct LaunchCuts {
    int64_t slabs, n, base, rem;
    LaunchCuts(int64_t m_full, int64_t chunk)
    {
        slabs = m_full / MMA_SLAB;
        n = (m_full + chunk - 1) / chunk;
        base = n ? slabs / n : 0;
        rem = n ? slabs % n : 0;
    }
    int64_t cut(int64_t k) const { return (k * base + (k < rem ? k : rem)) * MMA_SLAB; }
};

// where the head's tables of a two-stage search are
static uint16_t *screen_rank(const Layout &l, char *base, const ScreenShared *shared)
{
    return reinterpret_cast<uint16_t *>(shared ? shared->base + shared->lay.rank : base + l.plan_off + l.plan.rank_off);
}
static uint16_t *screen_feat(const Layout &l, char *base, const ScreenShared *shared)
{
    return reinterpret_cast<uint16_t *>(shared ? shared->base + shared->lay.feat : base + l.plan_off + l.plan.feat_off);
}

// The two stages of a screened search, launch by launch: images of the chunk, sweep, the lists of
// what the sweep could not rule out; then their exact evaluation and the outputs.  The plan (quad
// layout) is in the workspace already.
static int screen_search(const void *W, int f16, int64_t D, int64_t M, const float *norms,
                         const int32_t *rowptr, const int32_t *colidx, int64_t N, int head, int relabel,
                         const Layout &l, char *base, uint32_t *status, u64 *state, u64 *state2,
                         int32_t *out_bmu, float *out_dist, int32_t *out_bmu2, float *out_dist2,
                         ScreenShared *shared, cudaStream_t s)
{
    char *pw = base + l.plan_off, *sb = base + l.screen_off;
    const bool ranked = relabel != 2, top2 = state2 != nullptr;
    const ScreenLayout &cl = shared ? shared->lay : l.screen;           // of the arrays of the codebook
    char *cb = shared ? shared->base : sb;
    const uint16_t *feat = ranked ? screen_feat(l, base, shared) : nullptr;
    const uint16_t *rank = ranked ? screen_rank(l, base, shared) : nullptr;
    const int32_t *perm = reinterpret_cast<const int32_t *>(pw + l.plan.perm_off);
    float *scalars = reinterpret_cast<float *>(cb + cl.scalars), *earlier = nullptr;
    if (shared) {                                                       // two sets in turn
        if (shared->used) earlier = scalars + (shared->used - 1) % 2 * SC_SCALARS;
        scalars += shared->used++ % 2 * SC_SCALARS;
    }
    uint32_t *set_reach = reinterpret_cast<uint32_t *>(base + l.sets_off);
    ScreenArgs a;
    a.tile_len = reinterpret_cast<const uint32_t *>(pw + l.plan.tilelen_off);
    a.tile_off = reinterpret_cast<const uint32_t *>(pw + l.plan.tileoff_off);
    a.tile_ids = reinterpret_cast<const uint4 *>(pw + l.plan.tileids_off);
    a.tile_head = reinterpret_cast<const uint32_t *>(pw + l.plan.tilehead_off);
    int rc = launch_screen_prepare(W, f16, D, M, norms, rowptr, colidx, N, head, feat, rank, perm,
                                   reinterpret_cast<const uint32_t *>(pw + l.plan.docoff_off), a.tile_len, cb, cl,
                                   scalars, earlier, reinterpret_cast<float *>(sb + l.screen.sample),
                                   reinterpret_cast<float *>(sb + l.screen.window),
                                   reinterpret_cast<float2 *>(sb + l.screen.reach),
                                   reinterpret_cast<uint32_t *>(sb + l.screen.amin),
                                   reinterpret_cast<uint32_t *>(sb + l.screen.lcount), set_reach, l.screen.n_pad, top2,
                                   status, s);
    if (rc) return rc;
    const int64_t slabs = (M + SC_SLAB - 1) / SC_SLAB;
    const int64_t launches = (slabs + l.screen.chunk_slabs - 1) / l.screen.chunk_slabs;
    uint32_t *tickets = reinterpret_cast<uint32_t *>(sb + l.screen.tickets);
    uint32_t *nat_list = reinterpret_cast<uint32_t *>(sb + l.screen.nat_list);
    const int sets = (int)(l.screen.n_pad / SC_DOCS);
    const int64_t ord_launches = screen_order_possible(D, M, N) ? cl.ord_launches : 0;
    if (ord_launches && (rc = launch_screen_order(norms, D, M, N, launches, cb, cl, scalars, earlier, status, set_reach, sets,
                                                  tickets, nat_list, s)))
        return rc;
    a.kpack = reinterpret_cast<const uint32_t *>(cb + cl.kpack);
    a.scalars = scalars;
    a.window = reinterpret_cast<const float *>(sb + l.screen.window);
    a.cval = reinterpret_cast<float2 *>(sb + l.screen.cval);
    a.cval2 = reinterpret_cast<float *>(sb + l.screen.cval2);
    a.cmask = reinterpret_cast<uint4 *>(sb + l.screen.cmask);
    a.status = status; a.ticket = status + STATUS_SWEEP_TICKET;
    a.D = D; a.n_tiles = (N + 7) / 8; a.n_pad = l.screen.n_pad; a.tile_rows_cap = l.plan.tile_rows_cap;
    a.head = head; a.head_pad = l.screen.head_pad;
    a.splits = l.screen.splits; a.most_splits = l.screen.most_splits; a.blocks = sets; a.nat_list = nat_list;
    VerifyArgs v;
    v.W = W; v.f16 = f16; v.D = D; v.M = M; v.N = N; v.n_pad = a.n_pad; v.norms = norms;
    v.rowptr = rowptr; v.colidx = colidx; v.perm = perm; v.window = a.window;
    v.cval = a.cval; v.cval2 = a.cval2; v.cmask = a.cmask;
    v.amin = reinterpret_cast<float *>(sb + l.screen.amin);
    v.amin2 = reinterpret_cast<float *>(sb + l.screen.amin2);
    v.lcount = reinterpret_cast<uint32_t *>(sb + l.screen.lcount);
    v.lists = sb + l.screen.lists;
    v.state = state; v.state2 = state2; v.status = status; v.splits = a.splits; v.most_splits = a.most_splits;
    v.out_bmu = out_bmu; v.out_dist = out_dist; v.out_bmu2 = out_bmu2; v.out_dist2 = out_dist2;
    // ... and with slabs in the order of the norms, in the same room
    OrderedArgs o;
    o.reach = reinterpret_cast<const float2 *>(sb + l.screen.reach);
    v.set_reach = set_reach; v.reach = o.reach;
    v.bound = o.bound = reinterpret_cast<uint32_t *>(sb + l.screen.amin);
    o.lists = v.lists;
    o.count = v.lcount;
    o.items = reinterpret_cast<const uint2 *>(sb + l.screen.items);
    v.units = reinterpret_cast<const int32_t *>(cb + cl.units);
    OrderedImages g;
    g.head = head; g.sets = sets;
    g.set_reach = set_reach; g.reach = o.reach; g.window = a.window; g.bound = o.bound;
    g.items = reinterpret_cast<uint2 *>(sb + l.screen.items);
    v.dense = reinterpret_cast<uint32_t *>(sb + l.screen.cval);         // (after the last launch)
    v.dense_count = status + STATUS_DENSE;
    v.scalars = scalars;
    a.amin = v.amin; a.amin2 = v.amin2;
    // the slabs are dealt to the launches in turn, so that every launch sees the whole map: after
    // the first one a document's smallest value is near its final one and little joins its list
    // (two neighbouring slabs at a time: 134 us instead of 17 for collecting on a trained 75 x 75 map)
    v.launches = launches;
    const int sms = device_sms();
    for (int64_t k = 0; k < launches; ++k) {
        a.n_slabs = (int32_t)((slabs - k + launches - 1) / launches);
        a.first = v.first = k == 0;
        v.launch = k;
        const int64_t slot = shared ? k * cl.chunk_slabs : 0;
        a.img8 = reinterpret_cast<const unsigned char *>(cb + cl.img8) + (size_t)slot * (D + 1) * SC_SLAB;
        a.head_img = reinterpret_cast<const unsigned char *>(cb + cl.head_img) + (size_t)slot * cl.head_pad * SC_SLAB;
        a.normp = reinterpret_cast<const float *>(cb + cl.normp) + slot * SC_SLAB;
        if ((rc = launch_screen_quantize(W, f16, D, M, norms, k, launches, a.n_slabs, slot, head, feat, cb, cl,
                                         scalars, earlier != nullptr, s)))
            return rc;
        if ((rc = launch_sweep_screen(a, o, top2, false, sms, s))) return rc;
        if ((rc = launch_screen_collect(v, top2, s))) return rc;
    }
    // ... and those in the order of the norms, to one launch after the other
    int64_t slab0 = 0;
    for (int64_t k = 0; k < ord_launches; ++k, slab0 += a.n_slabs) {
        a.n_slabs = (int32_t)((slabs - k + launches - 1) / launches);
        const int64_t slot = shared ? k * cl.chunk_slabs : 0;
        a.img8 = reinterpret_cast<const unsigned char *>(cb + cl.ord8) + (size_t)slot * (D + 1) * SC_SLAB;
        a.head_img = reinterpret_cast<const unsigned char *>(cb + cl.ord_head) + (size_t)slot * cl.head_pad * SC_SLAB;
        a.normp = reinterpret_cast<const float *>(cb + cl.ord_normp) + slot * SC_SLAB;
        g.n_slabs = a.n_slabs; g.slab0 = o.slab0 = slab0; g.slot = slot; g.first = k == 0;
        o.tickets = g.tickets = tickets + k * (SC_PARTS + 1);
        o.unit_norm = reinterpret_cast<const float *>(cb + cl.unit_norm) + slab0 * SC_SLAB;
        if ((rc = launch_screen_ordered_images(W, f16, D, M, g, feat, cb, cl, scalars, sms, s))) return rc;
        if ((rc = launch_sweep_screen(a, o, top2, true, sms, s))) return rc;
    }
    if ((rc = launch_screen_verify(v, top2, s))) return rc;
    if (ord_launches && (rc = launch_screen_verify_units(v, top2, sms, s))) return rc;
    return launch_screen_dense(v, top2, sms, s);
}

static int search_impl(const float *W, int64_t D, int64_t M, const float *norms,
                       const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz,
                       int32_t *out_bmu, float *out_dist, const bmu_opts *opts_in, void *ws,
                       size_t ws_bytes, cudaStream_t s, int32_t *out_bmu2 = nullptr,
                       float *out_dist2 = nullptr, int phase = 0, ScreenShared *shared = nullptr)
{
    // phase 0: the whole search; 1: only the tiling pass (bmu_plan_create); 2: everything but
    // the tiling pass, whose results are still in the workspace (bmu_search_planned)
    const bool top2 = out_bmu2 != nullptr || out_dist2 != nullptr;
    int rc = check_sizes(D, M, N, nnz);
    if (rc) return rc;
    bmu_opts o;
    memset(&o, 0, sizeof(o));
    if (opts_in) o = *opts_in;
    if ((rc = check_opts(o))) return rc;
    if (N == 0) return BMU_OK;
    if (!rowptr || (nnz > 0 && !colidx) ||
        (phase != 1 && (!W || !out_bmu || !out_dist || (top2 && (!out_bmu2 || !out_dist2))))) {
        set_error("null pointer argument");
        return BMU_ERR_INVALID_ARG;
    }
    // a plan is made before the codebook is known: it assumes the aligned fast path, and the
    // search that uses it insists on it
    const uintptr_t w_addr = phase == 1 ? 0 : reinterpret_cast<uintptr_t>(W);
    if (phase == 2 && (w_addr & 15) != 0) {
        set_error("a planned search needs W 16-byte aligned");
        return BMU_ERR_UNSUPPORTED;
    }
    if (M == 0 || D == 0) {
        set_error("empty codebook (D=%lld, M=%lld): no neuron to return", (long long)D, (long long)M);
        return BMU_ERR_INVALID_ARG;
    }
    const int head = screen_wanted(o, D, M, N, nnz) ? screen_head_rows(o, D) : mma_head_rows(o, D);
    const size_t repack_bytes = mma_repack_bytes(o, D, M, N, nnz, top2);
    const Layout l = layout_of(o, D, M, N, nnz, top2, phase != 0);
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255) != 0 || ws_bytes < l.total) {
        set_error("workspace missing, not 256-byte aligned, or smaller than %zu bytes", l.total);
        return BMU_ERR_WORKSPACE;
    }
    char *base = static_cast<char *>(ws);
    u64 *state = reinterpret_cast<u64 *>(base + l.state_off);
    u64 *state2 = top2 ? reinterpret_cast<u64 *>(base + l.state2_off) : nullptr;
    if (!norms && phase != 1) {
        float *n = reinterpret_cast<float *>(base + l.norms_off);
        if ((rc = launch_norms(W, D, M, n, s))) return rc;
        norms = n;
    }
    uint32_t *status = reinterpret_cast<uint32_t *>(base + l.status_off);
    Route r;
    if ((rc = route_search(o, D, M, N, nnz, w_addr, r))) return rc;
    if (r.few && phase != 1) {
        BMU_CUDA(cudaMemsetAsync(status, 0, l.slots_off, s));        // and the tickets behind it
        FewArgs a;
        a.W = W; a.D = D; a.M = M; a.N = N; a.norms = norms; a.rowptr = rowptr; a.colidx = colidx;
        a.slots = reinterpret_cast<u64 *>(base + l.slots_off);
        a.tickets = reinterpret_cast<uint32_t *>(base + l.tickets_off);
        a.status = status;
        a.out_bmu = out_bmu; a.out_dist = out_dist; a.out_bmu2 = out_bmu2; a.out_dist2 = out_dist2;
        return launch_sweep_few(a, top2, device_sms(), s);
    }
    BMU_CUDA(cudaMemsetAsync(status, 0, l.tickets_off, s));          // and the counters behind it
    const bool mma = r.kernel == 6, tiled = r.kernel == 4, planned = r.kernel == 3;
    char *pw = base + l.plan_off;
    // dense head = the most frequent features by the corpus's own counts (bmu_opts.relabel)
    const int relabel = mma ? o.relabel : 2;        // 0 decide from the counts, 1 always, 2 never
    if ((planned || tiled || mma) && !r.two_stage && phase != 2)
        if ((rc = launch_plan(rowptr, colidx, N, nnz, plan_order(o, mma),
                              mma ? head : 0, relabel, D, pw, l.plan, status, s)))
            return rc;
    if (r.two_stage) {
        if (phase != 2 && (rc = launch_plan_screen(rowptr, colidx, N, nnz, screen_by_content(o, M, nnz, phase == 1),
                                                   head, relabel, D, pw, l.plan,
                                                   reinterpret_cast<uint32_t *>(base + l.count_off),
                                                   screen_rank(l, base, shared), screen_feat(l, base, shared),
                                                   shared && shared->used, status, s)))
            return rc;
        if (phase == 1) return BMU_OK;
        return screen_search(W, 0, D, M, norms, rowptr, colidx, N, head, relabel, l, base, status, state,
                             state2, out_bmu, out_dist, out_bmu2, out_dist2, shared, s);
    }
    if (mma) {
        if (phase != 2 &&
            (rc = launch_plan_tiles(rowptr, N, o.tile_order == 2, head, relabel, D, pw, l.plan, status, s)))
            return rc;
        if (phase == 1) return BMU_OK;
        const int64_t m_full = r.m_full;
        uint32_t *head_max = status + 16;
        unsigned char *img = reinterpret_cast<unsigned char *>(base + l.head_off);
        const uint16_t *feat = (relabel != 2 && l.plan.fsort_tmp_bytes > 0)
                                   ? reinterpret_cast<const uint16_t *>(pw + l.plan.feat_off) : nullptr;
        if ((rc = launch_head_split2(W, M, m_full, head, feat, head_max, img, s))) return rc;
        MmaArgs a;
        a.W = W; a.M = M; a.N = N; a.n_tiles = (N + 7) / 8; a.norms = norms;
        a.perm = reinterpret_cast<const int32_t *>(pw + l.plan.perm_off);
        a.tile_len = reinterpret_cast<const uint32_t *>(pw + l.plan.tilelen_off);
        a.tile_off = reinterpret_cast<const uint32_t *>(pw + l.plan.tileoff_off);
        a.tile_ids = reinterpret_cast<const uint4 *>(pw + l.plan.tileids_off);
        a.tile_head = reinterpret_cast<const uint32_t *>(pw + l.plan.tilehead_off);
        a.head_max = head_max; a.head = head; a.f16 = 0;
        a.state = state; a.state2 = state2; a.status = status;
        a.D = D; a.tile_rows_cap = l.plan.tile_rows_cap;
        const int64_t chunk = r.chunk;
        float *compact = repack_bytes ? reinterpret_cast<float *>(base + l.repack_off) : nullptr;
        const LaunchCuts cuts(m_full, chunk);
        for (int64_t k = 0; k < cuts.n; ++k) {
            const int64_t j = cuts.cut(k);
            a.j_lo = (int32_t)j;
            a.j_hi = (int32_t)cuts.cut(k + 1);
            a.first = j == 0;
            a.W = W; a.M = M;
            if (compact) {                 // gather from a compact copy of this chunk's columns
                const int32_t width = a.j_hi - a.j_lo;
                { repack_chunk_kernel<<<(unsigned)D, 256, 0, s>>>(
                    reinterpret_cast<const char *>(W), M * 4, j * 4, width * 4,
                    reinterpret_cast<char *>(compact)); BMU_LAUNCHED(); }
                a.W = reinterpret_cast<const float *>(reinterpret_cast<uintptr_t>(compact) -
                                                      (uintptr_t)j * sizeof(float));
                a.M = width;
            }
            // the image takes 4 * head bytes per neuron, slab after slab
            a.head_img = img + (size_t)j * head * 4;
            if ((rc = launch_sweep_mma2(a, o, s))) return rc;
        }
        if (m_full < M) {                      // ragged last slab: generic kernel, merged in
            SweepArgs g;
            g.W = W; g.D = D; g.M = M; g.norms = norms; g.rowptr = rowptr; g.colidx = colidx;
            g.N = N; g.state = state; g.state2 = state2; g.status = status; g.j_lo = (int32_t)m_full;
            g.j_hi = (int32_t)M; g.first = 0;
            bmu_opts go;
            memset(&go, 0, sizeof(go));
            if ((rc = launch_sweep_direct(g, go, s))) return rc;
        }
        return launch_finalize(state, state2, rowptr, N, out_bmu, out_dist, out_bmu2, out_dist2, s);
    }
    if (tiled) {
        const int head = (o.tile_head == 1 || D < TILE_HEAD_ROWS) ? 0 : TILE_HEAD_ROWS;
        if (phase != 2 &&
            (rc = launch_plan_tiles(rowptr, N, o.tile_order != 1, head, 2, D, pw, l.plan, status, s))) return rc;
        if (phase == 1) return BMU_OK;
        TileArgs a;
        a.W = W; a.M = M; a.N = N; a.n_tiles = (N + 7) / 8; a.norms = norms;
        a.perm = reinterpret_cast<const int32_t *>(pw + l.plan.perm_off);
        a.tile_len = reinterpret_cast<const uint32_t *>(pw + l.plan.tilelen_off);
        a.tile_off = reinterpret_cast<const uint32_t *>(pw + l.plan.tileoff_off);
        a.tile_ids = reinterpret_cast<const uint4 *>(pw + l.plan.tileids_off);
        a.tile_head = reinterpret_cast<const uint32_t *>(pw + l.plan.tilehead_off);
        a.head_rows = head;
        a.state = state; a.state2 = state2; a.status = status;
        a.D = D; a.tile_rows_cap = l.plan.tile_rows_cap;
        const int64_t chunk = r.chunk, m_full = r.m_full;
        for (int64_t j = 0; j < m_full; j += chunk) {
            a.j_lo = (int32_t)j;
            a.j_hi = (int32_t)(j + chunk < m_full ? j + chunk : m_full);
            a.first = j == 0;
            if ((rc = launch_sweep_tiles(a, o, s))) return rc;
        }
        if (m_full < M) {                      // ragged last slab: generic kernel, merged in
            SweepArgs g;
            g.W = W; g.D = D; g.M = M; g.norms = norms; g.rowptr = rowptr; g.colidx = colidx;
            g.N = N; g.state = state; g.state2 = state2; g.status = status; g.j_lo = (int32_t)m_full;
            g.j_hi = (int32_t)M; g.first = 0;
            bmu_opts go;
            memset(&go, 0, sizeof(go));
            if ((rc = launch_sweep_direct(g, go, s))) return rc;
        }
        return launch_finalize(state, state2, rowptr, N, out_bmu, out_dist, out_bmu2, out_dist2, s);
    }
    if (phase == 1) return BMU_OK;           // nothing more to prepare for the other kernels
    if (planned) {
        const int slab = rows_slab_width(o);
        RowsArgs a;
        a.W = W; a.M = M; a.N = N; a.norms = norms; a.rowptr = rowptr;
        a.perm = reinterpret_cast<const int32_t *>(pw + l.plan.perm_off);
        a.doc_off = reinterpret_cast<const uint32_t *>(pw + l.plan.docoff_off);
        a.ids = reinterpret_cast<const uint4 *>(pw + l.plan.ids_off);
        a.state = state; a.state2 = state2; a.status = status;
        a.D = D; a.id_groups_cap = l.plan.id_groups_cap;
        const int64_t chunk = r.chunk, m_full = r.m_full;
        for (int64_t j = 0; j < m_full; j += chunk) {
            a.j_lo = (int32_t)j;
            a.j_hi = (int32_t)(j + chunk < m_full ? j + chunk : m_full);
            a.first = j == 0;
            if ((rc = launch_sweep_rows(a, o, s))) return rc;
        }
        if (m_full < M) {                      // ragged last slab: generic kernel, merged in
            SweepArgs g;
            g.W = W; g.D = D; g.M = M; g.norms = norms; g.rowptr = rowptr; g.colidx = colidx;
            g.N = N; g.state = state; g.state2 = state2; g.status = status; g.j_lo = (int32_t)m_full; g.j_hi = (int32_t)M; g.first = 0;
            bmu_opts go;
            memset(&go, 0, sizeof(go));
            if ((rc = launch_sweep_direct(g, go, s))) return rc;
        }
        return launch_finalize(state, state2, rowptr, N, out_bmu, out_dist, out_bmu2, out_dist2, s);
    }
    if (o.warps == 4) { set_error("generic kernel: warps must be 8, 16 or 32"); return BMU_ERR_INVALID_ARG; }
    const int64_t chunk = r.chunk;
    SweepArgs a;
    a.W = W; a.D = D; a.M = M; a.norms = norms; a.rowptr = rowptr; a.colidx = colidx;
    a.N = N; a.state = state; a.state2 = state2; a.status = status;
    for (int64_t j = 0; j < M; j += chunk) {
        a.j_lo = (int32_t)j;
        a.j_hi = (int32_t)(j + chunk < M ? j + chunk : M);
        a.first = j == 0;
        if ((rc = launch_sweep_direct(a, o, s))) return rc;
    }
    return launch_finalize(state, state2, rowptr, N, out_bmu, out_dist, out_bmu2, out_dist2, s);
}

// ---- library-owned grow-only scratch (one per device) ----------------------
struct Scratch { void *p; size_t bytes; };
static Scratch g_scratch[64];
static std::mutex g_mu;

static int scratch_get(size_t bytes, void **out)
{
    int dev = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) { set_error("device ordinal %d out of range", dev); return BMU_ERR_UNSUPPORTED; }
    std::lock_guard<std::mutex> g(g_mu);
    Scratch &sc = g_scratch[dev];
    if (sc.bytes < bytes) {
        if (sc.p) {
            BMU_CUDA(cudaDeviceSynchronize());
            BMU_CUDA(cudaFree(sc.p));
            sc.p = nullptr; sc.bytes = 0;
        }
        const size_t want = align_up(bytes + bytes / 8, (size_t)1 << 20);
        BMU_CUDA(cudaMalloc(&sc.p, want));
        sc.bytes = want;
    }
    *out = sc.p;
    return BMU_OK;
}

// what a non-zero status word means, for the host entry points that read it back
static int status_error(uint32_t status)
{
    if (status & PLAN_STATUS_OVERFLOW) {
        set_error("the tiling pass found an offset beyond its reserved room (status word %u); "
                  "results are invalid", status);
        return BMU_ERR_WORKSPACE;
    }
    set_error("a bounded device-side wait ran out (status word %u); results are invalid", status);
    return BMU_ERR_TIMEOUT;
}

// ORs the status word of one search into a word that outlives the next search's clearing
__global__ void status_accumulate_kernel(const uint32_t *__restrict__ status,
                                         uint32_t *__restrict__ sticky)
{
    if (*status) atomicOr(sticky, *status);
}

// ---- CSR validation ---------------------------------------------------------
__global__ void validate_kernel(const int32_t *__restrict__ rowptr,
                                const int32_t *__restrict__ colidx, int64_t N, int64_t nnz,
                                int64_t D, int32_t *__restrict__ flags)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (t == 0) {
        if (rowptr[0] != 0) atomicOr(flags, 1);
        if ((int64_t)rowptr[N] != nnz) atomicOr(flags, 2);
    }
    for (int64_t i = t; i < N; i += stride) {
        if (rowptr[i + 1] < rowptr[i]) atomicOr(flags, 4);
        if ((int64_t)rowptr[i + 1] - rowptr[i] > 65535) atomicOr(flags, 16);
    }
    for (int64_t e = t; e < nnz; e += stride) {
        const int32_t f = colidx[e];
        if (f < 0 || (int64_t)f >= D) atomicOr(flags, 8);
    }
}

int launch_validate_csr(const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz,
                        int64_t D, int32_t *flags, cudaStream_t s)
{
    BMU_CUDA(cudaMemsetAsync(flags, 0, sizeof(int32_t), s));
    { validate_kernel<<<296, 256, 0, s>>>(rowptr, colidx, N, nnz, D, flags); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

}  // namespace bmu

using namespace bmu;

extern "C" {

const char *bmu_status_string(int status)
{
    switch (status) {
    case BMU_OK: return "ok";
    case BMU_ERR_INVALID_ARG: return "invalid argument";
    case BMU_ERR_UNSUPPORTED: return "unsupported size or option";
    case BMU_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case BMU_ERR_CUDA: return "CUDA runtime error";
    case BMU_ERR_TIMEOUT: return "device-side wait timed out";
    default: return "unknown status";
    }
}

const char *bmu_last_error(void) { return g_err; }

int bmu_version(void) { return 200; }

uint64_t bmu_kernel_launches(void) { return g_kernel_launches; }

int bmu_describe_search(int64_t D, int64_t M, int64_t N, int64_t nnz, const bmu_opts *opts,
                        bmu_search_desc *out)
{
    if (!out) { set_error("null pointer argument"); return BMU_ERR_INVALID_ARG; }
    memset(out, 0, sizeof(*out));
    int rc = check_sizes(D, M, N, nnz);
    if (rc) return rc;
    bmu_opts o;
    memset(&o, 0, sizeof(o));
    if (opts) o = *opts;
    if ((rc = check_opts(o))) return rc;
    if (M == 0 || D == 0) { set_error("empty codebook"); return BMU_ERR_INVALID_ARG; }
    Route r;
    if ((rc = route_search(o, D, M, N, nnz, 0, r))) return rc;
    out->kernel = r.kernel;
    out->head_rows = r.head;
    out->slab = r.slab;
    out->docs_per_block = r.docs_per_block;
    out->repack = r.repack;
    out->two_stage = r.two_stage;
    if (r.few) {                         // the generic sums, every piece of the neuron axis in one launch
        out->kernel = 1;
        out->slab = 128;
        out->docs_per_block = 4;
        out->chunk_neurons = M;
        out->sweep_launches = 1;
        out->ragged_neurons = 0;
        return BMU_OK;
    }
    out->chunk_neurons = r.chunk;
    out->sweep_launches = (int32_t)((r.m_full + r.chunk - 1) / r.chunk);
    out->ragged_neurons = (int32_t)(M - r.m_full);
    return BMU_OK;
}

int bmu_codebook_norms(const float *W, int64_t D, int64_t M, float *norms, void *stream)
{
    int rc = check_sizes(D, M, 0, 0);
    if (rc) return rc;
    if (M == 0) return BMU_OK;
    if (!norms || (D > 0 && !W)) { set_error("null pointer argument"); return BMU_ERR_INVALID_ARG; }
    return launch_norms(W, D, M, norms, static_cast<cudaStream_t>(stream));
}

size_t bmu_search_workspace_bytes(int64_t D, int64_t M, int64_t N, int64_t nnz,
                                  const bmu_opts *opts)
{
    if (D < 0 || M < 0 || N < 0 || nnz < 0) return 0;
    bmu_opts o;
    memset(&o, 0, sizeof(o));
    if (opts) o = *opts;
    return query_bytes(o, D, M, N, nnz, false, false);
}

int bmu_search_ws(const float *W, int64_t D, int64_t M, const float *norms,
                  const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz,
                  int32_t *out_bmu, float *out_dist, const bmu_opts *opts, void *workspace,
                  size_t workspace_bytes, void *stream)
{
    return search_impl(W, D, M, norms, rowptr, colidx, N, nnz, out_bmu, out_dist, opts,
                       workspace, workspace_bytes, static_cast<cudaStream_t>(stream));
}

size_t bmu_search_top2_workspace_bytes(int64_t D, int64_t M, int64_t N, int64_t nnz,
                                       const bmu_opts *opts)
{
    if (D < 0 || M < 0 || N < 0 || nnz < 0) return 0;
    bmu_opts o;
    memset(&o, 0, sizeof(o));
    if (opts) o = *opts;
    return query_bytes(o, D, M, N, nnz, true, false);
}

int bmu_search_top2_ws(const float *W, int64_t D, int64_t M, const float *norms,
                       const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz,
                       int32_t *out_bmu, float *out_dist, int32_t *out_bmu2, float *out_dist2,
                       const bmu_opts *opts, void *workspace, size_t workspace_bytes,
                       void *stream)
{
    if (N > 0 && (!out_bmu2 || !out_dist2)) {
        set_error("null pointer argument");
        return BMU_ERR_INVALID_ARG;
    }
    return search_impl(W, D, M, norms, rowptr, colidx, N, nnz, out_bmu, out_dist, opts, workspace,
                       workspace_bytes, static_cast<cudaStream_t>(stream), out_bmu2, out_dist2);
}

int bmu_codebook_norms_f16(const void *W16, int64_t D, int64_t M, float *norms, void *stream)
{
    int rc = check_sizes(D, M, 0, 0);
    if (rc) return rc;
    if (M == 0) return BMU_OK;
    if (!norms || (D > 0 && !W16)) { set_error("null pointer argument"); return BMU_ERR_INVALID_ARG; }
    if (M % 8 != 0 || (reinterpret_cast<uintptr_t>(W16) & 15) != 0) {
        set_error("half-precision codebook needs M %% 8 == 0 and 16-byte alignment");
        return BMU_ERR_UNSUPPORTED;
    }
    return launch_norms_f16(W16, D, M, norms, static_cast<cudaStream_t>(stream));
}

// Which kernel a half-precision search takes: large sweeps the wide tensor-core sweep (whole
// 256-neuron slabs only), the rest the planned kernel.  `ow` = the options of the wide sweep, its
// head resolved (576 by default: with 2-byte rows the gathered tail is cheap, so the balance
// point sits lower than the fp32 sweep's 640; config 4 at full length: 2364 / 2348 / 2331 / 2473
// ms per step at 448 / 512 / 576 / 704).
static bool f16_route(const bmu_opts &o, int64_t D, int64_t M, int64_t nnz, bmu_opts &ow, bool &wide)
{
    ow = o;
    ow.kernel = 6;
    if (!ow.head_rows) {
        const int64_t cap = D / 64 * 64;
        ow.head_rows = (int32_t)(cap < 576 ? (cap < 64 ? 64 : cap) : 576);
    }
    const bool wide_ok = M % MMA_SLAB == 0 && D >= ow.head_rows && o.cluster != 2;
    wide = wide_ok && (o.kernel == 6 || (o.kernel == 0 && (double)nnz * (double)M >= 2e10));
    return wide_ok;
}

static Layout f16_wide_layout(const bmu_opts &ow, int64_t D, int64_t M, int64_t N, int64_t nnz, bool top2)
{
    return layout_for(D, M, N, nnz, 6, top2, mma_head_rows(ow, D), mma_repack_bytes(ow, D, M, N, nnz, top2),
                      plan_order(ow, true));
}

size_t bmu_search_f16_workspace_bytes(int64_t D, int64_t M, int64_t N, int64_t nnz,
                                      const bmu_opts *opts)
{
    if (D < 0 || M < 0 || N < 0 || nnz < 0) return 0;
    bmu_opts o, ow;
    memset(&o, 0, sizeof(o));
    if (opts) o = *opts;
    bool wide = false;
    f16_route(o, D, M, nnz, ow, wide);
    // (as query_bytes: for every way that these or smaller sizes may take)
    size_t need = layout_for(D, M, N, nnz, 3, true).total;
    auto room = [&](const Layout &l) { if (l.total > need) need = l.total; };
    if (wide) room(f16_wide_layout(ow, D, M, N, nnz, true));
    if (screen_within(o, D, M, N, nnz, true)) room(screen_layout_of(o, D, M, N, nnz, true));
    return need;
}

int bmu_search_f16_ws(const void *W16, int64_t D, int64_t M, const float *norms,
                      const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz,
                      int32_t *out_bmu, float *out_dist, int32_t *out_bmu2, float *out_dist2,
                      const bmu_opts *opts, void *ws, size_t ws_bytes, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = check_sizes(D, M, N, nnz);
    if (rc) return rc;
    bmu_opts o;
    memset(&o, 0, sizeof(o));
    if (opts) o = *opts;
    if ((rc = check_opts(o))) return rc;
    if (N == 0) return BMU_OK;
    const bool top2 = out_bmu2 != nullptr || out_dist2 != nullptr;
    if (!W16 || !rowptr || !out_bmu || !out_dist || (nnz > 0 && !colidx) ||
        (top2 && (!out_bmu2 || !out_dist2))) {
        set_error("null pointer argument");
        return BMU_ERR_INVALID_ARG;
    }
    if (M % 256 != 0 || D < 1 || D > LANES_MAX_D || (reinterpret_cast<uintptr_t>(W16) & 15) != 0 ||
        (o.kernel != 0 && o.kernel != 3 && o.kernel != 6)) {
        set_error("half-precision search needs M %% 256 == 0, 1 <= D <= %d, 16-byte alignment and "
                  "the planned (3) or the wide tensor-core (6) kernel", LANES_MAX_D);
        return BMU_ERR_UNSUPPORTED;
    }
    if (screen_wanted(o, D, M, N, nnz, true)) {
        const Layout l = screen_layout_of(o, D, M, N, nnz, top2);
        if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255) != 0 || ws_bytes < l.total) {
            set_error("workspace missing, not 256-byte aligned, or smaller than %zu bytes", l.total);
            return BMU_ERR_WORKSPACE;
        }
        char *base = static_cast<char *>(ws), *pw = base + l.plan_off;
        u64 *state = reinterpret_cast<u64 *>(base + l.state_off);
        u64 *state2 = top2 ? reinterpret_cast<u64 *>(base + l.state2_off) : nullptr;
        uint32_t *status = reinterpret_cast<uint32_t *>(base + l.status_off);
        if (!norms) {
            float *n = reinterpret_cast<float *>(base + l.norms_off);
            if ((rc = launch_norms_f16(W16, D, M, n, s))) return rc;
            norms = n;
        }
        const int head = screen_head_rows(o, D);
        BMU_CUDA(cudaMemsetAsync(status, 0, l.tickets_off, s));      // and the counters behind it
        if ((rc = launch_plan_screen(rowptr, colidx, N, nnz, screen_by_content(o, M, nnz, false), head, o.relabel, D,
                                     pw, l.plan, reinterpret_cast<uint32_t *>(base + l.count_off),
                                     screen_rank(l, base, nullptr), screen_feat(l, base, nullptr), false, status, s)))
            return rc;
        return screen_search(W16, 1, D, M, norms, rowptr, colidx, N, head, o.relabel, l, base, status, state,
                             state2, out_bmu, out_dist, out_bmu2, out_dist2, nullptr, s);
    }
    if (o.two_stage == 1) {
        set_error("the two-stage sweep needs kernel 0 or 6, length-ordered documents (cluster != 2) and "
                  "head_rows <= %d", SC_MAX_HEAD);
        return BMU_ERR_UNSUPPORTED;
    }
    bmu_opts ow;
    bool wide = false;
    const bool wide_ok = f16_route(o, D, M, nnz, ow, wide);
    const int head = ow.head_rows;
    if (o.kernel == 6 && !wide_ok) {
        set_error("half-precision tensor-core sweep needs M %% %d == 0, D >= %d and length-ordered "
                  "documents", MMA_SLAB, head);
        return BMU_ERR_UNSUPPORTED;
    }
    const Layout l = wide ? f16_wide_layout(ow, D, M, N, nnz, top2) : layout_for(D, M, N, nnz, 3, top2);
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255) != 0 || ws_bytes < l.total) {
        set_error("workspace missing, not 256-byte aligned, or smaller than %zu bytes", l.total);
        return BMU_ERR_WORKSPACE;
    }
    char *base = static_cast<char *>(ws);
    u64 *state = reinterpret_cast<u64 *>(base + l.state_off);
    u64 *state2 = top2 ? reinterpret_cast<u64 *>(base + l.state2_off) : nullptr;
    if (!norms) {
        float *n = reinterpret_cast<float *>(base + l.norms_off);
        if ((rc = launch_norms_f16(W16, D, M, n, s))) return rc;
        norms = n;
    }
    if (wide) {
        uint32_t *status = reinterpret_cast<uint32_t *>(base + l.status_off);
        BMU_CUDA(cudaMemsetAsync(status, 0, 256, s));
        char *pw = base + l.plan_off;
        const int relabel = o.relabel;
        if ((rc = launch_plan(rowptr, colidx, N, nnz, plan_order(o, true), head, relabel, D, pw, l.plan,
                              status, s))) return rc;
        if ((rc = launch_plan_tiles(rowptr, N, o.tile_order == 2, head, relabel, D, pw, l.plan, status, s))) return rc;
        unsigned char *img = reinterpret_cast<unsigned char *>(base + l.head_off);
        const uint16_t *feat = (relabel != 2 && l.plan.fsort_tmp_bytes > 0)
                                   ? reinterpret_cast<const uint16_t *>(pw + l.plan.feat_off) : nullptr;
        if ((rc = launch_head_split2_f16(W16, M, M, head, feat, img, s))) return rc;
        MmaArgs a;
        a.W = static_cast<const float *>(W16); a.M = M; a.N = N; a.n_tiles = (N + 7) / 8; a.norms = norms;
        a.perm = reinterpret_cast<const int32_t *>(pw + l.plan.perm_off);
        a.tile_len = reinterpret_cast<const uint32_t *>(pw + l.plan.tilelen_off);
        a.tile_off = reinterpret_cast<const uint32_t *>(pw + l.plan.tileoff_off);
        a.tile_ids = reinterpret_cast<const uint4 *>(pw + l.plan.tileids_off);
        a.tile_head = reinterpret_cast<const uint32_t *>(pw + l.plan.tilehead_off);
        a.head_max = status + 16; a.head = head; a.f16 = 1;
        a.state = state; a.state2 = state2; a.status = status;
        a.D = D; a.tile_rows_cap = l.plan.tile_rows_cap;
        // twice the neurons per L2-resident chunk: the rows are half as wide
        const int64_t chunk = o.chunk_neurons ? mma_chunk(o, D, M) : 2 * mma_auto_chunk(D, M);
        const size_t repack_bytes = mma_repack_bytes(ow, D, M, N, nnz, top2);
        char *compact = (repack_bytes && M > chunk) ? base + l.repack_off : nullptr;
        const LaunchCuts cuts(M, chunk);
        for (int64_t k = 0; k < cuts.n; ++k) {
            const int64_t j = cuts.cut(k);
            a.j_lo = (int32_t)j;
            a.j_hi = (int32_t)cuts.cut(k + 1);
            a.first = j == 0;
            a.W = static_cast<const float *>(W16); a.M = M;
            if (compact) {                 // a compact copy of this chunk's columns (2 bytes each)
                const int32_t width = a.j_hi - a.j_lo;
                { repack_chunk_kernel<<<(unsigned)D, 256, 0, s>>>(static_cast<const char *>(W16), M * 2,
                                                              j * 2, width * 2, compact); BMU_LAUNCHED(); }
                a.W = reinterpret_cast<const float *>(reinterpret_cast<uintptr_t>(compact) -
                                                      (uintptr_t)j * 2);
                a.M = width;
            }
            a.head_img = img + (size_t)j * head * 2;     // one part: 2 * head bytes per neuron
            if ((rc = launch_sweep_mma2_f16(a, o, s))) return rc;
        }
        return launch_finalize(state, state2, rowptr, N, out_bmu, out_dist, out_bmu2, out_dist2, s);
    }
    uint32_t *status = reinterpret_cast<uint32_t *>(base + l.status_off);
    BMU_CUDA(cudaMemsetAsync(status, 0, 256, s));
    char *pw = base + l.plan_off;
    if ((rc = launch_plan(rowptr, colidx, N, nnz, o.cluster != 2, 0, 2, D, pw, l.plan, status, s))) return rc;
    RowsArgs a;
    a.status = status; a.D = D; a.id_groups_cap = l.plan.id_groups_cap;
    a.W = static_cast<const float *>(W16); a.M = M; a.N = N; a.norms = norms; a.rowptr = rowptr;
    a.perm = reinterpret_cast<const int32_t *>(pw + l.plan.perm_off);
    a.doc_off = reinterpret_cast<const uint32_t *>(pw + l.plan.docoff_off);
    a.ids = reinterpret_cast<const uint4 *>(pw + l.plan.ids_off);
    a.state = state; a.state2 = state2;
    // twice the neurons per L2-resident chunk: the rows are half as wide
    const int64_t chunk = o.chunk_neurons ? (o.chunk_neurons + 255) / 256 * 256
                                          : auto_chunk(D, M, 256) * 2;
    for (int64_t j = 0; j < M; j += chunk) {
        a.j_lo = (int32_t)j;
        a.j_hi = (int32_t)(j + chunk < M ? j + chunk : M);
        a.first = j == 0;
        if ((rc = launch_sweep_rows_f16(a, o, s))) return rc;
    }
    return launch_finalize(state, state2, rowptr, N, out_bmu, out_dist, out_bmu2, out_dist2, s);
}

int bmu_search(const float *W, int64_t D, int64_t M, const int32_t *rowptr,
               const int32_t *colidx, int64_t N, int32_t *out_bmu, float *out_dist,
               void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = check_sizes(D, M, N, 0);
    if (rc) return rc;
    if (N == 0) return BMU_OK;
    if (!rowptr) { set_error("null pointer argument"); return BMU_ERR_INVALID_ARG; }
    bmu_opts none;
    memset(&none, 0, sizeof(none));
    int32_t nnz = 0;
    // Few documents need no scratch by the listing.  Read back all the same where the few-documents kernel
    // takes more than half a millisecond even for short lists and long ones would go another way (10 us;
    // not while the stream is captured).
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (N < FEW_MAX_DOCS && N * M >= ONE_SHOT_READS) BMU_CUDA(cudaStreamIsCapturing(s, &capture));
    if (N >= FEW_MAX_DOCS || !colidx || (N * M >= ONE_SHOT_READS && capture == cudaStreamCaptureStatusNone)) {
        BMU_CUDA(cudaMemcpyAsync(&nnz, rowptr + N, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        BMU_CUDA(cudaStreamSynchronize(s));
    }
    const size_t need = layout_of(none, D, M, N, nnz, false).total;
    void *ws = nullptr;
    if ((rc = scratch_get(need, &ws))) return rc;
    return search_impl(W, D, M, nullptr, rowptr, colidx, N, nnz, out_bmu, out_dist, nullptr, ws,
                       need, s);
}

int bmu_search_host(const float *W, int64_t D, int64_t M, const int32_t *rowptr_host,
                    const int32_t *colidx_host, int64_t N, int32_t *out_bmu_host,
                    float *out_dist_host, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = check_sizes(D, M, N, 0);
    if (rc) return rc;
    if (N == 0) return BMU_OK;
    if (!rowptr_host || !out_bmu_host || !out_dist_host) {
        set_error("null pointer argument");
        return BMU_ERR_INVALID_ARG;
    }
    const int64_t nnz = rowptr_host[N];
    if (nnz < 0 || (nnz > 0 && !colidx_host)) { set_error("bad rowptr[N] or null colidx"); return BMU_ERR_INVALID_ARG; }
    const size_t ws_need = bmu_search_workspace_bytes(D, M, N, nnz, nullptr);
    const size_t rp_off = align_up(ws_need, 256);
    const size_t ci_off = align_up(rp_off + (size_t)(N + 1) * 4, 256);
    const size_t ob_off = align_up(ci_off + (size_t)nnz * 4, 256);
    const size_t od_off = align_up(ob_off + (size_t)N * 4, 256);
    const size_t total = align_up(od_off + (size_t)N * 4, 256);
    void *p = nullptr;
    if ((rc = scratch_get(total, &p))) return rc;
    char *b = static_cast<char *>(p);
    int32_t *rp = reinterpret_cast<int32_t *>(b + rp_off);
    int32_t *ci = reinterpret_cast<int32_t *>(b + ci_off);
    int32_t *ob = reinterpret_cast<int32_t *>(b + ob_off);
    float *od = reinterpret_cast<float *>(b + od_off);
    BMU_CUDA(cudaMemcpyAsync(rp, rowptr_host, (size_t)(N + 1) * 4, cudaMemcpyHostToDevice, s));
    if (nnz)
        BMU_CUDA(cudaMemcpyAsync(ci, colidx_host, (size_t)nnz * 4, cudaMemcpyHostToDevice, s));
    if ((rc = search_impl(W, D, M, nullptr, rp, ci, N, nnz, ob, od, nullptr, b, ws_need, s)))
        return rc;
    BMU_CUDA(cudaMemcpyAsync(out_bmu_host, ob, (size_t)N * 4, cudaMemcpyDeviceToHost, s));
    BMU_CUDA(cudaMemcpyAsync(out_dist_host, od, (size_t)N * 4, cudaMemcpyDeviceToHost, s));
    uint32_t status = 0;                               // first word of the workspace
    BMU_CUDA(cudaMemcpyAsync(&status, b, sizeof(status), cudaMemcpyDeviceToHost, s));
    BMU_CUDA(cudaStreamSynchronize(s));
    if (status) return status_error(status);
    return BMU_OK;
}

// The batches of one call share the 8-bit images of the codebook up to this size (a quarter of its own, and
// the head's); those of slabs in the order of the norms come on top: as many where the map takes one launch, half where it takes
// two, a quarter from four on, as at this limit.  The scratch keeps them until bmu_release_scratch.  150,000 documents
// in three batches to 128 x 128 units: 9.10 ms with ranges, head and images made for each batch, 8.2 shared.
static const size_t SHARED_IMAGE_MAX = (size_t)2 << 30;

// ---- streamed batches from host memory (config 5: a corpus fed in batches) ----
// Two staging buffers; the copy stream uploads batch k+1 and downloads the results
// of batch k-1 while the caller's stream searches batch k.
struct StreamCtx { cudaStream_t copy; cudaEvent_t h2d[2], done[2], d2h[2]; bool ready; };
static StreamCtx g_stream_ctx[64];

static int stream_ctx_get(int dev, StreamCtx **out)
{
    StreamCtx &c = g_stream_ctx[dev];
    if (!c.ready) {
        BMU_CUDA(cudaStreamCreateWithFlags(&c.copy, cudaStreamNonBlocking));
        for (int i = 0; i < 2; ++i) {
            BMU_CUDA(cudaEventCreateWithFlags(&c.h2d[i], cudaEventDisableTiming));
            BMU_CUDA(cudaEventCreateWithFlags(&c.done[i], cudaEventDisableTiming));
            BMU_CUDA(cudaEventCreateWithFlags(&c.d2h[i], cudaEventDisableTiming));
        }
        c.ready = true;
    }
    *out = &c;
    return BMU_OK;
}

int bmu_search_batches_host(const float *W, int64_t D, int64_t M, int32_t n_batches,
                            const int32_t *const *rowptr_host, const int32_t *const *colidx_host,
                            const int64_t *N, int32_t *const *out_bmu_host,
                            float *const *out_dist_host, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (n_batches < 0 || (n_batches > 0 && (!rowptr_host || !colidx_host || !N || !out_bmu_host ||
                                            !out_dist_host))) {
        set_error("null pointer argument or negative batch count");
        return BMU_ERR_INVALID_ARG;
    }
    int rc;
    int64_t max_n = 0, max_nnz = 0;
    for (int k = 0; k < n_batches; ++k) {
        if (N[k] < 0 || (N[k] > 0 && (!rowptr_host[k] || !out_bmu_host[k] || !out_dist_host[k]))) {
            set_error("batch %d: null pointer or negative size", k);
            return BMU_ERR_INVALID_ARG;
        }
        const int64_t nnz = N[k] > 0 ? rowptr_host[k][N[k]] : 0;
        if ((rc = check_sizes(D, M, N[k], nnz))) return rc;
        if (nnz > 0 && !colidx_host[k]) { set_error("batch %d: null colidx", k); return BMU_ERR_INVALID_ARG; }
        if (N[k] > max_n) max_n = N[k];
        if (nnz > max_nnz) max_nnz = nnz;
    }
    if (max_n == 0) return BMU_OK;
    // layout: status word of the whole call, shared norms | per buffer: workspace, rowptr,
    // colidx, out_bmu, out_dist
    size_t ws_need = 0;                    // (a smaller batch may take another route)
    for (int k = 0; k < n_batches; ++k) {
        const size_t w = N[k] > 0 ? bmu_search_workspace_bytes(D, M, N[k], rowptr_host[k][N[k]], nullptr) : 0;
        if (w > ws_need) ws_need = w;
    }
    const size_t norms_bytes = 256 + align_up((size_t)M * 4, 256);
    // the two-stage searches share what depends on the codebook alone
    bmu_opts none;
    memset(&none, 0, sizeof(none));
    auto two_stage = [&](int k) { return screen_wanted(none, D, M, N[k], rowptr_host[k][N[k]]); };
    int sharing = 0;
    for (int k = 0; k < n_batches; ++k) sharing += N[k] > 0 && two_stage(k);
    ScreenShared shared;
    memset(&shared, 0, sizeof(shared));
    if (sharing > 1) screen_shared_layout(D, M, screen_head_rows(none, D), screen_chunk(none, D), &shared.lay);
    if (shared.lay.map_total > SHARED_IMAGE_MAX) sharing = 0;
    const size_t shared_bytes = sharing > 1 ? align_up(shared.lay.total, 256) : 0;
    const size_t rp_off = align_up(ws_need, 256);
    const size_t ci_off = align_up(rp_off + (size_t)(max_n + 1) * 4, 256);
    const size_t ob_off = align_up(ci_off + (size_t)max_nnz * 4, 256);
    const size_t od_off = align_up(ob_off + (size_t)max_n * 4, 256);
    const size_t per_buf = align_up(od_off + (size_t)max_n * 4, 256);
    void *p = nullptr;
    if ((rc = scratch_get(norms_bytes + shared_bytes + 2 * per_buf, &p))) return rc;
    int dev = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    StreamCtx *c = nullptr;
    if ((rc = stream_ctx_get(dev, &c))) return rc;
    char *b = static_cast<char *>(p);
    uint32_t *sticky = reinterpret_cast<uint32_t *>(b);
    float *norms = reinterpret_cast<float *>(b + 256);
    shared.base = b + norms_bytes;
    BMU_CUDA(cudaMemsetAsync(sticky, 0, 256, s));
    if ((rc = launch_norms(W, D, M, norms, s))) return rc;
    for (int k = 0; k < n_batches; ++k) {
        if (N[k] == 0) continue;
        const int i = k & 1;
        char *buf = b + norms_bytes + shared_bytes + (size_t)i * per_buf;
        const int64_t n = N[k], nnz = rowptr_host[k][n];
        int32_t *rp = reinterpret_cast<int32_t *>(buf + rp_off);
        int32_t *ci = reinterpret_cast<int32_t *>(buf + ci_off);
        int32_t *ob = reinterpret_cast<int32_t *>(buf + ob_off);
        float *od = reinterpret_cast<float *>(buf + od_off);
        // upload: the buffer is free once the results of its previous batch are out
        if (k >= 2) BMU_CUDA(cudaStreamWaitEvent(c->copy, c->d2h[i], 0));
        BMU_CUDA(cudaMemcpyAsync(rp, rowptr_host[k], (size_t)(n + 1) * 4, cudaMemcpyHostToDevice, c->copy));
        if (nnz)
            BMU_CUDA(cudaMemcpyAsync(ci, colidx_host[k], (size_t)nnz * 4, cudaMemcpyHostToDevice, c->copy));
        BMU_CUDA(cudaEventRecord(c->h2d[i], c->copy));
        // search on the caller's stream
        BMU_CUDA(cudaStreamWaitEvent(s, c->h2d[i], 0));
        if ((rc = search_impl(W, D, M, norms, rp, ci, n, nnz, ob, od, nullptr, buf, ws_need, s, nullptr, nullptr, 0,
                              sharing > 1 && two_stage(k) ? &shared : nullptr)))
            return rc;
        // the next search of this buffer clears its status word: keep what this one left
        { status_accumulate_kernel<<<1, 1, 0, s>>>(reinterpret_cast<const uint32_t *>(buf), sticky); BMU_LAUNCHED(); }
        BMU_CUDA(cudaEventRecord(c->done[i], s));
        // download on the copy stream
        BMU_CUDA(cudaStreamWaitEvent(c->copy, c->done[i], 0));
        BMU_CUDA(cudaMemcpyAsync(out_bmu_host[k], ob, (size_t)n * 4, cudaMemcpyDeviceToHost, c->copy));
        BMU_CUDA(cudaMemcpyAsync(out_dist_host[k], od, (size_t)n * 4, cudaMemcpyDeviceToHost, c->copy));
        BMU_CUDA(cudaEventRecord(c->d2h[i], c->copy));
    }
    uint32_t status = 0;
    BMU_CUDA(cudaMemcpyAsync(&status, sticky, sizeof(status), cudaMemcpyDeviceToHost, s));
    BMU_CUDA(cudaStreamSynchronize(s));
    BMU_CUDA(cudaStreamSynchronize(c->copy));
    if (status) return status_error(status);
    return BMU_OK;
}

int bmu_status_of_word(uint32_t status_word)
{
    return status_word ? status_error(status_word) : BMU_OK;
}

int bmu_last_status(uint32_t *out_status, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!out_status) { set_error("null pointer argument"); return BMU_ERR_INVALID_ARG; }
    *out_status = 0;
    int dev = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) { set_error("device ordinal %d out of range", dev); return BMU_ERR_UNSUPPORTED; }
    void *p = nullptr;
    {
        std::lock_guard<std::mutex> g(g_mu);
        p = g_scratch[dev].p;
    }
    if (p) BMU_CUDA(cudaMemcpyAsync(out_status, p, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    BMU_CUDA(cudaStreamSynchronize(s));
    if (*out_status) return status_error(*out_status);
    return BMU_OK;
}

int bmu_selftest_wait_timeout(void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    void *p = nullptr;
    int rc = scratch_get(512, &p);          // word 0 of the scratch stays the searches' status word
    if (rc) return rc;
    uint32_t *status = reinterpret_cast<uint32_t *>(static_cast<char *>(p) + 256);
    BMU_CUDA(cudaMemsetAsync(status, 0, 256, s));
    if ((rc = launch_wait_timeout_selftest(status, s))) return rc;
    uint32_t h = 0;
    BMU_CUDA(cudaMemcpyAsync(&h, status, sizeof(h), cudaMemcpyDeviceToHost, s));
    BMU_CUDA(cudaStreamSynchronize(s));
    if (h) return status_error(h);
    return BMU_OK;
}

int bmu_release_scratch(void)
{
    int dev = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return BMU_OK;
    std::lock_guard<std::mutex> g(g_mu);
    Scratch &sc = g_scratch[dev];
    if (sc.p) {
        BMU_CUDA(cudaDeviceSynchronize());
        BMU_CUDA(cudaFree(sc.p));
        sc.p = nullptr; sc.bytes = 0;
    }
    return BMU_OK;
}

int bmu_validate_csr(const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz,
                     int64_t D, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = check_sizes(D, 0, N, nnz);
    if (rc) return rc;
    if (!rowptr || (nnz > 0 && !colidx)) { set_error("null pointer argument"); return BMU_ERR_INVALID_ARG; }
    void *p = nullptr;
    if ((rc = scratch_get(512, &p))) return rc;   // word 0 stays the searches' status word
    int32_t *flags = reinterpret_cast<int32_t *>(static_cast<char *>(p) + 256);
    if ((rc = launch_validate_csr(rowptr, colidx, N, nnz, D, flags, s))) return rc;
    int32_t h = 0;
    BMU_CUDA(cudaMemcpyAsync(&h, flags, sizeof(h), cudaMemcpyDeviceToHost, s));
    BMU_CUDA(cudaStreamSynchronize(s));
    if (h) {
        set_error("invalid CSR:%s%s%s%s%s", (h & 1) ? " rowptr[0] != 0;" : "",
                  (h & 2) ? " rowptr[N] != nnz;" : "", (h & 4) ? " rowptr decreases;" : "",
                  (h & 8) ? " colidx outside [0, D);" : "",
                  (h & 16) ? " a row lists more than 65535 ids;" : "");
        return BMU_ERR_INVALID_ARG;
    }
    return BMU_OK;
}

// ---- reusable tiling plan: a frozen corpus searched once per epoch ------------
struct bmu_plan {
    int64_t D, M, N, nnz;
    bmu_opts opts;
    const int32_t *rowptr, *colidx;
    void *ws;
    size_t ws_bytes;
};

size_t bmu_plan_workspace_bytes(int64_t N, int64_t nnz, int64_t D, int64_t M, const bmu_opts *opts)
{
    if (D < 0 || M < 0 || N < 0 || nnz < 0) return 0;
    bmu_opts o;
    memset(&o, 0, sizeof(o));
    if (opts) o = *opts;
    return query_bytes(o, D, M, N, nnz, false, true);
}

int bmu_plan_create(const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz, int64_t D,
                    int64_t M, const bmu_opts *opts, void *workspace, size_t workspace_bytes,
                    bmu_plan **plan, void *stream)
{
    if (!plan) { set_error("null pointer argument"); return BMU_ERR_INVALID_ARG; }
    *plan = nullptr;
    if (N <= 0) { set_error("a plan needs at least one document"); return BMU_ERR_INVALID_ARG; }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = search_impl(nullptr, D, M, nullptr, rowptr, colidx, N, nnz, nullptr, nullptr, opts,
                         workspace, workspace_bytes, s, nullptr, nullptr, 1);
    if (rc) return rc;
    // the searches that reuse the plan clear the status word: read the size checks of the
    // tiling pass now
    uint32_t status = 0;
    BMU_CUDA(cudaMemcpyAsync(&status, workspace, sizeof(status), cudaMemcpyDeviceToHost, s));
    BMU_CUDA(cudaStreamSynchronize(s));
    if (status) return status_error(status);
    bmu_plan *p = new (std::nothrow) bmu_plan;
    if (!p) { set_error("out of host memory"); return BMU_ERR_INVALID_ARG; }
    p->D = D; p->M = M; p->N = N; p->nnz = nnz;
    memset(&p->opts, 0, sizeof(p->opts));
    if (opts) p->opts = *opts;
    p->rowptr = rowptr; p->colidx = colidx; p->ws = workspace; p->ws_bytes = workspace_bytes;
    *plan = p;
    return BMU_OK;
}

int bmu_search_planned(const bmu_plan *plan, const float *W, const float *norms, int32_t *out_bmu,
                       float *out_dist, void *stream)
{
    if (!plan) { set_error("null plan"); return BMU_ERR_INVALID_ARG; }
    return search_impl(W, plan->D, plan->M, norms, plan->rowptr, plan->colidx, plan->N, plan->nnz,
                       out_bmu, out_dist, &plan->opts, plan->ws, plan->ws_bytes,
                       static_cast<cudaStream_t>(stream), nullptr, nullptr, 2);
}

int bmu_plan_order(const bmu_plan *plan, int32_t *out_order, void *stream)
{
    if (!plan || !out_order) { set_error("null pointer argument"); return BMU_ERR_INVALID_ARG; }
    Route r;
    int rc = route_search(plan->opts, plan->D, plan->M, plan->N, plan->nnz, 0, r);
    if (rc) return rc;
    if (r.kernel == 1) {
        set_error("the generic kernel makes no plan: documents keep the corpus order");
        return BMU_ERR_UNSUPPORTED;
    }
    const Layout l = layout_of(plan->opts, plan->D, plan->M, plan->N, plan->nnz, false, true);
    const char *perm = static_cast<const char *>(plan->ws) + l.plan_off + l.plan.perm_off;
    BMU_CUDA(cudaMemcpyAsync(out_order, perm, (size_t)plan->N * sizeof(int32_t),
                             cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream)));
    return BMU_OK;
}

void bmu_plan_destroy(bmu_plan *plan) { delete plan; }

// ---- the rest of a batch epoch (Table 4: scatter, blur, write-back) -----------
int bmu_update_scatter(const int32_t *rowptr, const int32_t *colidx, int64_t N, int64_t nnz,
                       const int32_t *bmu, int64_t D, int64_t M, uint32_t *num, uint32_t *cnt,
                       void *stream)
{
    int rc = check_sizes(D, M, N, nnz);
    if (rc) return rc;
    if (N == 0) return BMU_OK;
    if (!rowptr || !bmu || !num || !cnt || (nnz > 0 && !colidx)) {
        set_error("null pointer argument");
        return BMU_ERR_INVALID_ARG;
    }
    if (M == 0) { set_error("empty map: its documents have no unit"); return BMU_ERR_INVALID_ARG; }
    return launch_update_scatter(rowptr, colidx, N, bmu, D, M, num, cnt, static_cast<cudaStream_t>(stream));
}

int bmu_update_blur(const uint32_t *num, const uint32_t *cnt, int64_t D, int32_t edge_x,
                    int32_t edge_y, float sigma, float *num_blur, float *cnt_blur, void *stream)
{
    if (D < 0 || edge_x < 0 || edge_y < 0 || !(sigma >= 0.f)) {
        set_error("negative size or sigma");
        return BMU_ERR_INVALID_ARG;
    }
    int rc = check_sizes(D, (int64_t)edge_x * edge_y, 0, 0);
    if (rc) return rc;
    if (D > LANES_MAX_D) { set_error("blur: D beyond %d", LANES_MAX_D); return BMU_ERR_UNSUPPORTED; }
    if ((int64_t)edge_x * edge_y == 0) return BMU_OK;
    if (!cnt || !cnt_blur || (D > 0 && (!num || !num_blur))) {
        set_error("null pointer argument");
        return BMU_ERR_INVALID_ARG;
    }
    return launch_update_blur(num, cnt, D, edge_x, edge_y, sigma, num_blur, cnt_blur,
                              static_cast<cudaStream_t>(stream));
}

int bmu_update_writeback(const float *num_blur, const float *cnt_blur, int64_t D, int64_t M,
                         float *W, void *stream)
{
    int rc = check_sizes(D, M, 0, 0);
    if (rc) return rc;
    if (D * M == 0) return BMU_OK;
    if (D > 65535) { set_error("write-back: D beyond 65535"); return BMU_ERR_UNSUPPORTED; }
    if (!num_blur || !cnt_blur || !W) { set_error("null pointer argument"); return BMU_ERR_INVALID_ARG; }
    return launch_update_writeback(num_blur, cnt_blur, D, M, W, static_cast<cudaStream_t>(stream));
}

int bmu_score_block_argmin(const void *scores, int32_t half, int64_t n_rows, int64_t M,
                           const float *norms, const int32_t *rowptr, int32_t *out_bmu,
                           float *out_dist, void *stream)
{
    int rc = check_sizes(0, M, n_rows, 0);
    if (rc) return rc;
    if (n_rows == 0) return BMU_OK;
    if (!scores || !norms || !rowptr || !out_bmu || !out_dist) {
        set_error("null pointer argument");
        return BMU_ERR_INVALID_ARG;
    }
    if (M == 0) { set_error("empty score rows: no neuron to return"); return BMU_ERR_INVALID_ARG; }
    if (M % (half ? 8 : 4) != 0 || (reinterpret_cast<uintptr_t>(scores) & 15) != 0 ||
        (reinterpret_cast<uintptr_t>(norms) & 15) != 0) {
        set_error("score read-back needs M %% %d == 0 and 16-byte aligned scores and norms",
                  half ? 8 : 4);
        return BMU_ERR_UNSUPPORTED;
    }
    return launch_readback_argmin(scores, half != 0, n_rows, M, norms, rowptr, out_bmu, out_dist,
                                  static_cast<cudaStream_t>(stream));
}

size_t bmu_map_errors_workspace_bytes(void) { return map_errors_workspace_bytes(); }

int bmu_map_errors(const int32_t *bmu, const int32_t *bmu2, const float *dist, int64_t N,
                   int32_t edge_x, int32_t edge_y, int32_t adjacency, double *out, void *workspace,
                   size_t workspace_bytes, void *stream)
{
    if (N < 0 || N > MAX_I32 || edge_x < 1 || edge_y < 1 || (adjacency != 4 && adjacency != 8)) {
        set_error("map errors: need 0 <= N < 2^31, edges >= 1 and adjacency 4 or 8");
        return BMU_ERR_INVALID_ARG;
    }
    if (!out || (N > 0 && (!bmu || !bmu2 || !dist))) {
        set_error("null pointer argument");
        return BMU_ERR_INVALID_ARG;
    }
    if (N > 0 && (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0 ||
                  workspace_bytes < map_errors_workspace_bytes())) {
        set_error("workspace missing, not 256-byte aligned, or smaller than %zu bytes",
                  map_errors_workspace_bytes());
        return BMU_ERR_WORKSPACE;
    }
    return launch_map_errors(bmu, bmu2, dist, N, edge_x, adjacency, out, workspace,
                             static_cast<cudaStream_t>(stream));
}

}  // extern "C"

// ---- search with library-resident scratch (no allocation anywhere) ---------
// The scratch of the generic kernel's search -- norms and the running
// per-document minimum -- in an array that is part of the library image.  The
// name below is only a host-side handle: device code may use it directly, but
// host code must ask the runtime for its device address before handing it to a
// kernel, once per device and with that device current.
static const size_t STATIC_SCRATCH_BYTES = (size_t)8 << 20;
static __device__ __align__(256) unsigned char g_static_scratch[STATIC_SCRATCH_BYTES];
static void *g_static_scratch_addr[64];
static std::mutex g_static_mu;

extern "C" int bmu_search_static(const float *W, int64_t D, int64_t M, const int32_t *rowptr,
                                 const int32_t *colidx, int64_t N, int64_t nnz, int32_t *out_bmu,
                                 float *out_dist, void *stream)
{
    int rc = bmu::check_sizes(D, M, N, nnz);
    if (rc) return rc;
    if (N == 0) return BMU_OK;
    const size_t need = bmu::layout_for(D, M, N, nnz, 1).total;
    if (need > STATIC_SCRATCH_BYTES) {
        bmu::set_error("bmu_search_static: M=%lld and N=%lld need %zu bytes of scratch, the "
                       "built-in array holds %zu; split the batch or use bmu_search_ws",
                       (long long)M, (long long)N, need, STATIC_SCRATCH_BYTES);
        return BMU_ERR_UNSUPPORTED;
    }
    int dev = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) { bmu::set_error("device ordinal %d out of range", dev); return BMU_ERR_UNSUPPORTED; }
    void *scratch = nullptr;
    {
        std::lock_guard<std::mutex> g(g_static_mu);
        if (!g_static_scratch_addr[dev]) {
            void *p = nullptr;
            BMU_CUDA(cudaGetSymbolAddress(&p, g_static_scratch));
            g_static_scratch_addr[dev] = p;
        }
        scratch = g_static_scratch_addr[dev];
    }
    bmu_opts o;
    memset(&o, 0, sizeof(o));
    o.kernel = 1;
    return bmu::search_impl(W, D, M, nullptr, rowptr, colidx, N, nnz, out_bmu, out_dist, &o,
                            scratch, STATIC_SCRATCH_BYTES, static_cast<cudaStream_t>(stream));
}
