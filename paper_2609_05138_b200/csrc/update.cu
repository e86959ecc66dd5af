// The rest of a batch epoch after the search (Table 4: "scatter", "blur",
// "write-back"; Section 6: the scatter into accumulators is O(N.nnz), the blur is
// the O(M) term).  The paper times these steps without printing formulas; this is
// the textbook batch update on a rectangular, non-periodic map of edge_y rows by
// edge_x columns (neuron j = y * edge_x + x):
//
//   scatter     num[f][j] = #{ i : bmu_i = j and f in x_i },  cnt[j] = #{ i : bmu_i = j }
//               -- integer counters, exact
//   blur        B[f][j] = sum_k h(j, k) num[f][k],  c[j] = sum_k h(j, k) cnt[k],
//               h = exp(-(dx^2 + dy^2) / (2 sigma^2)) for |dx|, |dy| <= R = ceil(3 sigma)
//   write-back  W[f][j] = B[f][j] / c[j] where c[j] > 0, otherwise unchanged
//
// All three are bound by HBM: the scatter by its scattered 4-byte atomics, the
// blur and the write-back by one read and one write of a D x M plane set.
#include "common.cuh"

#include <math.h>

namespace bmu {

// One warp per document: its unit's counter, then one atomic per listed feature.
//
// The counters of a large map do not fit L2, and a document's counters lie scattered over all of it:
// in corpus order nearly every atomic fetches a sector of its own from DRAM and writes it back.  So
// the units are taken in `passes` ranges, one after the other along blockIdx.y, each with counters
// that stay in L2 while every document of the range is added: a block looks through SCATTER_DOCS
// documents for those of its range (a compare per document and pass) and its warps add them.
// 300,000 documents, 128 x 128 x 16,384: 467 us in corpus order, 335 us in
// 86 passes (72e9 atomics/s); 60,000 documents, 90 x 70 x 10,007: 74 and 76.
static const int SCATTER_DOCS = 2048;            // most documents a block looks through

__global__ void __launch_bounds__(256)
update_scatter_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                      int64_t N, const int32_t *__restrict__ bmu, int64_t M, int64_t units, int docs,
                      uint32_t *__restrict__ num, uint32_t *__restrict__ cnt)
{
    __shared__ int32_t s_doc[SCATTER_DOCS];
    __shared__ int s_n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t first = (int64_t)blockIdx.x * docs;
    const int64_t j_lo = (int64_t)blockIdx.y * units, j_hi = j_lo + units;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    for (int k = 0; k < docs / 256; ++k) {
        const int64_t i = first + 256 * k + threadIdx.x;
        const int64_t j = i < N ? (int64_t)__ldg(bmu + i) : -1;
        const bool in = j >= j_lo && j < j_hi;
        const uint32_t who = __ballot_sync(0xffffffffu, in);
        int at = 0;
        if (lane == 0 && who) at = atomicAdd(&s_n, __popc(who));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (in) s_doc[at + __popc(who & ((1u << lane) - 1u))] = (int32_t)i;
    }
    __syncthreads();
    const int n = s_n;
    for (int d = warp; d < n; d += 8) {
        const int64_t i = s_doc[d], j = __ldg(bmu + i);
        const int beg = __ldg(rowptr + i), end = __ldg(rowptr + i + 1);
        if (lane == 0) atomicAdd(cnt + j, 1u);
        for (int e = beg + lane; e < end; e += 32)
            atomicAdd(num + (int64_t)__ldg(colidx + e) * M + j, 1u);
    }
}

static const int BLUR_RMAX = 24;               // sigma <= 8
static const int BLUR_THREADS = 256, BLUR_WARPS = BLUR_THREADS / 32;

// taps g[|d|], twice each: the packed multiplier of two neighbouring values
struct BlurTaps { float2 g[BLUR_RMAX + 1]; };
struct BlurArgs {
    const uint32_t *num, *cnt;
    float *num_blur, *cnt_blur;
    int64_t D;
    int32_t vec;                               // rows are whole, aligned 16-byte pieces
    int32_t edge_x, edge_y, tx, ty, pitch;     // tile; 8-byte cells per staged row pair (a multiple of 4)
};

__device__ __forceinline__ void fma2(u64 &acc, u64 a, u64 b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ u64 pack2(float lo, float hi)
{
    return ((u64)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}

// One block per tile of one plane (planes 0 .. D-1 are the feature planes of `num`, plane D is
// `cnt`), the radius a template parameter so that every loop unrolls; packed fp32 arithmetic
// (fma.rn.f32x2) throughout.
//   stage  the tile, its halo columns (zero outside the map) and the halo rows that exist, as pairs
//          of rows: cell c of pair p holds (row 2p, row 2p + 1) of column c - R.  A cell is skipped
//          after every eighth, so that lanes eight columns apart hit distinct banks.
//   rows   a warp owns whole row pairs: a lane takes eight neighbouring outputs of both rows from
//          8 + 2R cells, and the results replace the pair in place, now as two plain rows -- no second
//          buffer, so the tile can be a whole map of 128 x 80 and has no halo to compute twice.
//   cols   a thread takes two neighbouring columns and eight rows, and stores them.
// Bound by the packed multiplier at large radii (two passes of 2R + 1 taps: 140 us of the 400 at radius
// 20, 90 x 70 x 10,007) and by the latency between its phases: 64 registers, for four blocks per SM,
// took a third off the same kernel at 128 (632 -> 400 us).
template <int R>
__global__ void __launch_bounds__(BLUR_THREADS, R <= 8 ? 5 : 4)
update_blur_kernel(const BlurArgs a, const __grid_constant__ BlurTaps taps)
{
    extern __shared__ __align__(16) float2 cells[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t plane = blockIdx.y, M = (int64_t)a.edge_x * a.edge_y;
    const uint32_t *src = plane < a.D ? a.num + plane * M : a.cnt;
    float *dst = plane < a.D ? a.num_blur + plane * M : a.cnt_blur;
    const int tiles_x = (a.edge_x + a.tx - 1) / a.tx;
    const int x0 = (int)(blockIdx.x % tiles_x) * a.tx, y0 = (int)(blockIdx.x / tiles_x) * a.ty;
    const int nx = min(a.tx, a.edge_x - x0), ny = min(a.ty, a.edge_y - y0);      // outputs
    const int y_lo = max(0, y0 - R), y_hi = min(a.edge_y, y0 + ny + R);          // staged rows
    const int rows = y_hi - y_lo, pairs = (rows + 1) / 2, segs = (nx + 7) / 8;
    auto g2 = [&](int d) { const float2 t = taps.g[d < 0 ? -d : d]; return pack2(t.x, t.y); };

    // stage: all loads of a step before its first store
    const int width = 8 * segs + 2 * R;                          // cells of a pair
    if (a.vec) {
        // rows are whole 16-byte pieces: pieces q of the columns from (x0 - R) rounded down to four
        const int xa = (x0 - R) & ~3, shift = x0 - R - xa, nq = (width + shift + 3) / 4;
        constexpr int K = 4;
        for (int i0 = threadIdx.x; i0 < pairs * nq; i0 += K * BLUR_THREADS) {
            uint4 v[K][2];
            int cell[K], pr[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int item = i0 + k * BLUR_THREADS;
                pr[k] = item / nq;
                const int x = xa + 4 * (item - pr[k] * nq);
                cell[k] = x - (x0 - R);
                v[k][0] = v[k][1] = make_uint4(0u, 0u, 0u, 0u);
                if (pr[k] < pairs && x >= 0 && x < a.edge_x) {
                    const uint32_t *r0 = src + (int64_t)(y_lo + 2 * pr[k]) * a.edge_x + x;
                    v[k][0] = __ldcs(reinterpret_cast<const uint4 *>(r0));
                    if (2 * pr[k] + 1 < rows) v[k][1] = __ldcs(reinterpret_cast<const uint4 *>(r0 + a.edge_x));
                }
            }
#pragma unroll
            for (int k = 0; k < K; ++k) {
                if (pr[k] >= pairs) break;
                float2 *row = cells + (size_t)pr[k] * a.pitch;
                const uint32_t e0[4] = {v[k][0].x, v[k][0].y, v[k][0].z, v[k][0].w};
                const uint32_t e1[4] = {v[k][1].x, v[k][1].y, v[k][1].z, v[k][1].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int c = cell[k] + i;
                    if (c >= 0 && c < width) row[c + (c >> 3)] = make_float2((float)e0[i], (float)e1[i]);
                }
            }
        }
    } else {
        constexpr int K = (128 + 2 * R + 31) / 32;               // steps of a warp over a pair
        for (int p = warp; p < pairs; p += BLUR_WARPS) {
            const uint32_t *r0 = src + (int64_t)(y_lo + 2 * p) * a.edge_x;
            const bool two = 2 * p + 1 < rows;
            uint32_t v[K][2];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int x = x0 - R + lane + 32 * k;
                const bool in = lane + 32 * k < width && x >= 0 && x < a.edge_x;
                v[k][0] = in ? __ldcs(r0 + x) : 0u;
                v[k][1] = in && two ? __ldcs(r0 + a.edge_x + x) : 0u;
            }
            float2 *row = cells + (size_t)p * a.pitch;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int c = lane + 32 * k;
                if (c < width) row[c + (c >> 3)] = make_float2((float)v[k][0], (float)v[k][1]);
            }
        }
    }
    __syncthreads();
    {
        const int per = segs >= 32 ? 1 : 32 / segs;              // row pairs a warp takes at a time
        const int sub = lane / segs, seg = lane - sub * segs;
        for (int p0 = warp * per; p0 < pairs; p0 += BLUR_WARPS * per) {
            const int p = p0 + sub;
            const bool act = sub < per && p < pairs;
            u64 acc[8] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
            float2 *row = cells + (size_t)p * a.pitch;
            if (act) {
                const u64 *win = reinterpret_cast<const u64 *>(row) + 9 * seg;
#pragma unroll
                for (int e = 0; e < 8 + 2 * R; ++e) {
                    const u64 v = win[e + (e >> 3)];
#pragma unroll
                    for (int o = 0; o < 8; ++o) {
                        const int d = e - o - R;                 // tap offset of input e for output o
                        if (d >= -R && d <= R) fma2(acc[o], g2(d), v);
                    }
                }
            }
            __syncwarp();                                        // the pair has been read
            if (act) {
                float4 *m = reinterpret_cast<float4 *>(reinterpret_cast<float *>(row) + 8 * seg);
                m[0] = make_float4(lo_f(acc[0]), lo_f(acc[1]), lo_f(acc[2]), lo_f(acc[3]));
                m[1] = make_float4(lo_f(acc[4]), lo_f(acc[5]), lo_f(acc[6]), lo_f(acc[7]));
                m = reinterpret_cast<float4 *>(reinterpret_cast<float *>(row) + a.pitch + 8 * seg);
                m[0] = make_float4(hi_f(acc[0]), hi_f(acc[1]), hi_f(acc[2]), hi_f(acc[3]));
                m[1] = make_float4(hi_f(acc[4]), hi_f(acc[5]), hi_f(acc[6]), hi_f(acc[7]));
            }
            __syncwarp();
        }
    }
    __syncthreads();
    const int cols2 = (nx + 1) / 2;
    const bool whole = (a.edge_x & 1) == 0 && (reinterpret_cast<uintptr_t>(dst) & 7) == 0;
    const float *mid = reinterpret_cast<const float *>(cells);
    for (int item = threadIdx.x; item < cols2 * ((ny + 7) / 8); item += BLUR_THREADS) {
        const int r8 = item / cols2, c2 = item - r8 * cols2;
        const int top = y0 + 8 * r8 - R - y_lo;                  // first row of the window, staged
        const float *col = mid + 2 * c2;
        u64 acc[8] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int e = 0; e < 8 + 2 * R; ++e) {
            const int r = top + e;                               // (row r sits at r * pitch floats)
            const u64 v = r >= 0 && r < rows ? *reinterpret_cast<const u64 *>(col + (size_t)r * a.pitch) : 0ull;
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                const int d = e - o - R;
                if (d >= -R && d <= R) fma2(acc[o], g2(d), v);
            }
        }
        float *out = dst + (int64_t)(y0 + 8 * r8) * a.edge_x + x0 + 2 * c2;
#pragma unroll
        for (int o = 0; o < 8; ++o)
            if (8 * r8 + o < ny) {
                if (whole) {
                    __stcs(reinterpret_cast<float2 *>(out), make_float2(lo_f(acc[o]), hi_f(acc[o])));
                } else {
                    __stcs(out, lo_f(acc[o]));
                    if (2 * c2 + 1 < nx) __stcs(out + 1, hi_f(acc[o]));
                }
                out += a.edge_x;
            }
    }
}

// Tiles: columns in as few equal parts of at most 128 as there must be; all rows if the staged tile
// then fits `room` bytes of shared memory (four blocks per SM for small radii, two for large ones,
// where halo rows computed twice would cost more than occupancy gives), else equal parts that do.
template <int R>
static int launch_blur(BlurArgs a, const BlurTaps &t, cudaStream_t s)
{
    const int room = R <= 8 ? 54 * 1024 : 108 * 1024;
    const int ntx = (a.edge_x + 127) / 128;
    a.tx = ((a.edge_x + ntx - 1) / ntx + 7) / 8 * 8;
    const int cells = a.tx + 2 * R;
    a.pitch = (cells + cells / 8 + 4) / 4 * 4;                   // (rows of a pair start on 16 bytes)
    const int most = room / (a.pitch * 4) / 2 * 2;               // staged rows
    a.ty = a.edge_y;
    if (a.edge_y > most) {
        const int nty = (a.edge_y + most - 2 * R - 1) / (most - 2 * R);
        a.ty = (a.edge_y + nty - 1) / nty;
    }
    const int rows = a.edge_y > most ? a.ty + 2 * R : a.edge_y;
    const size_t smem = (size_t)((rows + 1) / 2) * a.pitch * sizeof(float2);
    static bool configured[64];
    int dev = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && !configured[dev]) {
        BMU_CUDA(cudaFuncSetAttribute(update_blur_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024));
        configured[dev] = true;
    }
    const int64_t tiles = (int64_t)((a.edge_x + a.tx - 1) / a.tx) * ((a.edge_y + a.ty - 1) / a.ty);
    const dim3 grid((unsigned)tiles, (unsigned)(a.D + 1));
    { update_blur_kernel<R><<<grid, BLUR_THREADS, smem, s>>>(a, t); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

// radius -> instance
template <int R>
static int launch_blur_radius(int r, const BlurArgs &a, const BlurTaps &t, cudaStream_t s)
{
    if (r == R) return launch_blur<R>(a, t, s);
    if constexpr (R < BLUR_RMAX) return launch_blur_radius<R + 1>(r, a, t, s);
    return BMU_ERR_UNSUPPORTED;
}

// ---- the same blur for radii 1 .. 8 on maps whose rows are whole 16-byte pieces ----------
// One block per 64 x 64 tile of one plane, radius a template parameter so that every loop
// unrolls and the taps sit in registers.  Packed fp32 arithmetic throughout (fma.rn.f32x2):
// the row pass works on two map rows at once (the tile is staged as (row 2p, row 2p+1) pairs),
// the column pass on two neighbouring columns at once, and the outputs leave as 8-byte stores.
// Bound by its phases, load, rows, columns, store, of four to five blocks per SM that overlap only
// in part: 451 us at radius 2 and 589 at radius 6 for 128 x 128 x 16,384, where the bytes take 323.
template <int R> struct BlurFast {
    static constexpr int TX = 64, TY = 64;
    static constexpr int RP = (R + 3) / 4 * 4;          // halo in x, whole 16-byte pieces
    static constexpr int SPAN = TY + 2 * R;             // staged rows (even)
    static constexpr int NRP = SPAN / 2;                // staged row pairs
    static constexpr int NC = (TX + 2 * RP) / 4;        // 16-byte pieces per staged row
    static constexpr int PX = TX + 2 * RP + 1;          // pairs per staged row pair (odd pitch:
                                                        // lanes over row pairs hit distinct banks)
    static constexpr int PM = TX + 4;                   // floats per row of the row-pass result
    static constexpr size_t SMEM = (size_t)SPAN * PM * 4 + (size_t)NRP * PX * 8;
};

template <int R>
__global__ void __launch_bounds__(256, 4)
update_blur_fast_kernel(const uint32_t *__restrict__ num, const uint32_t *__restrict__ cnt, int64_t D,
                        int32_t edge_x, int32_t edge_y, const __grid_constant__ BlurTaps taps,
                        float *__restrict__ num_blur, float *__restrict__ cnt_blur)
{
    using F = BlurFast<R>;
    extern __shared__ __align__(16) unsigned char smraw[];
    float *mid = reinterpret_cast<float *>(smraw);                          // SPAN x PM
    float2 *in2 = reinterpret_cast<float2 *>(smraw + (size_t)F::SPAN * F::PM * 4);   // NRP x PX
    const int64_t plane = blockIdx.z, M = (int64_t)edge_x * edge_y;
    const uint32_t *src = plane < D ? num + plane * M : cnt;
    float *dst = plane < D ? num_blur + plane * M : cnt_blur;
    const int x0 = blockIdx.x * F::TX, y0 = blockIdx.y * F::TY;

    // taps g[-R .. R] are symmetric: ts[k] = (g[k], g[k]) for k = |d|
    u64 ts[R + 1];
#pragma unroll
    for (int k = 0; k <= R; ++k) ts[k] = pack2(taps.g[k].x, taps.g[k].y);

    // stage the tile and its halo as pairs of rows, zero outside the map: every load of a thread
    // before its first store
    constexpr int ITEMS = F::NRP * F::NC, K = (ITEMS + 255) / 256;
    uint4 st[K][2];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int item = threadIdx.x + 256 * k;
        const int rp = item / F::NC, q = item - rp * F::NC;
        const int x = x0 - F::RP + 4 * q, y = y0 - R + 2 * rp;
        st[k][0] = st[k][1] = make_uint4(0u, 0u, 0u, 0u);
        if (item < ITEMS && x >= 0 && x < edge_x) {
            if (y >= 0 && y < edge_y)
                st[k][0] = __ldcs(reinterpret_cast<const uint4 *>(src + (int64_t)y * edge_x + x));
            if (y + 1 >= 0 && y + 1 < edge_y)
                st[k][1] = __ldcs(reinterpret_cast<const uint4 *>(src + (int64_t)(y + 1) * edge_x + x));
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int item = threadIdx.x + 256 * k;
        if (item >= ITEMS) break;
        const int rp = item / F::NC, q = item - rp * F::NC;
        const uint4 a = st[k][0], b = st[k][1];
        float2 *o = in2 + rp * F::PX + 4 * q;
        const float2 v[4] = {make_float2((float)a.x, (float)b.x), make_float2((float)a.y, (float)b.y),
                             make_float2((float)a.z, (float)b.z), make_float2((float)a.w, (float)b.w)};
        // neighbouring lanes sit 32 bytes apart: lane l stores its four pairs starting with
        // pair (l / 4) % 4, so that 16 lanes hit 16 different bank pairs at every step
        const int rot = (threadIdx.x >> 2) & 3;
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const int kk = (n + rot) & 3;
            const float2 lo = (kk & 1) ? v[1] : v[0], hi = (kk & 1) ? v[3] : v[2];
            o[kk] = (kk & 2) ? hi : lo;
        }
    }
    __syncthreads();
    // row pass: item = (group of four outputs g4, row pair rp), lanes over row pairs
    for (int item = threadIdx.x; item < F::NRP * (F::TX / 4); item += 256) {
        const int g4 = item / F::NRP, rp = item - g4 * F::NRP;
        const u64 *win = reinterpret_cast<const u64 *>(in2 + rp * F::PX + (F::RP - R) + 4 * g4);
        u64 acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int e = 0; e < 4 + 2 * R; ++e) {
            const u64 v = win[e];
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const int d = e - o - R;                 // tap offset of input e for output o
                if (d >= -R && d <= R) fma2(acc[o], ts[d < 0 ? -d : d], v);
            }
        }
        float *m0 = mid + (2 * rp) * F::PM + 4 * g4;
        *reinterpret_cast<float4 *>(m0) = make_float4(lo_f(acc[0]), lo_f(acc[1]), lo_f(acc[2]), lo_f(acc[3]));
        *reinterpret_cast<float4 *>(m0 + F::PM) =
            make_float4(hi_f(acc[0]), hi_f(acc[1]), hi_f(acc[2]), hi_f(acc[3]));
    }
    __syncthreads();
    // column pass: a thread takes two neighbouring columns and eight rows
    {
        const int c2 = threadIdx.x & 31, rg = threadIdx.x >> 5;
        const float *col = mid + (8 * rg) * F::PM + 2 * c2;
        u64 acc[8] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int e = 0; e < 8 + 2 * R; ++e) {
            const u64 v = *reinterpret_cast<const u64 *>(col + e * F::PM);
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                const int d = e - o - R;
                if (d >= -R && d <= R) fma2(acc[o], ts[d < 0 ? -d : d], v);
            }
        }
        const int x = x0 + 2 * c2, y = y0 + 8 * rg;
        if (x < edge_x) {
#pragma unroll
            for (int o = 0; o < 8; ++o)
                if (y + o < edge_y)
                    __stcs(reinterpret_cast<float2 *>(dst + (int64_t)(y + o) * edge_x + x),
                           make_float2(lo_f(acc[o]), hi_f(acc[o])));
        }
    }
}

template <int R>
static int launch_blur_fast(const uint32_t *num, const uint32_t *cnt, int64_t D, int32_t edge_x,
                            int32_t edge_y, const BlurTaps &t, float *num_blur, float *cnt_blur,
                            cudaStream_t s)
{
    using F = BlurFast<R>;
    static bool configured[64];
    int dev = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && !configured[dev]) {
        BMU_CUDA(cudaFuncSetAttribute(update_blur_fast_kernel<R>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F::SMEM));
        configured[dev] = true;
    }
    const dim3 grid((unsigned)((edge_x + F::TX - 1) / F::TX), (unsigned)((edge_y + F::TY - 1) / F::TY),
                    (unsigned)(D + 1));
    { update_blur_fast_kernel<R><<<grid, 256, F::SMEM, s>>>(num, cnt, D, edge_x, edge_y, t, num_blur,
                                                         cnt_blur); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}


// ---- ... and of 16 to 512 units ------------------------------------------------------------
// A thread owns four neighbouring columns of one plane and walks down its rows.  Column pass in registers: a
// row is added, packed (fma.rn.f32x2), to the 2R + 1 sums it belongs to, which rotate through the unrolled
// loop; the sum that is complete goes to shared memory.  Row pass: two complete rows at a time, a thread reads
// the R columns on either side of its own four.  Rows come by asynchronous copies of sixteen bytes, AHEAD rows
// ahead, each into a place that only its own thread reads; one barrier per two rows, between two buffers.
// A block carries as many planes as fit its threads, and all rows of them, or an equal part of them with R more
// on either side where planes are too few to fill the chip.
//
// Up to radius 5 near what a copy takes (128 x 128 x 16,384, 2.15 GB: 369 us at radius 2, 374 at 5, 6 TB/s; four fifths
// of the issue slots are taken too); beyond, 429 us at radius 6 and 562 at 8, by issue with few warps (112 registers, 16 per
// SM) and by fetching instructions: the loop is unrolled 2 (2R + 1) times.  The tiled kernel above, which exchanges every
// tile through shared memory twice and is bound by that, took 457, 558, 594 and 677 us.
template <int R> struct BlurStrip {
    static constexpr int T = 2 * R + 1, PAD = (R + 3) / 4 * 4;
    static constexpr int AHEAD = 8;
    static constexpr int BLOCKS = R <= 2 ? 8 : R <= 4 ? 5 : 4;       // of 128 threads per SM
};

__device__ __forceinline__ void blur_copy16(uint32_t dst, const void *src, bool there)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(there ? 16 : 0) : "memory");
}

template <int R>
__global__ void __launch_bounds__(128, BlurStrip<R>::BLOCKS)
update_blur_strip_kernel(const uint32_t *__restrict__ num, const uint32_t *__restrict__ cnt, int64_t D,
                         int32_t edge_x, int32_t edge_y, int32_t planes, int32_t part, const __grid_constant__ BlurTaps taps,
                         float *__restrict__ num_blur, float *__restrict__ cnt_blur)
{
    using S = BlurStrip<R>;
    constexpr int T = S::T, PAD = S::PAD, AHEAD = S::AHEAD;
    extern __shared__ __align__(16) unsigned char smraw[];
    uint4 *ring = reinterpret_cast<uint4 *>(smraw);                          // [AHEAD][blockDim.x]
    const int pitch = edge_x + 2 * PAD;                                      // floats per plane and row
    float *rows = reinterpret_cast<float *>(ring + AHEAD * blockDim.x);      // [2][2][planes][pitch]
    const int lanes = edge_x / 4, mine = (int)threadIdx.x / lanes, x4 = (int)threadIdx.x - mine * lanes;
    const int64_t M = (int64_t)edge_x * edge_y, plane = (int64_t)blockIdx.x * planes + mine;
    const bool act = mine < planes && plane <= D;
    const uint32_t *src = act ? (plane < D ? num + plane * M : cnt) + 4 * x4 : cnt;
    float *dst = (act && plane < D ? num_blur + plane * M : cnt_blur) + 4 * x4;
    const int y0 = (int)blockIdx.y * part, y1 = min(edge_y, y0 + part), steps = y1 - y0 + 2 * R;
    for (int i = threadIdx.x; i < 4 * planes * pitch; i += blockDim.x) rows[i] = 0.f;      // (the columns outside the map)
    u64 ts[R + 1];
#pragma unroll
    for (int k = 0; k <= R; ++k) ts[k] = pack2(taps.g[k].x, taps.g[k].y);
    const uint32_t slot = (uint32_t)__cvta_generic_to_shared(ring + threadIdx.x);
    auto fetch = [&](int r) {                                                // row y0 - R + r of the plane
        const int y = y0 - R + r;
        const bool in = act && r < steps && y >= 0 && y < edge_y;
        blur_copy16(slot + (uint32_t)((r % AHEAD) * blockDim.x * 16), src + (int64_t)(in ? y : 0) * edge_x, in);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int r = 0; r < AHEAD - 1; ++r) fetch(r);
    const int row_floats = planes * pitch, at = (act ? mine : 0) * pitch + PAD + 4 * x4;
    u64 acc[T][2];
#pragma unroll
    for (int k = 0; k < T; ++k) acc[k][0] = acc[k][1] = 0ull;
    __syncthreads();
    for (int base = 0; base < steps; base += 2 * T) {
#pragma unroll
        for (int k = 0; k < 2 * T; ++k) {
            const int r = base + k;
            if (r >= steps + (steps & 1)) break;                             // (an odd last row has a partner that is not there)
            asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 2) : "memory");
            const uint4 v = ring[(r % AHEAD) * blockDim.x + threadIdx.x];
            fetch(r + AHEAD - 1);
            const u64 a = pack2((float)v.x, (float)v.y), b = pack2((float)v.z, (float)v.w);
#pragma unroll
            for (int d = 0; d < T; ++d) {                                    // output row r - d, tap |R - d|
                u64 *s = acc[(k + 2 * T - d) % T];
                const u64 g = ts[d < R ? R - d : d - R];
                if (d == 0) { s[0] = s[1] = 0ull; }
                fma2(s[0], g, a);
                fma2(s[1], g, b);
            }
            float *out = rows + ((r >> 1) & 1) * 2 * row_floats;
            if (act) {
                const u64 *s = acc[(k + 1) % T];
                *reinterpret_cast<float4 *>(out + (k & 1) * row_floats + at) = make_float4(lo_f(s[0]), hi_f(s[0]), lo_f(s[1]), hi_f(s[1]));
            }
            if (k & 1) {
                __syncthreads();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int y = y0 + r - 1 + h - 2 * R;
                    if (y < y0 || y >= y1) continue;
                    const float *c = out + h * row_floats + at - PAD;
                    float w[4 + 2 * PAD], o[4];
#pragma unroll
                    for (int i = 0; i < 4 + 2 * PAD; i += 4) {
                        const float4 t = *reinterpret_cast<const float4 *>(c + i);
                        w[i] = t.x; w[i + 1] = t.y; w[i + 2] = t.z; w[i + 3] = t.w;
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        o[i] = 0.f;
#pragma unroll
                        for (int d = -R; d <= R; ++d) o[i] = fmaf(lo_f(ts[d < 0 ? -d : d]), w[PAD + i + d], o[i]);
                    }
                    if (act) __stcs(reinterpret_cast<float4 *>(dst + (int64_t)y * edge_x), make_float4(o[0], o[1], o[2], o[3]));
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <int R>
static int launch_blur_strip(const uint32_t *num, const uint32_t *cnt, int64_t D, int32_t edge_x,
                             int32_t edge_y, const BlurTaps &t, float *num_blur, float *cnt_blur, int sms,
                             cudaStream_t s)
{
    using S = BlurStrip<R>;
    const int lanes = edge_x / 4, planes = 128 / lanes, threads = (planes * lanes + 31) / 32 * 32;
    const size_t smem = (size_t)S::AHEAD * threads * 16 + (size_t)4 * planes * (edge_x + 2 * S::PAD) * 4;
    const int64_t blocks = (D + planes) / planes;
    // parts of the rows: four waves of blocks, but no more halo rows than a quarter of the others
    int parts = (int)((4ll * S::BLOCKS * sms + blocks - 1) / blocks);
    const int most = edge_y / (8 * R) > 1 ? edge_y / (8 * R) : 1;
    if (parts > most) parts = most;
    const int part = (edge_y + parts - 1) / parts;
    const dim3 grid((unsigned)blocks, (unsigned)((edge_y + part - 1) / part));
    { update_blur_strip_kernel<R><<<grid, threads, smem, s>>>(num, cnt, D, edge_x, edge_y, planes, part, t, num_blur, cnt_blur); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

// b / c, rounded to nearest.  Most sums of a rare feature are 0, which the division hands to its slow
// path (475 us instead of 335 on such planes): divide something else there.
__device__ __forceinline__ float writeback_div(float b, float c)
{
    const float q = __fdiv_rn(b == 0.f ? c : b, c);
    return b == 0.f ? 0.f : q;
}

// One row of W per blockIdx.y; float4 pieces when the row pitch allows.  Four pieces in flight per
// thread; W itself is read only for a piece with a unit that keeps its weights (on a map whose
// neighbourhoods cover it there is none): 651 us with the read, 333 us without, at 1.07 GB (6.4
// TB/s).  Rows of other widths: eight 32-bit values in flight, 75 x 75 x 12,011: 293 -> 90 us.
template <bool VEC>
__global__ void __launch_bounds__(256)
update_writeback_kernel(const float *__restrict__ num_blur, const float *__restrict__ cnt_blur,
                        int64_t M, float *__restrict__ W)
{
    const int64_t row = (int64_t)blockIdx.y * M;
    if (VEC) {
        constexpr int K = 4;
        const int64_t n4 = M / 4;
        const float4 *src = reinterpret_cast<const float4 *>(num_blur + row);
        float4 *dst = reinterpret_cast<float4 *>(W + row);
        for (int64_t i0 = (int64_t)blockIdx.x * (256 * K) + threadIdx.x; i0 < n4;
             i0 += (int64_t)gridDim.x * (256 * K)) {
            float4 b[K], c[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int64_t i = i0 + 256 * k;
                if (i < n4) {
                    b[k] = __ldcs(src + i);
                    c[k] = __ldg(reinterpret_cast<const float4 *>(cnt_blur) + i);
                }
            }
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int64_t i = i0 + 256 * k;
                if (i >= n4) break;
                float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
                if (!(c[k].x > 0.f && c[k].y > 0.f && c[k].z > 0.f && c[k].w > 0.f)) w = dst[i];
                if (c[k].x > 0.f) w.x = writeback_div(b[k].x, c[k].x);
                if (c[k].y > 0.f) w.y = writeback_div(b[k].y, c[k].y);
                if (c[k].z > 0.f) w.z = writeback_div(b[k].z, c[k].z);
                if (c[k].w > 0.f) w.w = writeback_div(b[k].w, c[k].w);
                dst[i] = w;
            }
        }
    } else {
        constexpr int K = 8;
        for (int64_t i0 = (int64_t)blockIdx.x * (256 * K) + threadIdx.x; i0 < M;
             i0 += (int64_t)gridDim.x * (256 * K)) {
            float b[K], c[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int64_t i = i0 + 256 * k;
                c[k] = i < M ? __ldg(cnt_blur + i) : 0.f;
                b[k] = i < M ? __ldcs(num_blur + row + i) : 0.f;
            }
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (c[k] > 0.f) W[row + i0 + 256 * k] = writeback_div(b[k], c[k]);
        }
    }
}


// Stopping metrics of an epoch (Table 4 "stopping metric"; Section 5: the second-best unit feeds
// the topographic error): mean d, mean sqrt(max(d, 0)) and the fraction of documents whose best
// and second-best units are not neighbours on the map.  fp64 sums in a fixed order (grid-stride
// partition, shuffle tree, warps in order, blocks in order by the last block to finish), so a
// call gives the same bits every time.
static const int ME_BLOCKS = 592, ME_THREADS = 256;

__global__ void __launch_bounds__(ME_THREADS)
map_errors_kernel(const int32_t *__restrict__ bmu, const int32_t *__restrict__ bmu2,
                  const float *__restrict__ dist, int64_t N, int32_t edge_x, int32_t adjacency,
                  double *__restrict__ part, unsigned int *__restrict__ ticket,
                  double *__restrict__ out)
{
    double sd = 0.0, sr = 0.0, er = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * ME_THREADS + threadIdx.x; i < N;
         i += (int64_t)ME_BLOCKS * ME_THREADS) {
        const double d = (double)__ldg(dist + i);
        sd += d;
        sr += d > 0.0 ? sqrt(d) : 0.0;
        const int32_t b2 = __ldg(bmu2 + i);
        if (b2 >= 0) {
            const int32_t b1 = __ldg(bmu + i);
            const int32_t dx = abs(b1 % edge_x - b2 % edge_x), dy = abs(b1 / edge_x - b2 / edge_x);
            const bool near = adjacency == 8 ? max(dx, dy) == 1 : dx + dy == 1;
            er += near ? 0.0 : 1.0;
        }
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
        sd += __shfl_xor_sync(0xffffffffu, sd, m);
        sr += __shfl_xor_sync(0xffffffffu, sr, m);
        er += __shfl_xor_sync(0xffffffffu, er, m);
    }
    __shared__ double wsum[3][ME_THREADS / 32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { wsum[0][warp] = sd; wsum[1][warp] = sr; wsum[2][warp] = er; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0, e = 0.0;
        for (int w = 0; w < ME_THREADS / 32; ++w) { a += wsum[0][w]; b += wsum[1][w]; e += wsum[2][w]; }
        part[blockIdx.x] = a;
        part[ME_BLOCKS + blockIdx.x] = b;
        part[2 * ME_BLOCKS + blockIdx.x] = e;
        __threadfence();
        last = atomicAdd(ticket, 1u) == ME_BLOCKS - 1;
    }
    __syncthreads();
    if (last && threadIdx.x < 3) {
        __threadfence();
        const volatile double *p = part + threadIdx.x * ME_BLOCKS;
        double s = 0.0;
        for (int b = 0; b < ME_BLOCKS; ++b) s += p[b];
        out[threadIdx.x] = s / (double)N;
    }
}

int launch_update_scatter(const int32_t *rowptr, const int32_t *colidx, int64_t N,
                          const int32_t *bmu, int64_t D, int64_t M, uint32_t *num, uint32_t *cnt,
                          cudaStream_t s)
{
    if (N == 0) return BMU_OK;
    // ranges of units whose counters take about 0.1 of L2 (0.3: 372 us instead of 335); whole 128-byte lines of
    // them.  At most 256 ranges, every one of which looks at all documents: beyond some 3e9 bytes of counters
    // (200 x 200 units, 16,384 features) a range takes more than that, 0.5 of L2 on 512 x 512.
    int dev = 0, l2 = 0;
    BMU_CUDA(cudaGetDevice(&dev));
    BMU_CUDA(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev));
    int64_t passes = D > 0 ? (int64_t)((double)D * (double)M * 4.0 / (0.1 * (double)l2)) + 1 : 1;
    if (passes > 256) passes = 256;
    const int64_t units = ((M + passes - 1) / passes + 31) / 32 * 32;
    passes = (M + units - 1) / units;
    // enough documents for a block that each warp finds a few of its range
    int64_t docs = (passes * 8 + 255) / 256 * 256;
    if (docs > SCATTER_DOCS) docs = SCATTER_DOCS;
    const dim3 grid((unsigned)((N + docs - 1) / docs), (unsigned)passes);
    { update_scatter_kernel<<<grid, 256, 0, s>>>(rowptr, colidx, N, bmu, M, units, (int)docs,
                                                  num, cnt); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

int launch_update_blur(const uint32_t *num, const uint32_t *cnt, int64_t D, int32_t edge_x,
                       int32_t edge_y, float sigma, float *num_blur, float *cnt_blur,
                       cudaStream_t s)
{
    const int R = sigma > 0.f ? (int)ceil(3.0 * (double)sigma) : 0;
    if (R > BLUR_RMAX) {
        set_error("blur: sigma %.3f needs a radius of %d cells, the kernel holds %d (sigma <= 8)",
                  (double)sigma, R, BLUR_RMAX);
        return BMU_ERR_UNSUPPORTED;
    }
    BlurTaps t;
    for (int d = 0; d <= BLUR_RMAX; ++d) {
        const float g = d > R ? 0.f : sigma > 0.f
            ? (float)exp(-(double)(d * d) / (2.0 * (double)sigma * (double)sigma)) : 1.f;
        t.g[d] = make_float2(g, g);
    }
    BlurArgs a;
    a.num = num; a.cnt = cnt; a.num_blur = num_blur; a.cnt_blur = cnt_blur;
    a.D = D; a.edge_x = edge_x; a.edge_y = edge_y;
    a.vec = edge_x % 4 == 0 && ((reinterpret_cast<uintptr_t>(num) | reinterpret_cast<uintptr_t>(cnt)) & 15) == 0;
    // Maps of whole 16-byte rows of 16 to 512 units at radii up to 8: the kernel that walks down the columns, faster
    // than the others wherever it was measured there (4,096 x 32 x 32, radius 6: 24 us, 36; 6,000 x 100 x 90: 115, 211;
    // 2,000 x 512 x 512: 855, 1,165; narrower rows leave its staging too little room, wider ones more than its 128
    // threads).  Wider maps whose 64 x 64 tiles are at least three quarters map: the tiled one (500 x 2,048 x 512, radius
    // 2 / 6: 911 / 1,166 us, that of whole-map tiles 1,469 / 1,766; 2,000 x 576 x 64 142 / 175, 191 / 220; 1,000 x 1,000 x
    // 120 228 / 296, 290 / 387).  Everything else: the one of whole-map tiles (90 x 70 x 10,007, radius 6 / 20: 230 / 400
    // us; before it a kernel with the radius in a loop took 543 / 1721).
    const int64_t tiled_area = (int64_t)((edge_x + 63) / 64) * ((edge_y + 63) / 64) * 4096;
    const bool outs = ((reinterpret_cast<uintptr_t>(num_blur) | reinterpret_cast<uintptr_t>(cnt_blur)) & 15) == 0;
    int dev = 0, sms = 148;
    BMU_CUDA(cudaGetDevice(&dev));
    BMU_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (a.vec && outs && R >= 1 && R <= 8 && edge_x >= 16 && edge_x <= 512) {
        switch (R) {
        case 1: return launch_blur_strip<1>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, sms, s);
        case 2: return launch_blur_strip<2>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, sms, s);
        case 3: return launch_blur_strip<3>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, sms, s);
        case 4: return launch_blur_strip<4>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, sms, s);
        case 5: return launch_blur_strip<5>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, sms, s);
        case 6: return launch_blur_strip<6>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, sms, s);
        case 7: return launch_blur_strip<7>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, sms, s);
        default: return launch_blur_strip<8>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, sms, s);
        }
    }
    if (a.vec && outs && R >= 1 && R <= 8 && 3 * tiled_area <= 4 * (int64_t)edge_x * edge_y) {
        switch (R) {
        case 1: return launch_blur_fast<1>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, s);
        case 2: return launch_blur_fast<2>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, s);
        case 3: return launch_blur_fast<3>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, s);
        case 4: return launch_blur_fast<4>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, s);
        case 5: return launch_blur_fast<5>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, s);
        case 6: return launch_blur_fast<6>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, s);
        case 7: return launch_blur_fast<7>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, s);
        default: return launch_blur_fast<8>(num, cnt, D, edge_x, edge_y, t, num_blur, cnt_blur, s);
        }
    }
    return launch_blur_radius<0>(R, a, t, s);
}

int launch_update_writeback(const float *num_blur, const float *cnt_blur, int64_t D, int64_t M,
                            float *W, cudaStream_t s)
{
    if (D * M == 0) return BMU_OK;
    const bool vec = M % 4 == 0 && ((reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(num_blur) |
                                     reinterpret_cast<uintptr_t>(cnt_blur)) & 15) == 0;
    const int64_t per_row = vec ? M / 4 : M;
    const int64_t step = vec ? 1024 : 2048;
    const dim3 grid((unsigned)((per_row + step - 1) / step < 64 ? (per_row + step - 1) / step : 64), (unsigned)D);
    if (vec) { update_writeback_kernel<true><<<grid, 256, 0, s>>>(num_blur, cnt_blur, M, W); BMU_LAUNCHED(); }
    else { update_writeback_kernel<false><<<grid, 256, 0, s>>>(num_blur, cnt_blur, M, W); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

size_t map_errors_workspace_bytes() { return 256 + (size_t)3 * ME_BLOCKS * sizeof(double); }

int launch_map_errors(const int32_t *bmu, const int32_t *bmu2, const float *dist, int64_t N,
                      int32_t edge_x, int32_t adjacency, double *out, void *ws, cudaStream_t s)
{
    if (N == 0) {
        BMU_CUDA(cudaMemsetAsync(out, 0, 3 * sizeof(double), s));
        return BMU_OK;
    }
    unsigned int *ticket = static_cast<unsigned int *>(ws);
    double *part = reinterpret_cast<double *>(static_cast<char *>(ws) + 256);
    BMU_CUDA(cudaMemsetAsync(ticket, 0, sizeof(unsigned int), s));
    { map_errors_kernel<<<ME_BLOCKS, ME_THREADS, 0, s>>>(bmu, bmu2, dist, N, edge_x, adjacency, part,
                                                      ticket, out); BMU_LAUNCHED(); }
    BMU_CUDA(cudaGetLastError());
    return BMU_OK;
}

}  // namespace bmu
