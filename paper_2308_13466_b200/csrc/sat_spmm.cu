// CSR SpMM kernels of the sat_b200 library (aggregation with the propagation matrix P),
// row gather and row scatter.  All of them are bandwidth-bound: every feature row is moved
// with 128-bit loads, one group of lanes per work item, and nothing is accumulated with
// floating-point atomics (results are reproducible).
#include "sat_internal.h"

#include <algorithm>
#include <cstdlib>

__device__ __forceinline__ float4 ld4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ void fma4(float4 &a, float w, const float4 &x)
{
    // two packed FMAs (each component rounded as by fmaf)
    const float2 ww = make_float2(w, w);
    const float2 lo = __ffma2_rn(ww, make_float2(x.x, x.y), make_float2(a.x, a.y)), hi = __ffma2_rn(ww, make_float2(x.z, x.w), make_float2(a.z, a.w));
    a = make_float4(lo.x, lo.y, hi.x, hi.y);
}

// zero the components of float4 column `idx` of a row whose bits in the row's bit mask (word_base = row * words) are 0
__device__ __forceinline__ void mask4(float4 &r, const uint32_t *__restrict__ omask, int64_t word_base, int idx)
{
    const uint32_t m = __ldg(omask + word_base + (idx >> 3)) >> ((idx & 7) * 4);
    if (!(m & 1u)) r.x = 0.f;
    if (!(m & 2u)) r.y = 0.f;
    if (!(m & 4u)) r.z = 0.f;
    if (!(m & 8u)) r.w = 0.f;
}

// -------------------------------------------------------------------------------------
// Work lists.  Every product walks a list of 16-byte descriptors, one per run of at most `chunk` entries of one row:
//   {row, partial-sum slot or -1, first entry (low 32 bits), first entry (high 16 bits) | entries << 16}
// over an array of 8-byte entries {column, weight}.  Five kinds of rows (`mode`):
//   0  local CSR rows, all entries (forward)            1  their inner prefix (backward, P_in^T = P_in)
//   2  their halo suffix (transposed predictor convolution; rows without one are not in the list and are not written)
//   3  halo rows (halo-row CSR, columns = inner rows)    4  halo rows by cache slot, the self entry first
// Rows longer than a chunk leave one un-scaled partial sum per run, added in run order by k_spmm_fixup or by the run that ends last (fixed order:
// reproducible, and identical for one partition alone or all at once).
//
// Three things decide how fast such a list is walked (measured on the kernels below, graphs with the degree skew of the tests):
//  - short chunks: a run is a serial chain of dependent gathers, and 256-entry runs of hub rows were the tail of every launch (d = 64:
//    168 us at 256 entries, 112 at 64; d = 256: 294 -> 216; 2.5 M entries).  list_chunk picks the length.
//  - equal lengths side by side: inside windows of LIST_WINDOW items the list is ordered by length, so the lane groups of a warp and the
//    warps of a block end together (112 -> 87 us at d = 64, 138 -> 114 at d = 128); a window keeps the row order, and with it the
//    locality of neighbouring rows (a full sort costs 20 % at d = 256).
//  - source blocking for partitions several times the L2 (mode 0 only).  A row-major walk re-reads most sources from DRAM: every source
//    row is used by ~10-20 rows spread over the whole partition and is evicted between two uses.  The blocked list walks the
//    partition once per block of sources instead (the entries of a row are sorted by source, so a row meets a block in one
//    contiguous run); the rows gathered at any one time then belong to one or two blocks, which the L2 holds.  The price is one
//    partial sum per (row, block) and the pass that adds them.
// -------------------------------------------------------------------------------------
#define LIST_WINDOW 2048
#define FIXUP_HEAVY 16      /* k_spmm_fixup: rows with more runs than this are added by a thread block, the others by a thread per column */
#define LAST_RUN_MAX 64     /* small lists: up to this many runs the one that ends last adds them inside k_spmm (no second launch) */

// Longest run of a list with `entries` entries over `rows` rows.  Short runs balance a launch, but every run of a longer row costs a
// partial sum that is written and read again, so the length grows with the launch: 32 while the chip is not full and the longest
// run is the launch's duration, 64 / 128 / 256 from 1 / 8 / 16 M entries (on a skewed graph of 32 M entries, 64-entry runs
// moved 1.7 ms per epoch into the partial sums and gained 0.4 ms); and not below the mean row (rounded up to a power of two), so that an
// ordinary row of a dense graph stays in one piece (up to 512: 2 % of an epoch with 490 entries a row against 256).
//
// Small lists (chunk 32) have no second launch: the run of a row that ends last adds the row's partial sums (epoch of 900 nodes 99 -> 89 us,
// of 2708 nodes 285 -> 269).  Their chunk grows, up to 128, until the longest row has at most LAST_RUN_MAX runs; where 128 is not
// enough (a row above 8,192 entries) it stays at 32 and rows of more runs go to k_spmm_fixup.  Large lists keep k_spmm_fixup: the
// fence and ticket of every partial run cost more there than a launch (32 M entries: +4 %).
static int32_t list_chunk(int64_t entries, int64_t rows)
{
    const int64_t M = (int64_t)1 << 20;
    int32_t c = entries <= M ? 32 : entries <= 8 * M ? 64 : entries <= 16 * M ? 128 : 256;
    while (c < 512 && (int64_t)c * rows < entries) c <<= 1;
    return c;
}

struct ListRows {              // where the rows of a mode begin and end in its entry array
    const int64_t *ptr;
    const int32_t *inner_cnt;  // modes 1, 2
    int mode;
};
__device__ __forceinline__ void list_row(const ListRows &L, int64_t row, int64_t *rb, int64_t *re)
{
    const int64_t b = L.ptr[row], e = L.ptr[row + 1];
    *rb = L.mode == 2 ? b + L.inner_cnt[row] : L.mode == 4 ? b + row : b;
    *re = L.mode == 1 ? b + L.inner_cnt[row] : L.mode == 4 ? e + row + 1 : e;
}

__device__ __forceinline__ int64_t lower_bound_col(const int32_t *__restrict__ lenc, int64_t lo, int64_t hi, int64_t key)
{
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((int64_t)lenc[mid] < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// encoded column of source p of a partition whose sources are [n_rows inner rows from row0 ; halo rows from halo0]
__device__ __forceinline__ int64_t list_source_col(int64_t p, int64_t row0, int32_t n_rows, int32_t n, int64_t halo0)
{
    return p < n_rows ? row0 + p : (int64_t)n + halo0 + (p - n_rows);
}

struct ListPart {              // one partition of a list
    int64_t row0;              // its first row
    int32_t n_rows, n_blocks, min_run, n, chunk;
    int64_t halo0, block_rows;
};

// The run of entries [lo, hi) of `row` that is walked with source block j, or an empty run.  A row of `len` entries is cut into
// G = min(blocks, len / min_run) groups of consecutive blocks (a short row would otherwise leave a partial sum per block for
// a handful of entries each): group g covers blocks [ceil(g B / G), ceil((g + 1) B / G)) and its run is walked with the
// first of them.
__device__ __forceinline__ void list_run(const ListRows &L, const ListPart &P, const int32_t *__restrict__ lenc, int64_t row, int32_t j, int64_t *lo,
                                         int64_t *hi)
{
    int64_t rb, re;
    list_row(L, row, &rb, &re);
    if (P.n_blocks == 1) {
        *lo = rb;
        *hi = re;
        return;
    }
    int64_t G = P.min_run > 0 ? (re - rb) / P.min_run : P.n_blocks;
    G = G < 1 ? 1 : G > P.n_blocks ? P.n_blocks : G;
    const int64_t g = (int64_t)j * G / P.n_blocks;
    const int64_t j_first = (g * P.n_blocks + G - 1) / G, j_next = ((g + 1) * P.n_blocks + G - 1) / G;
    if (j != j_first) {
        *lo = *hi = rb;
        return;
    }
    *lo = j == 0 ? rb : lower_bound_col(lenc, rb, re, list_source_col((int64_t)j * P.block_rows, P.row0, P.n_rows, P.n, P.halo0));
    *hi = j_next >= P.n_blocks ? re : lower_bound_col(lenc, *lo, re, list_source_col(j_next * P.block_rows, P.row0, P.n_rows, P.n, P.halo0));
}

// count[j * n_rows + r] = items of row row0 + r in block j
__global__ void k_list_count(ListRows L, ListPart P, const int32_t *__restrict__ lenc, int32_t *__restrict__ count)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)P.n_rows * P.n_blocks) return;
    const int32_t j = (int32_t)(t / P.n_rows);
    int64_t lo, hi;
    list_run(L, P, lenc, P.row0 + (t - (int64_t)j * P.n_rows), j, &lo, &hi);
    count[t] = (int32_t)((hi - lo + P.chunk - 1) / P.chunk);
}

__global__ void k_list_row_totals(const int32_t *__restrict__ count, ListPart P, int32_t *__restrict__ tot, int32_t *__restrict__ slots,
                                  int32_t *__restrict__ multi, int32_t *__restrict__ heavy, int32_t last_max)
{
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= P.n_rows) return;
    int32_t s = 0;
    for (int32_t j = 0; j < P.n_blocks; ++j) s += count[(int64_t)j * P.n_rows + r];
    tot[P.row0 + r] = s;
    slots[P.row0 + r] = s > 1 ? s : 0;
    const bool fixup = s > 1 && s > last_max;
    multi[P.row0 + r] = fixup && s <= FIXUP_HEAVY ? 1 : 0;
    heavy[P.row0 + r] = fixup && s > FIXUP_HEAVY ? 1 : 0;
}

__global__ void k_list_fill(ListRows L, ListPart P, const int32_t *__restrict__ lenc, const int32_t *__restrict__ count,
                            const int64_t *__restrict__ item_off, const int32_t *__restrict__ tot, const int64_t *__restrict__ slot_off,
                            int4 *__restrict__ item)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)P.n_rows * P.n_blocks) return;
    const int32_t j = (int32_t)(t / P.n_rows), r = (int32_t)(t - (int64_t)j * P.n_rows);
    const int32_t c = count[t];
    if (c == 0) return;
    const int64_t row = P.row0 + r;
    int64_t lo, hi;
    list_run(L, P, lenc, row, j, &lo, &hi);
    int32_t before = 0;
    for (int32_t q = 0; q < j; ++q) before += count[(int64_t)q * P.n_rows + r];
    const bool multi = tot[row] > 1;
    const int64_t per = (hi - lo + c - 1) / c;   // equal runs
    for (int32_t q = 0; q < c; ++q) {
        const int64_t e0 = lo + q * per;
        const int32_t len = (int32_t)((hi - e0) < per ? (hi - e0) : per);
        item[item_off[t] + q] = make_int4((int32_t)row, multi ? (int32_t)(slot_off[row] + before + q) : -1, (int32_t)(uint32_t)(e0 & 0xffffffffll),
                                          (int32_t)((e0 >> 32) & 0xffff) | (len << 16));
    }
}

__global__ void k_list_rows(const int64_t *__restrict__ slot_off, const int32_t *__restrict__ multi, const int64_t *__restrict__ mrow_off,
                            const int32_t *__restrict__ heavy, const int64_t *__restrict__ hrow_off, int64_t n_rows, int32_t *__restrict__ slot0,
                            int32_t *__restrict__ mrows, int32_t *__restrict__ hrows)
{
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_rows) return;
    slot0[r] = (int32_t)slot_off[r];
    if (multi[r]) mrows[mrow_off[r]] = (int32_t)r;
    if (heavy[r]) hrows[hrow_off[r]] = (int32_t)r;
}

// out[0 .. M], [M+1 .. ], ..: first item, first partial slot, first row of a few runs and first row of many runs of every partition
__global__ void k_list_offsets(const int64_t *__restrict__ cbase, const int64_t *__restrict__ row_off, int32_t M, const int64_t *__restrict__ item_off,
                               const int64_t *__restrict__ slot_off, const int64_t *__restrict__ mrow_off, const int64_t *__restrict__ hrow_off,
                               int64_t *__restrict__ out)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m > M) return;
    out[m] = item_off[cbase[m]];
    out[M + 1 + m] = slot_off[row_off[m]];
    out[2 * (M + 1) + m] = mrow_off[row_off[m]];
    out[3 * (M + 1) + m] = hrow_off[row_off[m]];
}

// longest row of a list
__global__ void k_list_max(ListRows L, int64_t n_rows, int32_t *__restrict__ out)
{
    int32_t mx = 0;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n_rows; r += (int64_t)gridDim.x * blockDim.x) {
        int64_t rb, re;
        list_row(L, r, &rb, &re);
        mx = max(mx, (int32_t)(re - rb));
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(out, mx);
}

// orders the items of one window by length, longest first (a counting sort; the order among equal lengths does not matter)
__global__ void __launch_bounds__(256) k_list_sort(int4 *__restrict__ item, int64_t item0, int64_t n_items)
{
    constexpr int PER = LIST_WINDOW / 256;
    __shared__ int head[512];
    __shared__ int part[256];
    const int64_t w0 = item0 + (int64_t)blockIdx.x * LIST_WINDOW;
    const int64_t w1 = w0 + LIST_WINDOW < item0 + n_items ? w0 + LIST_WINDOW : item0 + n_items;
    int4 it[PER];
    head[threadIdx.x] = head[threadIdx.x + 256] = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int64_t i = w0 + threadIdx.x + 256 * k;
        if (i < w1) {
            it[k] = item[i];
            atomicAdd(&head[256 - (it[k].w >> 17)], 1);   // bin 0 = the longest possible run (512 entries); pairs of lengths share a bin
        }
    }
    __syncthreads();
    const int a = head[2 * threadIdx.x], b = head[2 * threadIdx.x + 1];
    part[threadIdx.x] = a + b;
    __syncthreads();
    for (int o = 1; o < 256; o <<= 1) {
        const int t = threadIdx.x >= o ? part[threadIdx.x - o] : 0;
        __syncthreads();
        part[threadIdx.x] += t;
        __syncthreads();
    }
    const int excl = part[threadIdx.x] - a - b;
    __syncthreads();
    head[2 * threadIdx.x] = excl;
    head[2 * threadIdx.x + 1] = excl + a;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int64_t i = w0 + threadIdx.x + 256 * k;
        if (i < w1) item[w0 + atomicAdd(&head[256 - (it[k].w >> 17)], 1)] = it[k];
    }
}

// Source blocking is used for partitions whose sources exceed `fit` bytes and whose rows meet a block with a run of at least
// `min_run` entries on average; inside such a partition a row of `len` entries is cut into at most len / row_run groups of
// blocks (list_run).  Defaults: blocks of 64 MiB; partitions from 192 MiB whose rows meet a block with 8 entries on average;
// row groups of at least 32 entries (measured on the 2.4 M-row graph: 0 / 8 / 16 / 32 / 64 entries give 6.47 / 6.26 / 6.11 /
// 6.06 / 6.13 ms per d = 100 launch; work items 4.39 M -> 3.53 M, partial-sum rows 2.37 M -> 1.30 M).  The environment variable SAT_SPMM_SRC_BLOCK = "<block bytes>[,<fit bytes>[,<min run>[,<row run>]]]" overrides them for a
// process (block bytes 0 = never blocked; row run 0 = every row cut at every block).
static ListKey list_key(int32_t d4, int mode)
{
    ListKey k;
    k.mode = mode;
    if (mode != 0) return k;
    int64_t block_bytes = (int64_t)64 << 20, fit_bytes = (int64_t)192 << 20;
    k.min_run = 8;
    k.row_run = 32;
    if (const char *e = getenv("SAT_SPMM_SRC_BLOCK")) {
        char *end = nullptr;
        block_bytes = strtoll(e, &end, 10);
        fit_bytes = 3 * block_bytes;
        if (end && *end == ',') fit_bytes = strtoll(end + 1, &end, 10);
        if (end && *end == ',') k.min_run = strtoll(end + 1, &end, 10);
        k.row_run = k.min_run;
        if (end && *end == ',') k.row_run = strtoll(end + 1, &end, 10);
    }
    if (block_bytes > 0) {
        k.block_rows = std::max<int64_t>(64, block_bytes / ((int64_t)d4 * 16) / 64 * 64);
        k.fit_rows = fit_bytes / ((int64_t)d4 * 16);
    }
    return k;
}

// source blocks of partition m (1: the plain walk)
static int64_t list_blocks_of(const sat_ctx *ctx, int m, const ListKey &k)
{
    const int64_t rows = ctx->h_inner_off[m + 1] - ctx->h_inner_off[m];
    const int64_t T = rows + (ctx->h_halo_off[m + 1] - ctx->h_halo_off[m]);
    if (k.block_rows <= 0 || T <= k.fit_rows || rows == 0) return 1;
    int64_t B = cdiv64(T, k.block_rows);
    if (B > 4096) B = 4096;
    // blocking pays where a row meets a block with a run of entries long enough to carry the extra partial sum
    const int64_t entries = ctx->h_lnnz_off[m + 1] - ctx->h_lnnz_off[m];
    return entries / (rows * B) >= k.min_run ? B : 1;
}

// A key under which no partition is blocked names the plain list (all such keys share it).
static ListKey list_key_effective(const sat_ctx *ctx, ListKey k)
{
    for (int m = 0; m < ctx->M; ++m)
        if (list_blocks_of(ctx, m, k) > 1) return k;
    ListKey plain;
    plain.mode = k.mode;
    return plain;
}

static sat_status list_build(sat_ctx *ctx, const ListKey &want, SpmmList **out)
{
    for (SpmmList &l : ctx->lists)
        if (l.asked == want) {
            *out = &l;
            return SAT_OK;
        }
    const ListKey key = list_key_effective(ctx, want);
    for (SpmmList &l : ctx->lists)
        if (l.key == key) {
            *out = &l;
            return SAT_OK;
        }
    const int32_t M = ctx->M, n = ctx->n;
    const int mode = key.mode;
    const bool halo_rows = mode >= 3;
    const int64_t n_rows = halo_rows ? ctx->nb : n;
    const int64_t cut = ctx->h_hrow_off.empty() ? 0 : ctx->h_hrow_off[M], all = ctx->nnz + n;
    const int64_t entries = mode == 0 ? all : mode == 1 ? all - cut : mode == 4 ? cut + ctx->nb : cut;
    int32_t chunk = list_chunk(entries, mode == 2 ? (ctx->n_slots > 0 ? ctx->n_slots : 1) : (n_rows > 0 ? n_rows : 1));
    ListRows L{halo_rows ? ctx->hrow_ptr : ctx->lrowptr, ctx->inner_cnt, mode};
    int32_t last_max = 0;
    if (chunk == 32 && n_rows > 0) {
        last_max = LAST_RUN_MAX;
        // a small launch: runs up to 128 entries where that lets the last run of the longest row do the adding (no second launch)
        int32_t longest = 0;
        SAT_CUDA(ctx, cudaMemsetAsync(ctx->d_flag + 3, 0, sizeof(int32_t), ctx->stream));
        k_list_max<<<(unsigned)std::min<int64_t>(cdiv64(n_rows, 256), ctx->sms), 256, 0, ctx->stream>>>(L, n_rows, ctx->d_flag + 3);
        SAT_LAUNCHED(ctx);
        SAT_CUDA(ctx, cudaMemcpyAsync(&longest, ctx->d_flag + 3, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
        SAT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        const int32_t want = (int32_t)cdiv64(cdiv64(longest, LAST_RUN_MAX), 8) * 8;
        if (want > chunk && want <= 128) chunk = want;
    }
    std::vector<ListPart> parts((size_t)M);
    std::vector<int64_t> off(2 * ((size_t)M + 1), 0);   // [first count | first row] of every partition
    int64_t *cbase = off.data(), *row_off = cbase + M + 1;
    for (int m = 0; m < M; ++m) {
        const int64_t a = halo_rows ? ctx->h_halo_off[m] : ctx->h_inner_off[m], b = halo_rows ? ctx->h_halo_off[m + 1] : ctx->h_inner_off[m + 1];
        const int64_t T = (b - a) + (ctx->h_halo_off[m + 1] - ctx->h_halo_off[m]);
        const int64_t B = list_blocks_of(ctx, m, key);
        parts[m] = ListPart{a, (int32_t)(b - a), (int32_t)B, (int32_t)(key.row_run < 0 ? 0 : key.row_run > (1 << 20) ? (1 << 20) : key.row_run), n, chunk,
                            ctx->h_halo_off[m], cdiv64(T > 0 ? T : 1, B)};   // equal blocks
        row_off[m + 1] = b;
        cbase[m + 1] = cbase[m] + (b - a) * B;
    }
    const int64_t total = cbase[M];
    // temporaries in one allocation, the list's arrays in another (an allocation costs more than the kernels that fill it)
    void *tmp = nullptr;
    SpmmList l;
    l.asked = want;
    l.key = key;
    l.last_max = last_max;
    auto cleanup = [&](bool drop) {
        cudaFree(tmp);
        if (drop) { cudaFree(l.item); cudaFree(l.slot0); }
    };
#define LB_TRY(expr)                       \
    do {                                   \
        sat_status s_ = (expr);            \
        if (s_ != SAT_OK) {                \
            cleanup(true);                 \
            return s_;                     \
        }                                  \
    } while (0)
#define LB_CUDA(call)                                                     \
    do {                                                                  \
        cudaError_t e_ = (call);                                          \
        if (e_ != cudaSuccess) {                                          \
            cleanup(true);                                                \
            return sat_check_cuda(ctx, e_, #call);                        \
        }                                                                 \
    } while (0)
    const int64_t words64 = (total + 1) + 3 * (n_rows + 1) + 6 * (M + 1);
    LB_CUDA(cudaMalloc(&tmp, (size_t)words64 * sizeof(int64_t) + (size_t)(total + 3 * n_rows) * sizeof(int32_t)));
    int64_t *item_off = (int64_t *)tmp, *slot_off = item_off + total + 1, *mrow_off = slot_off + n_rows + 1, *hrow_off = mrow_off + n_rows + 1,
            *d_off = hrow_off + n_rows + 1;
    int32_t *count = (int32_t *)(d_off + 6 * (M + 1)), *slots = count + total, *multi = slots + n_rows, *heavy = multi + n_rows;
    LB_CUDA(cudaMalloc((void **)&l.slot0, (size_t)(4 * (n_rows > 0 ? n_rows : 1)) * sizeof(int32_t)));
    l.tot = l.slot0 + n_rows;
    l.mrows = l.tot + n_rows;
    l.hrows = l.mrows + n_rows;
    LB_CUDA(cudaMemcpyAsync(d_off, off.data(), off.size() * sizeof(int64_t), cudaMemcpyHostToDevice, ctx->stream));
    for (int m = 0; m < M; ++m) {
        const ListPart &P = parts[m];
        if (P.n_rows == 0) continue;
        k_list_count<<<(unsigned)cdiv64((int64_t)P.n_rows * P.n_blocks, 256), 256, 0, ctx->stream>>>(L, P, ctx->lenc, count + cbase[m]);
        k_list_row_totals<<<(unsigned)cdiv64(P.n_rows, 256), 256, 0, ctx->stream>>>(count + cbase[m], P, l.tot, slots, multi, heavy, l.last_max);
        ctx->launches += 2;
    }
    LB_CUDA(cudaGetLastError());
    LB_TRY(sat_scan_i32(ctx, count, total, item_off));
    LB_TRY(sat_scan_i32(ctx, slots, n_rows, slot_off));
    LB_TRY(sat_scan_i32(ctx, multi, n_rows, mrow_off));
    LB_TRY(sat_scan_i32(ctx, heavy, n_rows, hrow_off));
    k_list_rows<<<(unsigned)cdiv64(n_rows > 0 ? n_rows : 1, 256), 256, 0, ctx->stream>>>(slot_off, multi, mrow_off, heavy, hrow_off, n_rows, l.slot0,
                                                                                         l.mrows, l.hrows);
    k_list_offsets<<<(unsigned)cdiv64(M + 1, 256), 256, 0, ctx->stream>>>(d_off, d_off + M + 1, M, item_off, slot_off, mrow_off, hrow_off, d_off + 2 * (M + 1));
    ctx->launches += 2;
    LB_CUDA(cudaGetLastError());
    l.off.assign(4 * ((size_t)M + 1), 0);
    LB_CUDA(cudaMemcpyAsync(l.off.data(), d_off + 2 * (M + 1), l.off.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
    LB_CUDA(cudaStreamSynchronize(ctx->stream));
    const int64_t n_items = l.off[M], n_slots = l.off[2 * M + 1];   // the entries of "partition M" are the totals
    if (n_items >= ((int64_t)1 << 31) || n_slots >= ((int64_t)1 << 31)) {
        cleanup(true);
        return sat_fail(ctx, SAT_EINVAL, "sat_spmm: too many work items");
    }
    LB_CUDA(cudaMalloc((void **)&l.item, (size_t)(n_items > 0 ? n_items : 1) * sizeof(int4)));
    for (int m = 0; m < M; ++m) {
        const ListPart &P = parts[m];
        if (P.n_rows == 0) continue;
        k_list_fill<<<(unsigned)cdiv64((int64_t)P.n_rows * P.n_blocks, 256), 256, 0, ctx->stream>>>(L, P, ctx->lenc, count + cbase[m], item_off + cbase[m],
                                                                                                   l.tot, slot_off, l.item);
        ctx->launches++;
    }
    for (int m = 0; m < M; ++m) {   // the windows of a partition are its own: a call on one partition walks whole windows
        const int64_t i0 = l.off[m], cnt = l.off[m + 1] - i0;
        if (cnt == 0) continue;
        k_list_sort<<<(unsigned)cdiv64(cnt, LIST_WINDOW), 256, 0, ctx->stream>>>(l.item, i0, cnt);
        ctx->launches++;
    }
    LB_CUDA(cudaGetLastError());
    LB_CUDA(cudaStreamSynchronize(ctx->stream));
#undef LB_TRY
#undef LB_CUDA
    cleanup(false);
    ctx->lists.push_back(std::move(l));
    *out = &ctx->lists.back();
    return SAT_OK;
}

// -------------------------------------------------------------------------------------
// One group of G lanes per work item; lane l owns float4 columns l, l + G, ..., l + (NV - 1) G of a slice of G NV columns
// (blockIdx.y).  Every lane reads the 8-byte entry itself (one broadcast transaction per group; sharing it through two
// shuffles was slower below 256 columns and equal there), U entries in flight, packed fp32 FMAs.
//   single-run rows write  out[row] = scale[row] * sum_e w_e * src[col_e]  (masked on request)
//   runs of longer rows write their un-scaled partial sum to `partial`, added in run order afterwards.
// Bound by the L2 -> SM path where the sources fit the L2 (dense graphs: 20 TB/s of gathered rows at d = 256, the rate of random
// rows out of an L2-resident buffer), by the latency of the short rows' chains (descriptor -> entries -> rows) and DRAM
// elsewhere.  Measured and dropped: cp.async rings (7 % faster than this at d = 256 on sparse graphs, 35 % slower on dense
// ones), one bulk copy per row (1.5-5 x slower), several rows per lane group with the entry stream walked across row ends (the
// kernel spills), descriptors of the next item fetched ahead (20-60 % slower), 6-8 blocks per SM at NV = 2 (fewer registers:
// fewer rows in flight).
// -------------------------------------------------------------------------------------
// result of row `row`, float4 column c, before the store: act(s * acc + bias + s1[row] v1 + s2[row] v2) (attention layer)
__device__ __forceinline__ float4 spmm_epilogue(const SpmmEpilogue &ep, int64_t row, int c, float4 r)
{
    float x[4] = {r.x, r.y, r.z, r.w};
    const float s1 = ep.s1 ? __ldg(ep.s1 + row) : 0.f, s2 = ep.s2 ? __ldg(ep.s2 + row) : 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int col = 4 * c + k;
        if (col >= ep.d) {   // padding columns hold zeros
            x[k] = 0.f;
            continue;
        }
        if (ep.bias) x[k] += __ldg(ep.bias + col);
        if (ep.s1) x[k] += s1 * __ldg(ep.v1 + col);
        if (ep.s2) x[k] += s2 * __ldg(ep.v2 + col);
        if (ep.relu) x[k] = fmaxf(x[k], 0.f);
    }
    const float4 out = make_float4(x[0], x[1], x[2], x[3]);
    if (ep.push) {
        const int32_t slot = __ldg(ep.push_slot + row);
        if (slot >= 0) *reinterpret_cast<float4 *>(ep.push + slot * ep.ld_push + 4 * c) = out;
    }
    return out;
}

// the row that is added to row `row`, column c
__device__ __forceinline__ void spmm_add(const SpmmAdd &add, int64_t row, int c, float4 &r)
{
    const int32_t slot = __ldg(add.slot + row);
    if (slot < 0) return;
    const float4 x = ld4(add.rows + slot * add.ld + 4 * c);
    r.x += x.x;
    r.y += x.y;
    r.z += x.z;
    r.w += x.w;
}

// largest magnitude of the columns 4 c .. 4 c + 3 that a row of d columns has
__device__ __forceinline__ float spmm_largest(float m, const float4 &r, int c, int32_t d)
{
    if (4 * c + 3 < d) return fmaxf(fmaxf(m, fmaxf(fabsf(r.x), fabsf(r.y))), fmaxf(fabsf(r.z), fabsf(r.w)));
    if (4 * c < d) m = fmaxf(m, fabsf(r.x));
    if (4 * c + 1 < d) m = fmaxf(m, fabsf(r.y));
    if (4 * c + 2 < d) m = fmaxf(m, fabsf(r.z));
    return m;
}

// Leaves the largest magnitude of a slice of row `row`: by row, or (attention layer) by the row's ring slot, where it has one, in the first of the two parts that
// stand for 256 columns there.
template <bool EPI>
__device__ __forceinline__ void spmm_put_max(const SpmmEpilogue &ep, int64_t row, unsigned slice, uint32_t m)
{
    if (EPI) {
        const int32_t slot = __ldg(ep.push_slot + row);
        if (slot < 0) return;
        ep.row_max.p[2 * slice * ep.row_max.stride + slot] = m;
        ep.row_max.p[(2 * slice + 1) * ep.row_max.stride + slot] = 0u;
    } else {
        ep.row_max.p[slice * ep.row_max.stride + row] = m;
    }
}

// K entries: their columns and weights, their rows (all in flight together), the sums
template <int G, int NV, int K, typename F>
__device__ __forceinline__ void spmm_step(const int2 *__restrict__ ents, const F &row_of, int col, int32_t d4, float4 (&acc)[NV])
{
    int2 q[K];
#pragma unroll
    for (int u = 0; u < K; ++u) q[u] = __ldg(ents + u);
    float4 x[K][NV];
#pragma unroll
    for (int u = 0; u < K; ++u) {
        const float4 *src = row_of(q[u].x);
#pragma unroll
        for (int v = 0; v < NV; ++v) x[u][v] = col + v * G < d4 ? __ldg(src + v * G) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < K; ++u)
#pragma unroll
        for (int v = 0; v < NV; ++v) fma4(acc[v], __int_as_float(q[u].y), x[u][v]);
}

template <int G, int NV, int U, int MINB, bool EPI, bool MAX>
__global__ void __launch_bounds__(256, MINB)
k_spmm(const int4 *__restrict__ items, int32_t n_items, int64_t slot_base, const int2 *__restrict__ ent, const float *__restrict__ scale, int32_t n,
       int32_t d4, const float *__restrict__ in_base, int64_t ld_in, const float *__restrict__ halo_base, int64_t ld_halo, float *__restrict__ out_base,
       int64_t ld_out, float *partial, const int32_t *__restrict__ slot0, const int32_t *__restrict__ tot, int32_t *ticket,
       int32_t last_max, const uint32_t *__restrict__ omask, int32_t omask_words, SpmmEpilogue ep, DbgLimits dbg)
{
    sat_grid_wait();
    const int lane = threadIdx.x & (G - 1);
    const int64_t gid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    if (gid >= n_items) return;
    const int col = blockIdx.y * (G * NV) + lane;
    const int4 it = __ldg(items + gid);
    const int2 *__restrict__ ents = ent + ((int64_t)(uint32_t)it.z | ((int64_t)(it.w & 0xffff) << 32));
    const int32_t len = it.w >> 16;
    // columns below n index the inner matrix, the others the halo matrix (addressed from its virtual row -n): one multiply-add
    // per row either way
    const uint32_t li = (uint32_t)(ld_in >> 2), lh = (uint32_t)(ld_halo >> 2);
    const float4 *in4 = reinterpret_cast<const float4 *>(in_base) + col;
    const float4 *halo4 = reinterpret_cast<const float4 *>(halo_base) + col - (int64_t)n * lh;
    auto row_of = [&](int32_t c) {
        const bool in = c < n;
        const uint32_t i = (uint32_t)(in ? SAT_IDX((int64_t)c, dbg.src_lo, dbg.src_hi, dbg.status)
                                         : n + SAT_IDX((int64_t)(c - n), dbg.halo_lo, dbg.halo_hi, dbg.status));
        return (in ? in4 : halo4) + (uint64_t)i * (in ? li : lh);
    };
    float4 acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    int32_t e = 0;
    for (; e + U <= len; e += U) spmm_step<G, NV, U>(ents + e, row_of, col, d4, acc);
    // the remainder by halves: each step is one chain of latencies (entry -> row), whatever its width
    if (U > 4 && ((len - e) & 4)) {
        spmm_step<G, NV, U < 4 ? U : 4>(ents + e, row_of, col, d4, acc);
        e += 4;
    }
    if ((len - e) & 2) {
        spmm_step<G, NV, 2>(ents + e, row_of, col, d4, acc);
        e += 2;
    }
    if ((len - e) & 1) spmm_step<G, NV, 1>(ents + e, row_of, col, d4, acc);
    float4 *pr = reinterpret_cast<float4 *>(partial) + ((int64_t)it.y - slot_base) * d4 + col;
    if (it.y >= 0) {
        // a run of a longer row: leave the partial sum.  Small launches: the group that finishes a row last (by its ticket) adds all of
        // them in run order.  (In large ones the fences in front of the tickets cost more than the second launch.)
#pragma unroll
        for (int v = 0; v < NV; ++v)
            if (col + v * G < d4) pr[v * G] = acc[v];
        if (!MAX && last_max == 0) return;
        const bool last = !MAX || last_max > 0;
        const int32_t first = last ? __ldg(slot0 + it.x) : 0, cnt = last ? __ldg(tot + it.x) : 0;
        if (cnt > last_max || !last) {   // k_spmm_fixup, which raises the row's maximum from zero
            if (MAX && lane == 0) spmm_put_max<EPI>(ep, it.x, blockIdx.y, 0u);
            return;
        }
        const unsigned mask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (threadIdx.x & 31 & ~(G - 1));
        __threadfence();
        __syncwarp(mask);
        int32_t before = 0;
        int32_t *t = ticket + (first - slot_base) * gridDim.y + blockIdx.y;
        if (lane == 0) {
            before = atomicAdd(t, 1);
            if (before == cnt - 1) *t = 0;   // zero again for the next launch
        }
        before = __shfl_sync(mask, before, 0, G);
        if (before != cnt - 1) return;
        __threadfence();
        const float4 *p0 = reinterpret_cast<const float4 *>(partial) + ((int64_t)first - slot_base) * d4 + col;
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int32_t q = 0; q < cnt; q += 4) {
            float4 x[4][NV];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < NV; ++v)
                    x[u][v] = q + u < cnt && col + v * G < d4 ? __ldcg(p0 + (int64_t)(q + u) * d4 + v * G) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    acc[v].x += x[u][v].x;
                    acc[v].y += x[u][v].y;
                    acc[v].z += x[u][v].z;
                    acc[v].w += x[u][v].w;
                }
        }
    }
    const int64_t row = SAT_IDX((int64_t)it.x, dbg.out_lo, dbg.out_hi, dbg.status);
    const float s = EPI ? 1.f : __ldg(scale + row);
    float4 *o = reinterpret_cast<float4 *>(out_base + row * ld_out) + col;
    float largest = 0.f;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        if (col + v * G < d4) {
            float4 r = make_float4(s * acc[v].x, s * acc[v].y, s * acc[v].z, s * acc[v].w);
            if (EPI) r = spmm_epilogue(ep, row, col + v * G, r);
            else {
                if (ep.add.rows) spmm_add(ep.add, row, col + v * G, r);
                if (omask) mask4(r, omask, row * omask_words, col + v * G);
            }
            o[v * G] = r;
            if (MAX) largest = spmm_largest(largest, r, col + v * G, ep.d);
        }
    }
    if (MAX) {
        unsigned lane_id;
        asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane_id));   // (not kept through the loops)
        const uint32_t m = __reduce_max_sync(G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (lane_id & ~(unsigned)(G - 1)), __float_as_uint(largest));
        if ((lane_id & (G - 1)) == 0) spmm_put_max<EPI>(ep, row, blockIdx.y, m);
    }
}

// Rows with several runs: the partial sums are added in a fixed order, scaled and stored.  The first blocks take the rows of many
// runs (a hub row of tens of thousands of entries has hundreds, and one thread walking them was the launch: 85 us), one block
// per row and 32 columns: warp w adds the w-th eighth of the runs, the eighths are added in order through shared memory.  The
// other rows take a thread per column.  Eight loads in flight either way.
__device__ __forceinline__ float4 fixup_range(const float4 *__restrict__ p, int32_t q0, int32_t q1, int32_t d4)
{
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int32_t q = q0; q < q1; q += 8) {
        float4 x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = q + u < q1 ? p[(int64_t)(q + u) * d4] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            a.x += x[u].x;
            a.y += x[u].y;
            a.z += x[u].z;
            a.w += x[u].w;
        }
    }
    return a;
}

template <bool MAX>
__global__ void __launch_bounds__(256)
k_spmm_fixup(const int32_t *__restrict__ hrows, int32_t n_hrows, const int32_t *__restrict__ mrows, int32_t n_mrows, const int32_t *__restrict__ slot0,
             const int32_t *__restrict__ tot, int64_t slot_base, const float *__restrict__ scale, int32_t d4, const float *__restrict__ partial,
             float *__restrict__ out_base, int64_t ld_out, const uint32_t *__restrict__ omask, int32_t omask_words, SpmmEpilogue ep, DbgLimits dbg)
{
    sat_grid_wait();
    __shared__ float4 part[8][32];
    const int32_t slabs = (d4 + 31) / 32;
    const int64_t n_hblk = (int64_t)n_hrows * slabs;
    int64_t row;
    int c;
    float4 a;
    if (blockIdx.x < n_hblk) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        row = SAT_IDX((int64_t)hrows[blockIdx.x / slabs], dbg.out_lo, dbg.out_hi, dbg.status);
        c = (int)(blockIdx.x % slabs) * 32 + lane;
        const int32_t cnt = tot[row];
        const float4 *p = reinterpret_cast<const float4 *>(partial) + ((int64_t)slot0[row] - slot_base) * d4 + c;
        part[warp][lane] = c < d4 ? fixup_range(p, cnt * warp / 8, cnt * (warp + 1) / 8, d4) : make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        if (warp != 0 || c >= d4) return;
        a = part[0][lane];
#pragma unroll
        for (int w = 1; w < 8; ++w) {
            const float4 x = part[w][lane];
            a.x += x.x;
            a.y += x.y;
            a.z += x.z;
            a.w += x.w;
        }
    } else {
        const int64_t t = ((int64_t)blockIdx.x - n_hblk) * blockDim.x + threadIdx.x;
        const int64_t i = sat_div(t, d4);
        c = (int)(t - i * d4);
        if (i >= n_mrows) return;
        row = SAT_IDX((int64_t)mrows[i], dbg.out_lo, dbg.out_hi, dbg.status);
        a = fixup_range(reinterpret_cast<const float4 *>(partial) + ((int64_t)slot0[row] - slot_base) * d4 + c, 0, tot[row], d4);
    }
    const float s = scale ? scale[row] : 1.f;
    float4 r = make_float4(s * a.x, s * a.y, s * a.z, s * a.w);
    if (!scale) r = spmm_epilogue(ep, row, c, r);
    else {
        if (ep.add.rows) spmm_add(ep.add, row, c, r);
        if (omask) mask4(r, omask, row * omask_words, c);
    }
    *reinterpret_cast<float4 *>(out_base + row * ld_out + 4 * c) = r;
    if (MAX) {   // the lanes of a warp that hold columns of the same row raise it together
        const unsigned same = __match_any_sync(__activemask(), (int32_t)row);
        const uint32_t m = __reduce_max_sync(same, __float_as_uint(spmm_largest(0.f, r, c, ep.d)));
        if ((threadIdx.x & 31) == __ffs((int)same) - 1) {
            const int64_t at = scale ? row : __ldg(ep.push_slot + row);
            if (at >= 0) atomicMax(ep.row_max.p + at, m);
        }
    }
}

struct SpmmArgs {
    const int2 *ent;
    const float *scale;          // per row of the list; null: no scaling, and the epilogue `ep` instead of the mask
    SpmmEpilogue ep;
    int32_t n;                   // columns below n address `in`, the others `halo`
    const float *in_base, *halo_base;
    int32_t ld_in, ld_halo;
    float *out_base;
    int32_t ld_out;
    const uint32_t *omask;
    int32_t omask_words;
    DbgRange src, halo, out;
};

template <int G, int NV, int U, int MINB, bool MAX = false>
static void launch_spmm(sat_ctx *ctx, const SpmmList &l, const int4 *items, int32_t n_items, int64_t slot_base, int32_t d4, const SpmmArgs &a, float *partial)
{
    dim3 grid((unsigned)cdiv64((int64_t)n_items * G, 256), (unsigned)cdiv64(d4, G * NV));
    const DbgLimits dbg = dbg_limits(a.src, a.halo, a.out, ctx->d_flag + 1);
    if (a.scale)
        sat_pdl(ctx->stream, k_spmm<G, NV, U, MINB, false, MAX>, grid, 256, 0)(items, n_items, slot_base, a.ent, a.scale, a.n, d4, a.in_base, a.ld_in, a.halo_base, a.ld_halo,
                                                                     a.out_base, a.ld_out, partial, l.slot0, l.tot, (int32_t *)ctx->buf_ticket.p, l.last_max, a.omask, a.omask_words, a.ep, dbg);
    else
        sat_pdl(ctx->stream, k_spmm<G, NV, U, MINB, true, MAX>, grid, 256, 0)(items, n_items, slot_base, a.ent, a.scale, a.n, d4, a.in_base, a.ld_in, a.halo_base, a.ld_halo,
                                                                    a.out_base, a.ld_out, partial, l.slot0, l.tot, (int32_t *)ctx->buf_ticket.p, l.last_max, a.omask, a.omask_words, a.ep, dbg);
}

// walks partitions [v.p0, v.p1) of a list
static sat_status run_list(sat_ctx *ctx, const PartView &v, const SpmmList &l, int32_t d4, const SpmmArgs &a)
{
    const int M1 = ctx->M + 1;
    const int64_t item0 = l.off[v.p0], n_items = l.off[v.p1] - item0;
    const int64_t slot_base = l.off[M1 + v.p0], n_slots = l.off[M1 + v.p1] - slot_base;
    const int64_t mrow0 = l.off[2 * M1 + v.p0], n_mrows = l.off[2 * M1 + v.p1] - mrow0;
    const int64_t hrow0 = l.off[3 * M1 + v.p0], n_hrows = l.off[3 * M1 + v.p1] - hrow0;
    if (n_items == 0) return SAT_OK;
    float *partial = nullptr;
    if (n_slots > 0) {
        // sized for all partitions at once: calls on one partition after the other would grow it again and again
        SAT_TRY(sat_ensure(ctx, ctx->buf_partial, (size_t)l.off[M1 + ctx->M] * d4 * 16));
        partial = (float *)ctx->buf_partial.p;
        // a ticket per (slot, column slice), all zero between launches
        const size_t need = l.last_max > 0 ? (size_t)l.off[M1 + ctx->M] * cdiv64(d4, 64) * sizeof(int32_t) : 0;
        if (need > ctx->buf_ticket.bytes) {
            SAT_TRY(sat_ensure(ctx, ctx->buf_ticket, need));
            SAT_CUDA(ctx, cudaMemsetAsync(ctx->buf_ticket.p, 0, ctx->buf_ticket.bytes, ctx->stream));
        }
    }
    // Lane groups by width.  Above 256 columns the launch walks slices of 256: a slice's sources fit the L2 twice as often, and two
    // passes of the 2-vector shape beat one pass of a 4-vector one (d = 512: 484 -> 391 us on the sparse graph, 1,334 -> 1,190 on
    // the dense one).
    const int4 *items = l.item + item0;
#define ARGS ctx, l, items, (int32_t)n_items, slot_base, d4, a, partial
    // A launch of at most three blocks of eight warps per SM, a warp per item, leaves most of the chip idle and is as long as its longest
    // run: eight entries in flight per step then, for more registers (epoch of 2,048 nodes 90.6 -> 84.4 us; 6,000 nodes and upward the
    // same, one drawn graph 515 -> 522)
    const bool small = n_items * 32 <= ctx->sms * 768;
    if (a.ep.row_max.p) small ? launch_spmm<32, 2, 8, 3, true>(ARGS) : launch_spmm<32, 2, 4, 5, true>(ARGS);   // (sat_tc_half: wide rows)
    else if (d4 <= 4) small ? launch_spmm<4, 1, 8, 3>(ARGS) : launch_spmm<4, 1, 4, 6>(ARGS);
    else if (d4 <= 8) small ? launch_spmm<8, 1, 8, 3>(ARGS) : launch_spmm<8, 1, 4, 6>(ARGS);
    else if (d4 <= 16) small ? launch_spmm<16, 1, 8, 3>(ARGS) : launch_spmm<16, 1, 4, 6>(ARGS);
    else if (d4 <= 32) small ? launch_spmm<16, 2, 8, 3>(ARGS) : launch_spmm<16, 2, 4, 5>(ARGS);
    else small ? launch_spmm<32, 2, 8, 3>(ARGS) : launch_spmm<32, 2, 4, 5>(ARGS);
#undef ARGS
    SAT_LAUNCHED(ctx);
    if (n_hrows + n_mrows > 0) {
        sat_pdl(ctx->stream, a.ep.row_max.p ? k_spmm_fixup<true> : k_spmm_fixup<false>, (unsigned)(n_hrows * cdiv64(d4, 32) + cdiv64(n_mrows * d4, 256)), 256, 0)(
            l.hrows + hrow0, (int32_t)n_hrows, l.mrows + mrow0, (int32_t)n_mrows, l.slot0, l.tot, slot_base, a.scale, d4, partial, a.out_base, a.ld_out, a.omask,
            a.omask_words, a.ep, dbg_limits(a.src, a.halo, a.out, ctx->d_flag + 1));
        SAT_LAUNCHED(ctx);
    }
    return SAT_OK;
}

// entries with halo columns as n + global node id or n + cache slot (`halo_id` of the halo position)
__global__ void k_ent_by_id(const int2 *__restrict__ ent, const int32_t *__restrict__ halo_id, int64_t count, int32_t n, int2 *__restrict__ out)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= count) return;
    const int2 q = ent[e];
    out[e] = make_int2(q.x < n ? q.x : n + halo_id[q.x - n], q.y);
}

// entries with every column as a global node id (inner columns through the partition-major order, halo columns through the halo list)
__global__ void k_ent_all_gid(const int2 *__restrict__ ent, const int32_t *__restrict__ perm, const int32_t *__restrict__ halo_gid,
                              int64_t count, int32_t n, int2 *__restrict__ out)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= count) return;
    const int2 q = ent[e];
    out[e] = make_int2(q.x < n ? perm[q.x] : halo_gid[q.x - n], q.y);
}

sat_status sat_spmm(sat_ctx *ctx, const PartView &v, int inner_only, int32_t d, const float *in_base, int32_t ld_in,
                    const float *halo_base, int32_t ld_halo, float *out_base, int32_t ld_out, const uint32_t *omask, int32_t omask_words,
                    SpmmHalo halo_kind, bool in_global, const SpmmAdd &add, const RowMaxOut &row_max)
{
    if (v.n_rows == 0) return SAT_OK;
    const int32_t d4 = (d + 3) / 4;
    SpmmArgs a;
    a.ent = ctx->ent;
    a.halo = DbgRange{v.halo0, v.halo0 + v.n_halo};
    a.src = DbgRange{v.row0, (int64_t)v.row0 + v.n_rows};
    a.out = a.src;
    const int64_t lnnz = ctx->nnz + ctx->n;
    if (in_global) {
        // inner and halo rows both come from one matrix over all nodes (`in_base`, global id order): every column becomes a
        // node id (all below n, so the kernel takes its inner branch for each of them)
        if (!ctx->ent_all_gid) {
            SAT_CUDA(ctx, cudaMalloc((void **)&ctx->ent_all_gid, (size_t)lnnz * sizeof(int2)));
            k_ent_all_gid<<<(unsigned)cdiv64(lnnz, 256), 256, 0, ctx->stream>>>(ctx->ent, ctx->perm, ctx->halo_gid, lnnz, ctx->n, ctx->ent_all_gid);
            SAT_LAUNCHED(ctx);
        }
        a.ent = ctx->ent_all_gid;
        a.src = DbgRange{0, ctx->n};
        a.halo = DbgRange{0, 0};
    } else if (halo_kind != SpmmHalo::by_position && inner_only == 0) {
        const bool slot = halo_kind == SpmmHalo::by_slot;
        int2 *&ent = slot ? ctx->ent_slot : ctx->ent_gid;
        if (!ent) {
            SAT_CUDA(ctx, cudaMalloc((void **)&ent, (size_t)lnnz * sizeof(int2)));
            k_ent_by_id<<<(unsigned)cdiv64(lnnz, 256), 256, 0, ctx->stream>>>(ctx->ent, slot ? ctx->halo_slot : ctx->halo_gid, lnnz, ctx->n, ent);
            SAT_LAUNCHED(ctx);
        }
        a.ent = ent;
        a.halo = DbgRange{0, slot ? ctx->n_slots : ctx->n};
    }
    // algorithmic bytes: column ids + row offsets + dinv, every source row once, every output row once (a halo source over
    // all nodes holds at most n distinct rows)
    const double n_halo_src = halo_kind != SpmmHalo::by_position && v.n_halo > ctx->n ? (double)ctx->n : (double)v.n_halo;
    double n_src = inner_only == 1 ? (double)v.n_rows : inner_only == 2 ? n_halo_src : (double)v.n_rows + n_halo_src;
    if (in_global && n_src > ctx->n) n_src = ctx->n;
    // the backward reads the inner prefix of every row, the transposed predictor convolution the halo suffix
    const double n_ent = (double)(inner_only == 1 ? v.lnnz - v.hnnz : inner_only == 2 ? v.hnnz : v.lnnz);
    ProfScope prof(ctx, inner_only ? SATK_SPMM_BWD : SATK_SPMM_FWD,
                   4.0 * n_ent + 12.0 * v.n_rows + 4.0 * n_src + 4.0 * d * (n_src + v.n_rows), 2.0 * n_ent * d);
    SpmmList *l = nullptr;
    SAT_TRY(list_build(ctx, list_key(d4, inner_only), &l));
    a.scale = ctx->dinv_enc;
    a.ep.add = add;
    a.ep.row_max = row_max;
    a.ep.d = d;
    a.n = ctx->n;
    a.in_base = in_base;
    a.ld_in = ld_in;
    a.halo_base = halo_base;
    a.ld_halo = ld_halo;
    a.out_base = out_base;
    a.ld_out = ld_out;
    a.omask = omask;
    a.omask_words = omask_words;
    return run_list(ctx, v, *l, d4, a);
}

sat_status sat_spmm_entries(sat_ctx *ctx, const PartView &v, int mode, int32_t d, const int2 *ent, const float *in_base, int32_t ld_in,
                            const float *halo_base, int32_t ld_halo, float *out_base, int32_t ld_out, const SpmmEpilogue &ep)
{
    SpmmList *l = nullptr;
    SAT_TRY(list_build(ctx, list_key((d + 3) / 4, mode), &l));
    SpmmArgs a;
    a.ent = ent;
    a.scale = nullptr;
    a.ep = ep;
    a.ep.d = d;
    a.n = mode == 0 ? ctx->n : INT32_MAX;
    a.in_base = in_base;
    a.ld_in = ld_in;
    a.halo_base = halo_base;
    a.ld_halo = ld_halo;
    a.out_base = out_base;
    a.ld_out = ld_out;
    a.omask = nullptr;
    a.omask_words = 0;
    a.src = DbgRange{v.row0, (int64_t)v.row0 + v.n_rows};
    a.halo = DbgRange{v.halo0, v.halo0 + v.n_halo};
    a.out = mode == 3 ? a.halo : a.src;
    return run_list(ctx, v, *l, (d + 3) / 4, a);
}

sat_status sat_spmm_items(sat_ctx *ctx, const PartView &v, int mode, int32_t d, const int4 **items, int64_t *n_items)
{
    SpmmList *l = nullptr;
    SAT_TRY(list_build(ctx, list_key((d + 3) / 4, mode), &l));
    *items = l->item + l->off[v.p0];
    *n_items = l->off[v.p1] - l->off[v.p0];
    return SAT_OK;
}

extern "C" sat_status sat_spmm_plan(sat_ctx *ctx, int32_t part, int32_t d, int32_t *n_blocks, int64_t *n_items, int64_t *n_partial_rows)
{
    CHECK_CTX(ctx);
    PartView v;
    SAT_TRY(sat_part_view(ctx, part, &v));
    if (d < 1) return sat_fail(ctx, SAT_EINVAL, "sat_spmm_plan: d = %d", d);
    SpmmList *l = nullptr;
    SAT_TRY(list_build(ctx, list_key((d + 3) / 4, 0), &l));
    int32_t nb = 1;
    for (int m = v.p0; m < v.p1; ++m) nb = std::max<int32_t>(nb, (int32_t)list_blocks_of(ctx, m, l->key));
    if (n_blocks) *n_blocks = nb;
    if (n_items) *n_items = l->off[v.p1] - l->off[v.p0];
    if (n_partial_rows) *n_partial_rows = l->off[ctx->M + 1 + v.p1] - l->off[ctx->M + 1 + v.p0];
    return SAT_OK;
}

// -------------------------------------------------------------------------------------
// Halo-row products (rows = halo entries of the partition, columns = their neighbours
// inside the partition):
//   out[j] = dinv[u_j] * ( [self] dinv[u_j] * src[halo_slot_j] + sum_e dinv[v_e] * src[idx_e] )
// idx_e is the partition-major row of v_e (by_slot = 0, no self term) or its cache slot (by_slot = 1, with the self term, which is
// the first entry of the row).  Used for the predictor's graph convolution on the LSTM state (by slot) and for the optional halo
// gradient P_out^T G_AGG and the gradient-side history (by row).
// -------------------------------------------------------------------------------------
__global__ void k_hent(const int64_t *__restrict__ hrow_ptr, const int32_t *__restrict__ hrow_col, const float *__restrict__ hrow_w, int64_t nb,
                       const int32_t *__restrict__ halo_slot, const float *__restrict__ dinv_halo, int self, int2 *__restrict__ out)
{
    const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (j >= nb) return;
    const int64_t b = hrow_ptr[j], e = hrow_ptr[j + 1];
    int2 *o = out + (self ? b + j + 1 : b);
    for (int64_t i = b + lane; i < e; i += 32) o[i - b] = make_int2(hrow_col[i], __float_as_int(hrow_w[i]));
    if (self && lane == 0) o[-1] = make_int2(halo_slot[j], __float_as_int(dinv_halo[j]));
}

sat_status sat_spmm_hrow(sat_ctx *ctx, const PartView &v, int32_t d, const float *src_base, int32_t ld_src, int by_slot, float *out_base,
                         int32_t ld_out)
{
    if (v.n_halo == 0) return SAT_OK;
    const int32_t d4 = (d + 3) / 4;
    int2 *&ent = by_slot ? ctx->hent_slot : ctx->hent_pos;
    if (!ent) {
        SAT_CUDA(ctx, cudaMalloc((void **)&ent, (size_t)(ctx->nnz_cut + (by_slot ? ctx->nb : 0)) * sizeof(int2)));
        k_hent<<<(unsigned)cdiv64(ctx->nb * 32, 256), 256, 0, ctx->stream>>>(ctx->hrow_ptr, by_slot ? ctx->hrow_slot : ctx->hrow_pos, ctx->hrow_w, ctx->nb,
                                                                             ctx->halo_slot, ctx->dinv_enc + ctx->n, by_slot, ent);
        SAT_LAUNCHED(ctx);
    }
    // algorithmic bytes: column + weight per entry, row offsets / slot / dinv per halo row, every source row once (the
    // boundary rows of the selection, plus the halo nodes' own rows for the self term), every output row once
    const double n_src = (double)v.n_push + (by_slot ? (double)v.n_halo : 0.0);
    ProfScope prof(ctx, SATK_SPMM_HROW, 8.0 * (double)v.hnnz + 12.0 * (double)v.n_halo + 4.0 * d * (n_src + (double)v.n_halo),
                   2.0 * d * ((double)v.hnnz + (by_slot ? (double)v.n_halo : 0.0)));
    SpmmList *l = nullptr;
    SAT_TRY(list_build(ctx, list_key(d4, by_slot ? 4 : 3), &l));
    SpmmArgs a;
    a.ent = ent;
    a.scale = ctx->dinv_enc + ctx->n;
    a.n = INT32_MAX;
    a.in_base = src_base;
    a.ld_in = ld_src;
    a.halo_base = nullptr;
    a.ld_halo = 0;
    a.out_base = out_base;
    a.ld_out = ld_out;
    a.omask = nullptr;
    a.omask_words = 0;
    a.src = by_slot ? DbgRange{0, ctx->n_slots} : DbgRange{v.row0, (int64_t)v.row0 + v.n_rows};
    a.halo = DbgRange{0, 0};
    a.out = DbgRange{v.halo0, v.halo0 + v.n_halo};
    return run_list(ctx, v, *l, d4, a);
}

// -------------------------------------------------------------------------------------
// row gather / scatter (pull of raw features, push into the cache, identity predictor)
// -------------------------------------------------------------------------------------
__global__ void k_gather_rows(const int32_t *__restrict__ idx, int64_t count, int32_t d4, const float *__restrict__ src, int64_t ld_src,
                              float *__restrict__ out, int64_t ld_out, DbgLimits dbg)
{
    sat_grid_wait();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = sat_div(t, d4);
    const int c = (int)(t - i * d4);
    if (i >= count) return;
    const float4 x = ld4(src + SAT_IDX((int64_t)idx[i], dbg.src_lo, dbg.src_hi, dbg.status) * ld_src + 4 * c);
    *reinterpret_cast<float4 *>(out + i * ld_out + 4 * c) = x;
}

sat_status sat_gather(sat_ctx *ctx, const int32_t *idx, int64_t count, int32_t d, const float *src, int32_t ld_src, float *out,
                      int32_t ld_out, DbgRange src_rows)
{
    if (count == 0) return SAT_OK;
    const int32_t d4 = (d + 3) / 4;
    ProfScope prof(ctx, SATK_GATHER, (8.0 * d + 4.0) * (double)count, 0.0);
    sat_pdl(ctx->stream, k_gather_rows, (unsigned)cdiv64(count * d4, 256), 256, 0)(idx, count, d4, src, ld_src, out, ld_out,
                                                                              dbg_limits(src_rows, DbgRange{0, 0}, DbgRange{0, count}, ctx->d_flag + 1));
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

__global__ void k_scatter_rows(const int32_t *__restrict__ src_row, const int32_t *__restrict__ dst_row, int64_t count, int32_t d4,
                               const float *__restrict__ src_base, int64_t ld_src, float *__restrict__ dst, int64_t ld_dst, DbgLimits dbg)
{
    sat_grid_wait();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = sat_div(t, d4);
    const int c = (int)(t - i * d4);
    if (i >= count) return;
    const float4 x = ld4(src_base + SAT_IDX((int64_t)src_row[i], dbg.src_lo, dbg.src_hi, dbg.status) * ld_src + 4 * c);
    *reinterpret_cast<float4 *>(dst + SAT_IDX((int64_t)dst_row[i], dbg.out_lo, dbg.out_hi, dbg.status) * ld_dst + 4 * c) = x;
}

// the same, a warp per row, leaving the largest magnitude of every row by its destination (the first of `parts` parts; the others hold zeros)
__global__ void __launch_bounds__(256)
k_scatter_rows_max(const int32_t *__restrict__ src_row, const int32_t *__restrict__ dst_row, int64_t count, int32_t d, const float *__restrict__ src_base,
                   int64_t ld_src, float *__restrict__ dst, int64_t ld_dst, RowMaxOut row_max, int32_t parts, DbgLimits dbg)
{
    sat_grid_wait();
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= count) return;
    const float *src = src_base + SAT_IDX((int64_t)src_row[i], dbg.src_lo, dbg.src_hi, dbg.status) * ld_src;
    const int64_t slot = SAT_IDX((int64_t)dst_row[i], dbg.out_lo, dbg.out_hi, dbg.status);
    float largest = 0.f;
#pragma unroll 4
    for (int c = lane; 4 * c < d; c += 32) {
        const float4 x = ld4(src + 4 * c);
        reinterpret_cast<float4 *>(dst + slot * ld_dst)[c] = x;
        largest = spmm_largest(largest, x, c, d);
    }
    const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(largest));
    for (int32_t p = lane; p < parts; p += 32) row_max.p[p * row_max.stride + slot] = p == 0 ? m : 0u;
}

sat_status sat_scatter(sat_ctx *ctx, const int32_t *src_row, const int32_t *dst_row, int64_t count, int32_t d, const float *src_base,
                       int32_t ld_src, float *dst, int32_t ld_dst, DbgRange src_rows, DbgRange dst_rows, const RowMaxOut &row_max, int32_t parts)
{
    if (count == 0) return SAT_OK;
    const int32_t d4 = (d + 3) / 4;
    const DbgLimits dbg = dbg_limits(src_rows, DbgRange{0, 0}, dst_rows, ctx->d_flag + 1);
    ProfScope prof(ctx, SATK_SCATTER, (8.0 * d + 8.0) * (double)count, 0.0);
    if (row_max.p) sat_pdl(ctx->stream, k_scatter_rows_max, (unsigned)cdiv64(count * 32, 256), 256, 0)(src_row, dst_row, count, d, src_base, ld_src, dst, ld_dst, row_max, parts, dbg);
    else sat_pdl(ctx->stream, k_scatter_rows, (unsigned)cdiv64(count * d4, 256), 256, 0)(src_row, dst_row, count, d4, src_base, ld_src, dst, ld_dst, dbg);
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

__global__ void k_scatter_add_rows(const int32_t *__restrict__ src_row, const int32_t *__restrict__ dst_row, int64_t count, int32_t d4,
                                   const float *__restrict__ src_base, int64_t ld_src, float *__restrict__ dst, int64_t ld_dst,
                                   const uint32_t *__restrict__ mask, int32_t mask_words, DbgLimits dbg)
{
    sat_grid_wait();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = sat_div(t, d4);
    const int c = (int)(t - i * d4);
    if (i >= count) return;
    float4 x = ld4(src_base + (src_row ? SAT_IDX((int64_t)src_row[i], dbg.src_lo, dbg.src_hi, dbg.status) : i) * ld_src + 4 * c);
    const int64_t r = SAT_IDX((int64_t)dst_row[i], dbg.out_lo, dbg.out_hi, dbg.status);
    if (mask) mask4(x, mask, r * mask_words, c);
    float4 *o = reinterpret_cast<float4 *>(dst + r * ld_dst + 4 * c);
    float4 y = *o;
    y.x += x.x;
    y.y += x.y;
    y.z += x.z;
    y.w += x.w;
    *o = y;
}

sat_status sat_scatter_add(sat_ctx *ctx, const int32_t *src_row, const int32_t *dst_row, int64_t count, int32_t d, const float *src_base,
                           int32_t ld_src, float *dst, int32_t ld_dst, const uint32_t *mask, int32_t mask_words, DbgRange src_rows, DbgRange dst_rows)
{
    if (count == 0) return SAT_OK;
    const int32_t d4 = (d + 3) / 4;
    ProfScope prof(ctx, SATK_SCATTER, (12.0 * d + 8.0) * (double)count, 0.0);
    sat_pdl(ctx->stream, k_scatter_add_rows, (unsigned)cdiv64(count * d4, 256), 256, 0)(src_row, dst_row, count, d4, src_base, ld_src, dst, ld_dst, mask,
                                                                                   mask_words, dbg_limits(src_rows, DbgRange{0, 0}, dst_rows, ctx->d_flag + 1));
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

// -------------------------------------------------------------------------------------
// Halo positions by cache slot: the inverse of halo_slot[].  A boundary node is a halo node of every other partition it has
// a neighbour in; reductions over "all copies of a node" (gradient-side history, transposed predictor convolution) read
// their terms through this index, one writer per slot, in ascending partition order.
// -------------------------------------------------------------------------------------
__global__ void k_hs_count(const int32_t *__restrict__ halo_slot, int64_t nb, int32_t *__restrict__ cnt)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < nb) atomicAdd(cnt + halo_slot[p], 1);   // integer counts: the result does not depend on the order
}

// the halo slots of one partition are distinct, so the cursor of a slot is touched by one thread per launch; the partitions
// are launched in ascending order
__global__ void k_hs_fill(const int32_t *__restrict__ halo_slot, int64_t p0, int64_t count, const int64_t *__restrict__ hs_ptr,
                          int32_t *__restrict__ cursor, int32_t *__restrict__ hs_pos)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const int32_t s = halo_slot[p0 + i];
    const int32_t k = cursor[s];
    cursor[s] = k + 1;
    hs_pos[hs_ptr[s] + k] = (int32_t)(p0 + i);
}

static sat_status build_halo_by_slot(sat_ctx *ctx)
{
    if (ctx->hs_ptr) return SAT_OK;
    const int64_t ns = ctx->n_slots, nb = ctx->nb;
    int32_t *cnt = nullptr;
    SAT_CUDA(ctx, cudaMalloc(&cnt, (size_t)(ns + 1) * sizeof(int32_t)));
    cudaError_t e = cudaMalloc(&ctx->hs_ptr, (size_t)(ns + 1) * sizeof(int64_t));
    if (e == cudaSuccess) e = cudaMalloc(&ctx->hs_pos, (size_t)(nb > 0 ? nb : 1) * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, (size_t)(ns + 1) * sizeof(int32_t), ctx->stream);
    sat_status rc = SAT_OK;
    if (e == cudaSuccess && nb > 0) {
        k_hs_count<<<(unsigned)cdiv64(nb, 256), 256, 0, ctx->stream>>>(ctx->halo_slot, nb, cnt);
        ctx->launches++;
    }
    if (e == cudaSuccess) rc = sat_scan_i32(ctx, cnt, ns, ctx->hs_ptr);
    if (e == cudaSuccess && rc == SAT_OK) e = cudaMemsetAsync(cnt, 0, (size_t)(ns + 1) * sizeof(int32_t), ctx->stream);
    for (int32_t m = 0; e == cudaSuccess && rc == SAT_OK && m < ctx->M; ++m) {
        const int64_t p0 = ctx->h_halo_off[m], count = ctx->h_halo_off[m + 1] - p0;
        if (count == 0) continue;
        k_hs_fill<<<(unsigned)cdiv64(count, 256), 256, 0, ctx->stream>>>(ctx->halo_slot, p0, count, ctx->hs_ptr, cnt, ctx->hs_pos);
        ctx->launches++;
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    cudaFree(cnt);
    if (e != cudaSuccess || rc != SAT_OK) {
        cudaFree(ctx->hs_ptr);
        cudaFree(ctx->hs_pos);
        ctx->hs_ptr = nullptr;
        ctx->hs_pos = nullptr;
        return rc != SAT_OK ? rc : sat_check_cuda(ctx, e, "halo positions by slot");
    }
    return SAT_OK;
}

__global__ void __launch_bounds__(256)
k_sum_by_slot(const int64_t *__restrict__ hs_ptr, const int32_t *__restrict__ hs_pos, int32_t n_slots, const float *__restrict__ dinv_enc,
              int32_t n, int32_t d4, const float *__restrict__ src, int64_t ld_src, int self_scale, int add, float *__restrict__ out, int64_t ld_out,
              DbgLimits dbg)
{
    sat_grid_wait();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t s = sat_div(t, d4);
    const int c = (int)(t - s * d4);
    if (s >= n_slots) return;
    const int64_t b = hs_ptr[s], e = hs_ptr[s + 1];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t i = b; i < e; ++i) {
        const float4 x = ld4(src + SAT_IDX((int64_t)__ldg(hs_pos + i), dbg.src_lo, dbg.src_hi, dbg.status) * ld_src + 4 * c);
        acc.x += x.x;
        acc.y += x.y;
        acc.z += x.z;
        acc.w += x.w;
    }
    if (self_scale && e > b) {
        const float du = __ldg(dinv_enc + n + hs_pos[b]);
        const float p = du * du;
        acc.x *= p;
        acc.y *= p;
        acc.z *= p;
        acc.w *= p;
    }
    float4 *o = reinterpret_cast<float4 *>(out + s * ld_out + 4 * c);
    if (add) {
        const float4 y = *o;
        acc.x += y.x;
        acc.y += y.y;
        acc.z += y.z;
        acc.w += y.w;
    }
    *o = acc;
}

sat_status sat_sum_by_slot(sat_ctx *ctx, int32_t d, const float *src, int32_t ld_src, int self_scale, int add, float *out, int32_t ld_out)
{
    if (ctx->n_slots == 0) return SAT_OK;
    SAT_TRY(build_halo_by_slot(ctx));
    const int32_t d4 = (d + 3) / 4;
    ProfScope prof(ctx, SATK_SCATTER, 8.0 * (double)ctx->nb + 4.0 * d * ((double)ctx->nb + (add ? 2.0 : 1.0) * ctx->n_slots), 0.0);
    sat_pdl(ctx->stream, k_sum_by_slot, (unsigned)cdiv64((int64_t)ctx->n_slots * d4, 256), 256, 0)(ctx->hs_ptr, ctx->hs_pos, ctx->n_slots, ctx->dinv_enc,
                                                                                              ctx->n, d4, src, ld_src, self_scale, add, out, ld_out,
                                                                                              dbg_limits(DbgRange{0, ctx->nb}, DbgRange{0, 0}, DbgRange{0, ctx->n_slots}, ctx->d_flag + 1));
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}


// -------------------------------------------------------------------------------------
// Measurement aid: what the L2 -> SM path of this GPU delivers, measured in the run that quotes it.
//   stream: every thread block reads a contiguous 128-bit-per-lane stream of a buffer that fits in L2;
//   gather: one warp per item reads `row_floats`-wide rows of that buffer in a seeded pseudo-random order with the
//           access shape of the SpMM (lanes own 128-bit column slices, several rows in flight), accumulating them.
// Results are kept live through a predicated store that never fires for finite data.
// -------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_l2_stream(const float4 *__restrict__ buf, int64_t n_vec, int reps, float *__restrict__ sink)
{
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int r = 0; r < reps; ++r) {
        int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        for (; i + 3 * stride < n_vec; i += 4 * stride) {
            const float4 a = __ldg(buf + i), b = __ldg(buf + i + stride), c = __ldg(buf + i + 2 * stride), d = __ldg(buf + i + 3 * stride);
            acc.x += a.x + b.x + c.x + d.x;
            acc.y += a.y + b.y + c.y + d.y;
            acc.z += a.z + b.z + c.z + d.z;
            acc.w += a.w + b.w + c.w + d.w;
        }
        for (; i < n_vec; i += stride) {
            const float4 a = __ldg(buf + i);
            acc.x += a.x; acc.y += a.y; acc.z += a.z; acc.w += a.w;
        }
    }
    if (acc.x + acc.y + acc.z + acc.w == 12345.678f) sink[0] = acc.x;   // never true for the zero-filled buffer
}

template <int NV>
__global__ void __launch_bounds__(256, NV <= 2 ? 8 : 4)
k_l2_gather(const float *__restrict__ buf, uint32_t row_mask, int32_t d4, int64_t n_items, int per_item, float *__restrict__ sink)
{
    const int lane = threadIdx.x & 31;
    const int64_t item = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (item >= n_items) return;
    float4 acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    uint64_t state = 0x9E3779B97F4A7C15ull * (uint64_t)(item + 1);
    for (int e = 0; e < per_item; e += 4) {
        int64_t r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            state = state * 6364136223846793005ull + 1442695040888963407ull;   // the same sequence in every lane of the warp
            r[u] = (int64_t)((uint32_t)(state >> 24) & row_mask);   // the row count is a power of two
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float *src = buf + r[u] * (4 * (int64_t)d4);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int idx = lane + 32 * v;
                if (idx < d4) fma4(acc[v], 0.5f, ld4(src + 4 * idx));
            }
        }
    }
    float t = 0.f;
#pragma unroll
    for (int v = 0; v < NV; ++v) t += acc[v].x + acc[v].y + acc[v].z + acc[v].w;
    if (t == 12345.678f) sink[0] = t;
}

extern "C" sat_status sat_profile_l2_rates(sat_ctx *ctx, int32_t row_floats, double *stream_gbs, double *gather_gbs)
{
    CHECK_CTX(ctx);
    if (row_floats < 4 || row_floats > 1024 || (row_floats & 3)) return sat_fail(ctx, SAT_EINVAL, "sat_profile_l2_rates: row width must be a multiple of 4 in [4, 1024]");
    const size_t bytes = (size_t)64 << 20;                        // well inside the 126 MB L2
    const int32_t d4 = row_floats / 4;
    int64_t n_rows = 1;                                           // the largest power of two of rows that fits the buffer
    while (2 * n_rows * (int64_t)row_floats * 4 <= (int64_t)bytes) n_rows *= 2;
    float *buf = nullptr, *sink = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaMalloc((void **)&buf, bytes);
    if (e == cudaSuccess) e = cudaMalloc((void **)&sink, 256);
    if (e == cudaSuccess) e = cudaMemsetAsync(buf, 0, bytes, ctx->stream);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    float ms_stream = 0.f, ms_gather = 0.f;
    const int reps = 8, per_item = 64;
    const int64_t n_items = (int64_t)1 << 20;                      // 64 rows each: 64 Mi row reads per launch
    if (e == cudaSuccess) {
        const int64_t n_vec = (int64_t)(bytes / 16);
        for (int pass = 0; pass < 2 && e == cudaSuccess; ++pass) {  // first pass warms the L2 and the instruction cache
            cudaEventRecord(e0, ctx->stream);
            k_l2_stream<<<ctx->sms * 8, 256, 0, ctx->stream>>>((const float4 *)buf, n_vec, reps, sink);
            cudaEventRecord(e1, ctx->stream);
            ctx->launches++;
            e = cudaEventSynchronize(e1);
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms_stream, e0, e1);
        }
        for (int pass = 0; pass < 2 && e == cudaSuccess; ++pass) {
            cudaEventRecord(e0, ctx->stream);
            const unsigned grid = (unsigned)cdiv64(n_items * 32, 256);
            if (d4 <= 32) k_l2_gather<1><<<grid, 256, 0, ctx->stream>>>(buf, (uint32_t)(n_rows - 1), d4, n_items, per_item, sink);
            else if (d4 <= 64) k_l2_gather<2><<<grid, 256, 0, ctx->stream>>>(buf, (uint32_t)(n_rows - 1), d4, n_items, per_item, sink);
            else if (d4 <= 128) k_l2_gather<4><<<grid, 256, 0, ctx->stream>>>(buf, (uint32_t)(n_rows - 1), d4, n_items, per_item, sink);
            else k_l2_gather<8><<<grid, 256, 0, ctx->stream>>>(buf, (uint32_t)(n_rows - 1), d4, n_items, per_item, sink);
            cudaEventRecord(e1, ctx->stream);
            ctx->launches++;
            e = cudaEventSynchronize(e1);
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms_gather, e0, e1);
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(buf);
    cudaFree(sink);
    if (e != cudaSuccess) return sat_check_cuda(ctx, e, "sat_profile_l2_rates");
    if (stream_gbs) *stream_gbs = (double)bytes * reps / (ms_stream * 1e-3) / 1e9;
    if (gather_gbs) *gather_gbs = (double)n_items * per_item * row_floats * 4.0 / (ms_gather * 1e-3) / 1e9;
    return SAT_OK;
}
