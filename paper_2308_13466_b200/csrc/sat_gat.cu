// Graph-attention layer as the local layer of a partition (the paper also evaluates SAT with a GAT backbone; the layer
// itself is the standard single-head graph attention layer).  For inner node v, over the entries u of its local CSR row
// (neighbours inside the partition, v itself, neighbours outside = halo rows with cached / predicted embeddings):
//     z_u = h_u W;  e_vu = LeakyReLU_0.2(a_dst . z_v + a_src . z_u);  alpha_vu = softmax_u(e_vu);
//     o_v = sum_u alpha_vu z_u + bias;  h'_v = ReLU(o_v) or o_v.
// Backward with the halo embeddings constant (their z still depends on W):
//     D = g o [o > 0];  dalpha_vu = D_v . z_u;  t_v = sum_u alpha_vu dalpha_vu;
//     dpre_vu = alpha_vu (dalpha_vu - t_v) LeakyReLU'(pre_vu);  ds_dst[v] = sum_u dpre_vu;  ds_src[u] = sum_v dpre_vu;
//     dZ_u = sum_v alpha_vu D_v + ds_src[u] a_src (+ ds_dst[u] a_dst for inner u);
//     G_W = H^T dZ over inner and halo rows;  G_a_src = Z^T ds_src;  G_a_dst = Z_in^T ds_dst;  G_b = 1^T D;  G_in = dZ_in W^T.
// Every sum has a single writer and a fixed order.  How it is cut into passes:
//   forward   k_gat_alpha: softmax of every row, written as {column, alpha} entries; the weighted sums of z rows are then the product
//             kernel of the GCN layer (sat_spmm_entries) with those entries and a bias / ReLU epilogue.
//   backward  k_gat_dots: D_v . z_u of every entry, once (a gather of z rows, doubles out); k_gat_rows: t_v, ds_dst and the entry's
//             dpre; k_gat_cols brings alpha and dpre to the column side through an index of mirrored entries (gat_prepare) and sums
//             ds_src; dZ is again the product kernel, with D rows gathered and the a_src / a_dst terms in its epilogue.
// The first version recomputed alpha and the dot product in each of three gather sweeps and walked every halo row with one warp:
// 169 k nodes, 2.6 M entries, 256 wide: 763 + 626 + 911 us per layer in its sweeps against 389 (dots) + 65 (rows, cols) + 370 (the two
// products) now.
#include "sat_internal.h"

#define GAT_SLOPE 0.2f
#define GAT_MAX_NV 8   /* float4 per lane: widths up to 1024 */


__device__ __forceinline__ float warp_sum(float x)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}
__device__ __forceinline__ float lrelu(float x) { return x > 0.f ? x : GAT_SLOPE * x; }

// s_src[r] = a_src . z_r, s_dst[r] = a_dst . z_r (when asked for).  A warp takes four rows: the vectors' elements are loaded once for them and
// four row loads are in flight (with one row a warp the kernel was bound by its scalar loads, 50 us for 169343 x 256: epoch 6257 -> 6177 us).
#define GAT_SCORE_ROWS 4
__global__ void __launch_bounds__(256)
k_gat_scores(const float *__restrict__ z, int64_t ld, int64_t rows, int32_t d, const float *__restrict__ a_src, const float *__restrict__ a_dst,
             float *__restrict__ s_src, float *__restrict__ s_dst)
{
    sat_grid_wait();
    const int64_t r0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * GAT_SCORE_ROWS;
    const int lane = threadIdx.x & 31;
    if (r0 >= rows) return;
    float ps[GAT_SCORE_ROWS] = {}, pd[GAT_SCORE_ROWS] = {};
    for (int c4 = lane; 4 * c4 < d; c4 += 32) {   // rows are 16-byte aligned and padded with zeros, the vectors end at d
        float4 x[GAT_SCORE_ROWS];
#pragma unroll
        for (int i = 0; i < GAT_SCORE_ROWS; ++i)
            x[i] = r0 + i < rows ? __ldg(reinterpret_cast<const float4 *>(z + (r0 + i) * ld) + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
        float as[4], ad[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = 4 * c4 + k;
            as[k] = c < d ? __ldg(a_src + c) : 0.f;
            ad[k] = a_dst && c < d ? __ldg(a_dst + c) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < GAT_SCORE_ROWS; ++i) {
            ps[i] = fmaf(x[i].w, as[3], fmaf(x[i].z, as[2], fmaf(x[i].y, as[1], fmaf(x[i].x, as[0], ps[i]))));
            if (a_dst) pd[i] = fmaf(x[i].w, ad[3], fmaf(x[i].z, ad[2], fmaf(x[i].y, ad[1], fmaf(x[i].x, ad[0], pd[i]))));
        }
    }
#pragma unroll
    for (int i = 0; i < GAT_SCORE_ROWS; ++i) {
        ps[i] = warp_sum(ps[i]);
        if (a_dst) pd[i] = warp_sum(pd[i]);
        if (lane == 0 && r0 + i < rows) {
            s_src[r0 + i] = ps[i];
            if (a_dst) s_dst[r0 + i] = pd[i];
        }
    }
}

// A row is worked on by a team of T threads: 16 lanes of a warp for the ordinary rows, a thread block for rows of more than GAT_LONG
// entries (a hub's ten thousand entries were the whole launch for one warp).
#define GAT_TEAM 16
#define GAT_LONG SAT_HROW_LONG

template <int T, typename V, typename F>
__device__ __forceinline__ V team_reduce(V x, F op, V *sh)
{
    if (T < 256) {
        const unsigned mask = ((1u << (T & 31)) - 1u) << (threadIdx.x & 31 & ~(T - 1));
#pragma unroll
        for (int o = T / 2; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(mask, x, o));
        return x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    x = sh[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) x = op(x, sh[w]);
    return x;
}
struct OpAdd {
    template <typename V> __device__ V operator()(V a, V b) const { return a + b; }
};
struct OpMax {
    __device__ float operator()(float a, float b) const { return fmaxf(a, b); }
};

// softmax of one row: ent[e] = {column, alpha}
template <int T>
__device__ __forceinline__ void gat_alpha_row(int tid, int64_t e0, int64_t e1, float sd, const int32_t *__restrict__ lenc, int32_t n,
                                              const float *__restrict__ s_in, const float *__restrict__ s_halo, int2 *__restrict__ ent, float *sh)
{
    auto logit = [&](int32_t c) { return lrelu(sd + (c < n ? s_in[c] : s_halo[c - n])); };
    // the first entry of every thread stays in registers (most rows have no more); the others are fetched again per pass
    const int64_t ef = e0 + tid;
    const int32_t c_first = ef < e1 ? lenc[ef] : 0;
    const float l_first = ef < e1 ? logit(c_first) : -INFINITY;
    float mx = l_first;
#pragma unroll 4
    for (int64_t e = ef + T; e < e1; e += T) mx = fmaxf(mx, logit(lenc[e]));
    mx = team_reduce<T>(mx, OpMax(), sh);
    const float x_first = ef < e1 ? expf(l_first - mx) : 0.f;
    float den = x_first;
#pragma unroll 4
    for (int64_t e = ef + T; e < e1; e += T) den += expf(logit(lenc[e]) - mx);
    den = team_reduce<T>(den, OpAdd(), sh);
    if (ef < e1) ent[ef] = make_int2(c_first, __float_as_int(x_first / den));
#pragma unroll 4
    for (int64_t e = ef + T; e < e1; e += T) {
        const int32_t c = lenc[e];
        ent[e] = make_int2(c, __float_as_int(expf(logit(c) - mx) / den));
    }
}

__global__ void __launch_bounds__(256)
k_gat_alpha(const int64_t *__restrict__ lrowptr, const int32_t *__restrict__ lenc, int32_t n, int32_t row0, int32_t n_rows,
            const int32_t *__restrict__ long_rows, int32_t n_long, const float *__restrict__ s_in, const float *__restrict__ s_halo,
            const float *__restrict__ s_dst, int2 *__restrict__ ent)
{
    sat_grid_wait();
    __shared__ float sh[8];
    if ((int32_t)blockIdx.x < n_long) {
        const int32_t row = long_rows[blockIdx.x];
        gat_alpha_row<256>(threadIdx.x, lrowptr[row], lrowptr[row + 1], s_dst[row], lenc, n, s_in, s_halo, ent, sh);
        return;
    }
    const int64_t w = ((int64_t)(blockIdx.x - n_long) * 256 + threadIdx.x) / GAT_TEAM;
    if (w >= n_rows) return;
    const int32_t row = row0 + (int32_t)w;
    const int64_t e0 = lrowptr[row], e1 = lrowptr[row + 1];
    if (e1 - e0 > GAT_LONG) return;
    gat_alpha_row<GAT_TEAM>(threadIdx.x & (GAT_TEAM - 1), e0, e1, s_dst[row], lenc, n, s_in, s_halo, ent, sh);
}

// dots[e] = D_v . z_u for every entry (v, u): a group of G lanes per work item, D_v in registers, four z rows in flight.  The products
// are summed in double ((dalpha - t_v) cancels most of their size); the sums of four entries are reduced together, six
// shuffles for the four.
//
// The conversion instruction runs at 16 lanes per clock and SM, 256 of them per entry at d = 256 (392 us at 2.6 M entries).  gat_scaled
// builds a double from the bits instead: sign, exponent and fraction of x in their places of the double without moving the exponent's
// bias are exactly 2^-896 x, zeros and subnormals included.  D is scaled by 2^800 (no overflow for any float) and the sum by 2^96,
// both exact.  Non-finite z give a finite product here: k_gat_rows takes care of those (gat_not_finite).
__device__ __forceinline__ double gat_scaled(float x)
{
    const int b = __float_as_int(x);
    return __hiloint2double((b >> 3) & (int)0x8FFFFFFFu, b << 29);
}
template <int G, int NV>
__global__ void __launch_bounds__(256, NV <= 2 ? 4 : NV <= 4 ? 2 : 1)
k_gat_dots(const int4 *__restrict__ items, int32_t n_items, const int32_t *__restrict__ lenc, int32_t n, int32_t d4, const float *__restrict__ z_in,
           const float *__restrict__ z_halo, uint32_t ldz4, const float *__restrict__ D, double *__restrict__ dots)
{
    sat_grid_wait();
    const int lane = threadIdx.x & (G - 1);
    const int64_t gid = ((int64_t)blockIdx.x * 256 + threadIdx.x) / G;
    if (gid >= n_items) return;
    const unsigned mask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (threadIdx.x & 31 & ~(G - 1));
    const int4 it = __ldg(items + gid);
    const int64_t e0 = (int64_t)(uint32_t)it.z | ((int64_t)(it.w & 0xffff) << 32);
    const int32_t len = it.w >> 16;
    const float4 *zi = reinterpret_cast<const float4 *>(z_in) + lane, *zh = reinterpret_cast<const float4 *>(z_halo) + lane - (int64_t)n * ldz4;
    double dv[NV][4];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const float4 x = lane + v * G < d4 ? __ldg(reinterpret_cast<const float4 *>(D) + (int64_t)it.x * ldz4 + lane + v * G) : make_float4(0.f, 0.f, 0.f, 0.f);
        dv[v][0] = 0x1p800 * (double)x.x;
        dv[v][1] = 0x1p800 * (double)x.y;
        dv[v][2] = 0x1p800 * (double)x.z;
        dv[v][3] = 0x1p800 * (double)x.w;
    }
    const int32_t *__restrict__ cols = lenc + e0;
    for (int32_t e = 0; e < len; e += 4) {
        float4 x[4][NV];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int32_t c = __ldg(cols + (e + u < len ? e + u : len - 1));
            const float4 *src = (c < n ? zi : zh) + (uint64_t)(uint32_t)c * ldz4;
#pragma unroll
            for (int v = 0; v < NV; ++v) x[u][v] = lane + v * G < d4 ? __ldg(src + v * G) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        double p[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            p[u] = 0.0;
#pragma unroll
            for (int v = 0; v < NV; ++v)
                p[u] += dv[v][0] * gat_scaled(x[u][v].x) + dv[v][1] * gat_scaled(x[u][v].y) + dv[v][2] * gat_scaled(x[u][v].z) + dv[v][3] * gat_scaled(x[u][v].w);
        }
        // lanes with bit 1 keep entries 2 and 3, the others 0 and 1; then bit 0 picks one; then the lanes that hold the same entry add up
        const bool b1 = lane & 2, b0 = lane & 1;
        double q0 = (b1 ? p[2] : p[0]) + __shfl_xor_sync(mask, b1 ? p[0] : p[2], 2);
        double q1 = (b1 ? p[3] : p[1]) + __shfl_xor_sync(mask, b1 ? p[1] : p[3], 2);
        double r = (b0 ? q1 : q0) + __shfl_xor_sync(mask, b0 ? q0 : q1, 1);
#pragma unroll
        for (int o = G / 2; o > 2; o >>= 1) r += __shfl_xor_sync(mask, r, o);
        if (lane < 4 && e + lane < len) dots[e0 + e + lane] = 0x1p96 * r;
    }
}

// The dot product of a z row that holds an infinity or a NaN is not a number, whatever D is.  Its score is not finite then, so finite scores
// settle it; the others are rare and have their row looked at (a score may overflow over a finite row).  This matters where the score is
// minus infinity, and alpha zero: anything else makes alpha a NaN by itself.
__device__ __forceinline__ bool gat_not_finite(float score, const float *__restrict__ z, int32_t d)
{
    if (isfinite(score)) return false;
    for (int32_t k = 0; k < d; ++k)
        if (!isfinite(z[k])) return true;
    return false;
}

// per row v: t_v = sum alpha dot / sum alpha and ds_dst[v]; per entry, over the dot product: dpre = alpha slope (dot - t_v)
// (the sums in double and divided by sum alpha: the fp32 weights sum to 1 + eps, and ds_dst, exactly zero where all slopes agree,
// would inherit -eps t_v; dpre stays in double until its column is summed, the dpre of a column cancel as well)
template <int T>
__device__ __forceinline__ void gat_row(int tid, int64_t e0, int64_t e1, float sd, const int2 *__restrict__ ent, int32_t n,
                                        const float *__restrict__ s_in, const float *__restrict__ s_halo, const float *__restrict__ z_in,
                                        const float *__restrict__ z_halo, int64_t ld_z, int32_t d, double *__restrict__ dots,
                                        float *__restrict__ ds_dst, double *sh)
{
    auto score = [&](int32_t c) { return c < n ? s_in[c] : s_halo[c - n]; };
    auto slope = [&](float s) { return sd + s > 0.f ? 1.f : GAT_SLOPE; };
    const int64_t ef = e0 + tid;
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0, p_first = 0.0;
    float as_first = 0.f;
#pragma unroll 4
    for (int64_t e = ef; e < e1; e += T) {
        const int2 q = ent[e];
        const float al = __int_as_float(q.y), s = score(q.x), sl = slope(s);
        const double as = (double)al * (double)sl;
        double p = dots[e];
        if (gat_not_finite(s, q.x < n ? z_in + q.x * ld_z : z_halo + (q.x - n) * ld_z, d)) p = __longlong_as_double(0x7ff8000000000000ll);
        a0 += (double)al;
        a1 += (double)al * p;
        a2 += as * p;
        a3 += as;
        if (e == ef) {
            p_first = p;
            as_first = al * sl;
        }
    }
    a0 = team_reduce<T>(a0, OpAdd(), sh);
    a1 = team_reduce<T>(a1, OpAdd(), sh);
    a2 = team_reduce<T>(a2, OpAdd(), sh);
    a3 = team_reduce<T>(a3, OpAdd(), sh);
    const double t = a1 / a0;
    if (tid == 0) *ds_dst = (float)(a2 / a0 - t * (a3 / a0));
    if (ef < e1) dots[ef] = (double)as_first * (p_first - t);
#pragma unroll 4
    for (int64_t e = ef + T; e < e1; e += T) {
        const int2 q = ent[e];
        dots[e] = (double)(__int_as_float(q.y) * slope(score(q.x))) * (dots[e] - t);   // (t is a NaN where a product is)
    }
}

__global__ void __launch_bounds__(256)
k_gat_rows(const int64_t *__restrict__ lrowptr, const int2 *__restrict__ ent, int32_t n, int32_t row0, int32_t n_rows, const int32_t *__restrict__ long_rows,
           int32_t n_long, const float *__restrict__ s_in, const float *__restrict__ s_halo, const float *__restrict__ s_dst,
           const float *__restrict__ z_in, const float *__restrict__ z_halo, int64_t ld_z, int32_t d, double *dots, float *__restrict__ ds_dst)
{
    sat_grid_wait();
    __shared__ double sh[8];
    if ((int32_t)blockIdx.x < n_long) {
        const int32_t row = long_rows[blockIdx.x];
        gat_row<256>(threadIdx.x, lrowptr[row], lrowptr[row + 1], s_dst[row], ent, n, s_in, s_halo, z_in, z_halo, ld_z, d, dots, ds_dst + row, sh);
        return;
    }
    const int64_t w = ((int64_t)(blockIdx.x - n_long) * 256 + threadIdx.x) / GAT_TEAM;
    if (w >= n_rows) return;
    const int32_t row = row0 + (int32_t)w;
    const int64_t e0 = lrowptr[row], e1 = lrowptr[row + 1];
    if (e1 - e0 > GAT_LONG) return;
    gat_row<GAT_TEAM>(threadIdx.x & (GAT_TEAM - 1), e0, e1, s_dst[row], ent, n, s_in, s_halo, z_in, z_halo, ld_z, d, dots, ds_dst + row, sh);
}

// column side of node u: its entries are the mirror images map[e] of row entries (v, u); ent_out[e] = {v, alpha_vu}, ds_src[u] = sum dpre_vu
template <int T>
__device__ __forceinline__ void gat_col(int tid, int64_t e0, int64_t e1, const int32_t *__restrict__ idx, const uint32_t *__restrict__ map,
                                        const int2 *__restrict__ ent, const double *__restrict__ dpre, int2 *__restrict__ ent_out,
                                        float *__restrict__ ds_src, double *sh)
{
    double s = 0.0;
#pragma unroll 4
    for (int64_t e = e0 + tid; e < e1; e += T) {
        const uint32_t m = map[e];
        ent_out[e] = make_int2(idx[e], ent[m].y);
        s += dpre[m];
    }
    s = team_reduce<T>(s, OpAdd(), sh);
    if (tid == 0) *ds_src = (float)s;
}

__global__ void __launch_bounds__(256)
k_gat_cols(const int64_t *__restrict__ ptr, const int32_t *__restrict__ cnt, int64_t u0, int64_t n_u, const int32_t *__restrict__ long_u, int32_t n_long,
           const int32_t *__restrict__ idx, const uint32_t *__restrict__ map, const int2 *__restrict__ ent, const double *__restrict__ dpre,
           int2 *__restrict__ ent_out, float *__restrict__ ds_src)
{
    sat_grid_wait();
    __shared__ double sh[8];
    if ((int32_t)blockIdx.x < n_long) {
        const int32_t u = long_u[blockIdx.x];
        gat_col<256>(threadIdx.x, ptr[u], cnt ? ptr[u] + cnt[u] : ptr[u + 1], idx, map, ent, dpre, ent_out, ds_src + u, sh);
        return;
    }
    const int64_t w = ((int64_t)(blockIdx.x - n_long) * 256 + threadIdx.x) / GAT_TEAM;
    if (w >= n_u) return;
    const int64_t u = u0 + w, e0 = ptr[u];
    if (ptr[u + 1] - e0 > GAT_LONG) return;
    gat_col<GAT_TEAM>(threadIdx.x & (GAT_TEAM - 1), e0, cnt ? e0 + cnt[u] : ptr[u + 1], idx, map, ent, dpre, ent_out, ds_src + u, sh);
}

// mirror images: entry e = (r, c) of the inner block is entry rev[e] = (c, r); entry i of halo row j (node u, inner neighbour v) is the
// entry (v, u) of v's local row.  Columns are ascending inside both parts of a row.
__device__ __forceinline__ uint32_t gat_find(const int32_t *__restrict__ lenc, int64_t lo, int64_t hi, int32_t key)
{
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (lenc[mid] < key) lo = mid + 1;
        else hi = mid;
    }
    return (uint32_t)lo;
}
__global__ void k_gat_rev(const int64_t *__restrict__ lrowptr, const int32_t *__restrict__ lenc, const int32_t *__restrict__ inner_cnt, int32_t n,
                          uint32_t *__restrict__ rev, int32_t *__restrict__ is_long)
{
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= n) return;
    const int64_t e0 = lrowptr[r], e1 = e0 + inner_cnt[r];
    for (int64_t e = e0 + lane; e < e1; e += 32) {
        const int32_t c = lenc[e];
        rev[e] = gat_find(lenc, lrowptr[c], lrowptr[c] + inner_cnt[c], (int32_t)r);
    }
    if (lane == 0) is_long[r] = lrowptr[r + 1] - e0 > GAT_LONG ? 1 : 0;
}
__global__ void k_gat_hmap(const int64_t *__restrict__ hrow_ptr, const int32_t *__restrict__ hrow_pos, const int64_t *__restrict__ lrowptr,
                           const int32_t *__restrict__ lenc, const int32_t *__restrict__ inner_cnt, int32_t n, int64_t nb, uint32_t *__restrict__ hmap)
{
    const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (j >= nb) return;
    for (int64_t i = hrow_ptr[j] + lane; i < hrow_ptr[j + 1]; i += 32) {
        const int32_t v = hrow_pos[i];
        hmap[i] = gat_find(lenc, lrowptr[v] + inner_cnt[v], lrowptr[v + 1], (int32_t)(n + j));
    }
}
__global__ void k_gat_long(const int32_t *__restrict__ is_long, const int64_t *__restrict__ off, int32_t n, int32_t *__restrict__ out)
{
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n && is_long[r]) out[off[r]] = (int32_t)r;
}

// part1[b][c] = sum over the rows r of block b of w1[r] x[r][c], and part2 with w2 where given: one pass over x for both.  tpr threads
// (a power of two) walk a row with 128-bit accesses, four rows in flight per thread; the row groups of a block are added in order.
#define GAT_WSUM_ROWS 256
__global__ void __launch_bounds__(256)
k_gat_wcolsum(const float *__restrict__ x, int64_t ld, int64_t rows, int32_t d, int32_t tpr, const float *__restrict__ w1, const float *__restrict__ w2,
              float *__restrict__ part1, float *__restrict__ part2)
{
    sat_grid_wait();
    __shared__ float4 red[2][256];
    const int c4 = threadIdx.x % tpr, rg = threadIdx.x / tpr, n_rg = 256 / tpr, d4 = (d + 3) >> 2;
    const int64_t r0 = (int64_t)blockIdx.x * GAT_WSUM_ROWS, r1 = r0 + GAT_WSUM_ROWS < rows ? r0 + GAT_WSUM_ROWS : rows;
    float4 s1 = make_float4(0.f, 0.f, 0.f, 0.f), s2 = s1;
    if (c4 < d4) {
        for (int64_t r = r0 + rg; r < r1; r += 4 * n_rg) {
            float4 v[4];
            float a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t rr = r + (int64_t)u * n_rg;
                const bool ok = rr < r1;
                v[u] = ok ? __ldg(reinterpret_cast<const float4 *>(x + rr * ld) + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
                a[u] = ok ? __ldg(w1 + rr) : 0.f;
                b[u] = ok && w2 ? __ldg(w2 + rr) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                s1.x = fmaf(a[u], v[u].x, s1.x); s1.y = fmaf(a[u], v[u].y, s1.y); s1.z = fmaf(a[u], v[u].z, s1.z); s1.w = fmaf(a[u], v[u].w, s1.w);
                s2.x = fmaf(b[u], v[u].x, s2.x); s2.y = fmaf(b[u], v[u].y, s2.y); s2.z = fmaf(b[u], v[u].z, s2.z); s2.w = fmaf(b[u], v[u].w, s2.w);
            }
        }
    }
    red[0][threadIdx.x] = s1;
    red[1][threadIdx.x] = s2;
    __syncthreads();
    if (rg < 2 && rg < n_rg && c4 < d4) {
        for (int k = rg; k < (w2 ? 2 : 1); k += n_rg < 2 ? 1 : 2) {
            float4 t = red[k][c4];
            for (int g = 1; g < n_rg; ++g) {
                const float4 y = red[k][g * tpr + c4];
                t.x += y.x; t.y += y.y; t.z += y.z; t.w += y.w;
            }
            float *o = (k ? part2 : part1) + (int64_t)blockIdx.x * d + 4 * c4;
            o[0] = t.x;
            if (4 * c4 + 1 < d) o[1] = t.y;
            if (4 * c4 + 2 < d) o[2] = t.z;
            if (4 * c4 + 3 < d) o[3] = t.w;
        }
    }
}

// -------------------------------------------------------------------------------------
// host side
// -------------------------------------------------------------------------------------
static sat_status gat_nn(sat_ctx *ctx, int64_t m, int32_t n, int32_t k, const float *A, int32_t lda, const float *W, float *C, int32_t ldc)
{
    if (m == 0) return SAT_OK;
    if (sat_use_tc(n, k)) {
        TcWeights Wp;
        SAT_TRY(sat_tc_weights(ctx, W, n, k, nullptr, 0, 0, n, 1, ctx->buf_wsplit, &Wp));
        TcEpilogueHost eh;
        eh.C = C;
        eh.ldc = ldc;
        return sat_gemm_tc(ctx, m, n, A, lda, k, nullptr, 0, 0, Wp, eh, SATK_GEMM_NN);
    }
    GemmEpilogue ep;
    return sat_gemm_nn(ctx, m, n, k, A, lda, W, n, C, ldc, ep);
}

static sat_status gat_nt(sat_ctx *ctx, int64_t m, int32_t n, int32_t k, const float *A, int32_t lda, const float *W, float *C, int32_t ldc)
{
    if (m == 0) return SAT_OK;
    if (sat_use_tc(n, k)) {
        TcWeights Wp;
        SAT_TRY(sat_tc_weights(ctx, W, k, k, nullptr, 0, 0, n, 0, ctx->buf_wsplit, &Wp));
        TcEpilogueHost eh;
        eh.C = C;
        eh.ldc = ldc;
        return sat_gemm_tc(ctx, m, n, A, lda, k, nullptr, 0, 0, Wp, eh, SATK_GEMM_NT);
    }
    return sat_gemm_nt(ctx, m, n, k, A, lda, nullptr, 0, W, k, C, ldc);
}

static sat_status gat_tn(sat_ctx *ctx, int64_t rows, int32_t m, int32_t n, const float *A, int32_t lda, const float *B, int32_t ldb, float *C,
                         int accumulate)
{
    if (rows == 0) {
        if (!accumulate) SAT_CUDA(ctx, cudaMemsetAsync(C, 0, (size_t)m * n * sizeof(float), ctx->stream));
        return SAT_OK;
    }
    if (sat_use_tc(n, m) && rows >= 256) {
        if (n <= 64) return sat_gemm_tn_narrow(ctx, rows, m, n, A, lda, B, ldb, C, n, accumulate);
        return sat_gemm_tc_tn(ctx, rows, m, n, A, lda, B, ldb, C, n, accumulate);
    }
    return sat_gemm_tn(ctx, rows, m, n, A, lda, B, ldb, nullptr, 0, C, n, nullptr, accumulate);
}

// out1[c] (+)= sum_r w1[r] x[r][c], and the same with w2 / out2 where given
static sat_status gat_wcolsum(sat_ctx *ctx, const float *x, int32_t ld, int64_t rows, int32_t d, const float *w1, float *out1, const float *w2,
                              float *out2, int accumulate)
{
    if (rows == 0) {
        if (!accumulate) {
            SAT_CUDA(ctx, cudaMemsetAsync(out1, 0, (size_t)d * sizeof(float), ctx->stream));
            if (out2) SAT_CUDA(ctx, cudaMemsetAsync(out2, 0, (size_t)d * sizeof(float), ctx->stream));
        }
        return SAT_OK;
    }
    const int64_t blocks = cdiv64(rows, GAT_WSUM_ROWS);
    SAT_TRY(sat_ensure(ctx, ctx->buf_colsum, (size_t)2 * blocks * d * sizeof(float)));
    float *p1 = (float *)ctx->buf_colsum.p, *p2 = w2 ? p1 + (size_t)blocks * d : nullptr;
    int tpr = 1;
    while (tpr < (d + 3) / 4) tpr <<= 1;   // d <= 1024: at most 256
    sat_pdl(ctx->stream, k_gat_wcolsum, (unsigned)blocks, 256, 0)(x, ld, rows, d, tpr, w1, w2, p1, p2);
    SAT_LAUNCHED(ctx);
    return sat_splitk_reduce(ctx, p1, d, (int32_t)blocks, accumulate, out1, d, d, p2, d, out2);
}

// what the attention layer needs to know about the partitioning: the mirror image of every inner entry and of every halo-row entry, and
// the rows that get a thread block (built on first use, freed with the partition)
static sat_status gat_prepare(sat_ctx *ctx)
{
    if (ctx->gat_rev) return SAT_OK;
    const int32_t n = ctx->n, M = ctx->M;
    const int64_t lnnz = ctx->nnz + n, nb = ctx->nb;
    if (lnnz >= ((int64_t)1 << 32)) return sat_fail(ctx, SAT_EINVAL, "sat_gat_fwd: more than 2^32 entries");
    uint32_t *rev = nullptr, *hmap = nullptr;
    int32_t *flag = nullptr, *rows = nullptr;
    int64_t *off = nullptr;
    std::vector<int64_t> h((size_t)M + 1, 0);
    sat_status rc = SAT_OK;
    cudaError_t e = cudaMalloc((void **)&rev, (size_t)lnnz * sizeof(uint32_t));
    if (e == cudaSuccess) e = cudaMalloc((void **)&hmap, (size_t)(ctx->nnz_cut > 0 ? ctx->nnz_cut : 1) * sizeof(uint32_t));
    if (e == cudaSuccess) e = cudaMalloc((void **)&flag, (size_t)n * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMalloc((void **)&off, ((size_t)n + 1) * sizeof(int64_t));
    if (e == cudaSuccess) {
        k_gat_rev<<<(unsigned)cdiv64((int64_t)n * 32, 256), 256, 0, ctx->stream>>>(ctx->lrowptr, ctx->lenc, ctx->inner_cnt, n, rev, flag);
        if (nb > 0)
            k_gat_hmap<<<(unsigned)cdiv64(nb * 32, 256), 256, 0, ctx->stream>>>(ctx->hrow_ptr, ctx->hrow_pos, ctx->lrowptr, ctx->lenc, ctx->inner_cnt, n, nb, hmap);
        ctx->launches += nb > 0 ? 2 : 1;
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) rc = sat_scan_i32(ctx, flag, n, off);
    for (int m = 0; e == cudaSuccess && rc == SAT_OK && m <= M; ++m)
        e = cudaMemcpyAsync(&h[m], off + ctx->h_inner_off[m], sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess && rc == SAT_OK) e = cudaStreamSynchronize(ctx->stream);
    if (e == cudaSuccess && rc == SAT_OK) e = cudaMalloc((void **)&rows, (size_t)(h[M] > 0 ? h[M] : 1) * sizeof(int32_t));
    if (e == cudaSuccess && rc == SAT_OK) {
        k_gat_long<<<(unsigned)cdiv64(n, 256), 256, 0, ctx->stream>>>(flag, off, n, rows);
        ctx->launches++;
        e = cudaStreamSynchronize(ctx->stream);
    }
    cudaFree(flag);
    cudaFree(off);
    if (e != cudaSuccess || rc != SAT_OK) {
        cudaFree(rev);
        cudaFree(hmap);
        cudaFree(rows);
        return rc != SAT_OK ? rc : sat_check_cuda(ctx, e, "mirrored entries of the attention layer");
    }
    ctx->gat_rev = rev;
    ctx->gat_hmap = hmap;
    ctx->gat_long = rows;
    ctx->h_gat_long_off = h;
    return SAT_OK;
}

extern "C" sat_status sat_gat_fwd(sat_ctx *ctx, int32_t part, int32_t layer, int32_t d_in, int32_t d_out, const float *h_in, int32_t ld_in,
                                  const float *h_halo, int32_t ld_halo, const float *W, const float *a_src, const float *a_dst,
                                  const float *bias, int act, float *h_out, int32_t ld_out)
{
    CHECK_CTX(ctx);
    const bool push = act & SAT_FWD_PUSH;
    act &= ~SAT_FWD_PUSH;
    PartView v;
    SAT_TRY(sat_part_view(ctx, part, &v));
    if (layer < 1 || layer > SAT_MAX_LAYERS) return sat_fail(ctx, SAT_EINVAL, "sat_gat_fwd: layer must be in [1, %d]", SAT_MAX_LAYERS);
    if (d_in <= 0 || d_out <= 0 || d_out > 128 * GAT_MAX_NV || !W || !a_src || !a_dst) return sat_fail(ctx, SAT_EINVAL, "sat_gat_fwd: bad widths or null parameters");
    if (act != SAT_ACT_NONE && act != SAT_ACT_RELU) return sat_fail(ctx, SAT_EINVAL, "sat_gat_fwd: unknown activation");
    CacheLayer *pc = nullptr;
    if (push) {
        if (!ctx->cache_ok || layer > ctx->n_cached) return sat_fail(ctx, SAT_ESTATE, "sat_gat_fwd: SAT_FWD_PUSH without a cached layer %d", layer);
        pc = &ctx->cache[layer - 1];
        if (pc->width != d_out) return sat_fail(ctx, SAT_EINVAL, "sat_gat_fwd: SAT_FWD_PUSH of %d columns into a cached layer of %d", d_out, pc->width);
    }
    if (v.n_rows > 0 && (!h_in || !h_out || !ok_ld(ld_in, d_in) || !ok_ld(ld_out, d_out) || !aligned16(h_in) || !aligned16(h_out)))
        return sat_fail(ctx, SAT_EINVAL, "sat_gat_fwd: null / misaligned h_in / h_out or bad leading dimension");
    if (v.n_halo > 0 && (!h_halo || !ok_ld(ld_halo, d_in) || !aligned16(h_halo))) return sat_fail(ctx, SAT_EINVAL, "sat_gat_fwd: null / misaligned h_halo");
    GatState &G = ctx->gat[layer];
    const int32_t ld_z = round_up4(d_out);
    const int64_t n = ctx->n, nb = ctx->nb;
    if (G.d_out != d_out || G.valid.size() != (size_t)ctx->M) {
        // buffers over all rows / halo positions of the graph (any partition may be called); zeroed once so that the padding
        // columns of the z rows, which no kernel writes, read as zero
        SAT_TRY(sat_ensure(ctx, G.z_in, (size_t)(n > 0 ? n : 1) * ld_z * sizeof(float)));
        SAT_TRY(sat_ensure(ctx, G.z_halo, (size_t)(nb > 0 ? nb : 1) * ld_z * sizeof(float)));
        SAT_TRY(sat_ensure(ctx, G.scal, (size_t)(2 * (n > 0 ? n : 1) + (nb > 0 ? nb : 1)) * sizeof(float)));
        SAT_TRY(sat_ensure(ctx, G.ent, (size_t)(ctx->nnz + n) * sizeof(int2)));
        SAT_CUDA(ctx, cudaMemsetAsync(G.z_in.p, 0, G.z_in.bytes, ctx->stream));
        SAT_CUDA(ctx, cudaMemsetAsync(G.z_halo.p, 0, G.z_halo.bytes, ctx->stream));
        G.d_out = d_out;
        G.valid.assign(ctx->M, 0);
    }
    G.relu = act == SAT_ACT_RELU;
    float *z_in = (float *)G.z_in.p, *z_halo = (float *)G.z_halo.p;
    float *s_in = (float *)G.scal.p, *s_dst = s_in + n, *s_halo = s_dst + n;
    SAT_TRY(gat_prepare(ctx));
    SAT_TRY(gat_nn(ctx, v.n_rows, d_out, d_in, h_in, ld_in, W, z_in + (int64_t)v.row0 * ld_z, ld_z));
    SAT_TRY(gat_nn(ctx, v.n_halo, d_out, d_in, h_halo, ld_halo, W, z_halo + v.halo0 * ld_z, ld_z));
    ProfScope prof(ctx, SATK_GAT, 0.0, 0.0);
    if (v.n_rows > 0) {
        sat_pdl(ctx->stream, k_gat_scores, (unsigned)cdiv64(v.n_rows, 8 * GAT_SCORE_ROWS), 256, 0)(z_in + (int64_t)v.row0 * ld_z, ld_z, v.n_rows, d_out, a_src, a_dst,
                                                                                           s_in + v.row0, s_dst + v.row0);
        SAT_LAUNCHED(ctx);
    }
    if (v.n_halo > 0) {
        sat_pdl(ctx->stream, k_gat_scores, (unsigned)cdiv64(v.n_halo, 8 * GAT_SCORE_ROWS), 256, 0)(z_halo + v.halo0 * ld_z, ld_z, v.n_halo, d_out, a_src, nullptr,
                                                                                  s_halo + v.halo0, nullptr);
        SAT_LAUNCHED(ctx);
    }
    if (v.n_rows > 0) {
        const int64_t l0 = ctx->h_gat_long_off[v.p0], n_long = ctx->h_gat_long_off[v.p1] - l0;
        sat_pdl(ctx->stream, k_gat_alpha, (unsigned)(n_long + cdiv64((int64_t)v.n_rows * GAT_TEAM, 256)), 256, 0)(
            ctx->lrowptr, ctx->lenc, ctx->n, v.row0, v.n_rows, ctx->gat_long + l0, (int32_t)n_long, s_in, s_halo, s_dst, (int2 *)G.ent.p);
        SAT_LAUNCHED(ctx);
        SpmmEpilogue ep;
        ep.bias = bias;
        ep.relu = G.relu;
        if (push && ctx->n_slots > 0) {   // boundary rows go to the ring from the product's epilogue (a pass of its own: 66 us of 169343 x 256)
            SAT_TRY(sat_row_slots(ctx, &ep.push_slot));
            ep.push = ring_buf(ctx, pc, ctx->write_idx);
            ep.ld_push = pc->ld;
            if (!pc->proj_tag.empty()) pc->proj_tag[ctx->write_idx] = 0;   // the buffer changes: its cached input projection is stale
            ep.row_max = sat_ring_max(ctx, pc, ctx->write_idx);
        }
        SAT_TRY(sat_spmm_entries(ctx, v, 0, d_out, (const int2 *)G.ent.p, z_in, ld_z, z_halo, ld_z, h_out - (int64_t)v.row0 * ld_out, ld_out, ep));
        if (ep.row_max.p && part == SAT_ALL_PARTS) pc->row_max_ok[ctx->write_idx] = 1;
    }
    for (int m = (part == SAT_ALL_PARTS ? 0 : part); m < (part == SAT_ALL_PARTS ? ctx->M : part + 1); ++m) G.valid[m] = 1;
    return SAT_OK;
}

// the attention scores kept by the forward call, for checkpoints and tests
extern "C" sat_status sat_gat_scores(sat_ctx *ctx, int32_t layer, float *s_src_inner_host, float *s_dst_host, float *s_src_halo_host)
{
    CHECK_CTX(ctx);
    if (layer < 1 || layer > SAT_MAX_LAYERS) return sat_fail(ctx, SAT_EINVAL, "sat_gat_scores: layer must be in [1, %d]", SAT_MAX_LAYERS);
    GatState &G = ctx->gat[layer];
    if (G.d_out <= 0 || G.valid.size() != (size_t)ctx->M) return sat_fail(ctx, SAT_ESTATE, "sat_gat_scores: sat_gat_fwd has not run for layer %d", layer);
    for (int m = 0; m < ctx->M; ++m)
        if (!G.valid[m]) return sat_fail(ctx, SAT_ESTATE, "sat_gat_scores: sat_gat_fwd has not run for partition %d of layer %d", m, layer);
    const int64_t n = ctx->n, nb = ctx->nb;
    const float *s_in = (const float *)G.scal.p, *s_dst = s_in + n, *s_halo = s_dst + n;
    if (s_src_inner_host) SAT_CUDA(ctx, cudaMemcpyAsync(s_src_inner_host, s_in, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, ctx->stream));
    if (s_dst_host) SAT_CUDA(ctx, cudaMemcpyAsync(s_dst_host, s_dst, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, ctx->stream));
    if (s_src_halo_host && nb > 0) SAT_CUDA(ctx, cudaMemcpyAsync(s_src_halo_host, s_halo, (size_t)nb * sizeof(float), cudaMemcpyDeviceToHost, ctx->stream));
    SAT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return SAT_OK;
}

extern "C" sat_status sat_gat_bwd(sat_ctx *ctx, int32_t part, int32_t layer, const float *g_out, int32_t ld_g, const float *h_out, int32_t ld_out,
                                  const float *h_in, int32_t ld_in, const float *h_halo, int32_t ld_halo, int32_t d_in, const float *W,
                                  const float *a_src, const float *a_dst, float *g_W, float *g_a_src, float *g_a_dst, float *g_b,
                                  int accumulate, float *g_in, int32_t ld_gin)
{
    CHECK_CTX(ctx);
    PartView v;
    SAT_TRY(sat_part_view(ctx, part, &v));
    if (layer < 1 || layer > SAT_MAX_LAYERS) return sat_fail(ctx, SAT_EINVAL, "sat_gat_bwd: layer must be in [1, %d]", SAT_MAX_LAYERS);
    GatState &G = ctx->gat[layer];
    if (G.d_out <= 0 || G.valid.size() != (size_t)ctx->M) return sat_fail(ctx, SAT_ESTATE, "sat_gat_bwd: sat_gat_fwd has not run for layer %d", layer);
    for (int m = (part == SAT_ALL_PARTS ? 0 : part); m < (part == SAT_ALL_PARTS ? ctx->M : part + 1); ++m)
        if (!G.valid[m]) return sat_fail(ctx, SAT_ESTATE, "sat_gat_bwd: sat_gat_fwd has not run for partition %d of layer %d", m, layer);
    const int32_t d_out = G.d_out, ld_z = round_up4(d_out);
    if (d_in <= 0 || !W || !a_src || !a_dst || !g_W || !g_a_src || !g_a_dst || !g_b) return sat_fail(ctx, SAT_EINVAL, "sat_gat_bwd: null parameter or gradient array");
    if (accumulate != 0 && accumulate != 1) return sat_fail(ctx, SAT_EINVAL, "sat_gat_bwd: accumulate must be 0 or 1");
    if (v.n_rows > 0 && (!g_out || !h_in || !ok_ld(ld_g, d_out) || !ok_ld(ld_in, d_in) || !aligned16(g_out) || !aligned16(h_in) ||
                         (G.relu && (!h_out || !ok_ld(ld_out, d_out)))))
        return sat_fail(ctx, SAT_EINVAL, "sat_gat_bwd: null / misaligned g_out / h_in / h_out or bad leading dimension");
    if (v.n_halo > 0 && (!h_halo || !ok_ld(ld_halo, d_in) || !aligned16(h_halo))) return sat_fail(ctx, SAT_EINVAL, "sat_gat_bwd: null / misaligned h_halo");
    if (g_in && v.n_rows > 0 && (!ok_ld(ld_gin, d_in) || !aligned16(g_in))) return sat_fail(ctx, SAT_EINVAL, "sat_gat_bwd: misaligned g_in or bad ld_gin");
    const int64_t n = ctx->n;
    float *z_in = (float *)G.z_in.p, *z_halo = (float *)G.z_halo.p;
    float *s_in = (float *)G.scal.p, *s_dst = s_in + n, *s_halo = s_dst + n;
    // scratch of the call, by row / halo position / entry of the selection: dot products (then dpre), entries of the inner and
    // of the halo column side, D, dZ, ds_dst, ds_src
    const int64_t ent0 = ctx->h_lnnz_off[v.p0], cut0 = ctx->h_hrow_off[v.p0];
    const size_t f_rows = (size_t)(v.n_rows > 0 ? v.n_rows : 1), f_halo = (size_t)(v.n_halo > 0 ? v.n_halo : 1), f_ent = (size_t)v.lnnz + 2,
                 f_cut = (size_t)v.hnnz + 2;
    SAT_TRY(sat_ensure(ctx, ctx->buf_gat_items, (2 * f_ent + f_cut) * sizeof(double) + 32));
    double *dots = (double *)ctx->buf_gat_items.p;
    int2 *ent_in = (int2 *)(dots + f_ent), *ent_halo = ent_in + f_ent;
    SAT_TRY(sat_ensure(ctx, ctx->buf_gat, ((2 * f_rows + f_halo) * ld_z + 2 * f_rows + f_halo + 64) * sizeof(float)));
    float *D = (float *)ctx->buf_gat.p, *dz_in = D + f_rows * ld_z, *dz_halo = dz_in + f_rows * ld_z;
    float *ds_dst = dz_halo + f_halo * ld_z, *ds_in = ds_dst + f_rows, *ds_halo = ds_in + f_rows;
    // virtual bases indexed by partition-major row / global halo position / entry
    const float *Db = D - (int64_t)v.row0 * ld_z;
    float *dz_in_b = dz_in - (int64_t)v.row0 * ld_z, *dz_halo_b = dz_halo - v.halo0 * ld_z;
    float *ds_dst_b = ds_dst - v.row0, *ds_in_b = ds_in - v.row0, *ds_halo_b = ds_halo - v.halo0;
    double *dots_b = dots - ent0;
    int2 *ent_in_b = ent_in - ent0, *ent_halo_b = ent_halo - cut0;
    const int32_t d4 = (d_out + 3) / 4;
    if (v.n_rows > 0) {
        SAT_TRY(sat_mask_rows(ctx, g_out, ld_g, v.n_rows, d_out, nullptr, 0, D, ld_z, g_b, accumulate, G.relu ? h_out : nullptr, ld_out));
        ProfScope prof(ctx, SATK_GAT, 0.0, 0.0);
        const int4 *items = nullptr;
        int64_t n_items = 0;
        SAT_TRY(sat_spmm_items(ctx, v, 0, d_out, &items, &n_items));
#define CALL(GG, NV)                                                                                                                            \
    sat_pdl(ctx->stream, k_gat_dots<GG, NV>, (unsigned)cdiv64(n_items * GG, 256), 256, 0)(items, (int32_t)n_items, ctx->lenc, ctx->n, d4, z_in, z_halo, \
                                                                                     (uint32_t)(ld_z / 4), Db, dots_b)
        if (d4 <= 8) CALL(8, 1);
        else if (d4 <= 16) CALL(16, 1);
        else if (d4 <= 32) CALL(32, 1);
        else if (d4 <= 64) CALL(32, 2);
        else if (d4 <= 128) CALL(32, 4);
        else CALL(32, 8);
#undef CALL
        SAT_LAUNCHED(ctx);
        const int64_t l0 = ctx->h_gat_long_off[v.p0], n_long = ctx->h_gat_long_off[v.p1] - l0;
        const unsigned grid = (unsigned)(n_long + cdiv64((int64_t)v.n_rows * GAT_TEAM, 256));
        sat_pdl(ctx->stream, k_gat_rows, grid, 256, 0)(ctx->lrowptr, (const int2 *)G.ent.p, ctx->n, v.row0, v.n_rows, ctx->gat_long + l0, (int32_t)n_long, s_in,
                                                  s_halo, s_dst, z_in, z_halo, ld_z, d_out, dots_b, ds_dst_b);
        SAT_LAUNCHED(ctx);
        sat_pdl(ctx->stream, k_gat_cols, grid, 256, 0)(ctx->lrowptr, ctx->inner_cnt, v.row0, v.n_rows, ctx->gat_long + l0, (int32_t)n_long, ctx->lenc,
                                                  ctx->gat_rev, (const int2 *)G.ent.p, dots_b, ent_in_b, ds_in_b);
        SAT_LAUNCHED(ctx);
        SpmmEpilogue ep;
        ep.s1 = ds_in_b;
        ep.v1 = a_src;
        ep.s2 = ds_dst_b;
        ep.v2 = a_dst;
        SAT_TRY(sat_spmm_entries(ctx, v, 1, d_out, ent_in_b, Db, ld_z, nullptr, 0, dz_in_b, ld_z, ep));
    } else if (!accumulate) {
        SAT_CUDA(ctx, cudaMemsetAsync(g_b, 0, (size_t)d_out * sizeof(float), ctx->stream));
    }
    if (v.n_halo > 0 && v.n_rows > 0) {
        ProfScope prof(ctx, SATK_GAT, 0.0, 0.0);
        sat_pdl(ctx->stream, k_gat_cols, (unsigned)(v.n_hlong + cdiv64(v.n_halo * GAT_TEAM, 256)), 256, 0)(
            ctx->hrow_ptr, nullptr, v.halo0, v.n_halo, ctx->hlong ? ctx->hlong + v.hlong0 : nullptr, v.n_hlong, ctx->hrow_pos, ctx->gat_hmap,
            (const int2 *)G.ent.p, dots_b, ent_halo_b, ds_halo_b);
        SAT_LAUNCHED(ctx);
        SpmmEpilogue ep;
        ep.s1 = ds_halo_b;
        ep.v1 = a_src;
        SAT_TRY(sat_spmm_entries(ctx, v, 3, d_out, ent_halo_b, Db, ld_z, nullptr, 0, dz_halo_b, ld_z, ep));
    }
    const int64_t halo_rows = v.n_rows > 0 ? v.n_halo : 0;
    // parameter gradients
    SAT_TRY(gat_tn(ctx, v.n_rows, d_in, d_out, h_in, ld_in, dz_in, ld_z, g_W, accumulate));
    if (halo_rows > 0) SAT_TRY(gat_tn(ctx, halo_rows, d_in, d_out, h_halo, ld_halo, dz_halo, ld_z, g_W, 1));
    SAT_TRY(gat_wcolsum(ctx, z_in + (int64_t)v.row0 * ld_z, ld_z, v.n_rows, d_out, ds_in, g_a_src, ds_dst, g_a_dst, accumulate));
    if (halo_rows > 0) SAT_TRY(gat_wcolsum(ctx, z_halo + v.halo0 * ld_z, ld_z, halo_rows, d_out, ds_halo, g_a_src, nullptr, nullptr, 1));
    // input gradient of the inner rows
    if (g_in && v.n_rows > 0) SAT_TRY(gat_nt(ctx, v.n_rows, d_in, d_out, dz_in, ld_z, W, g_in, ld_gin));
    return SAT_OK;
}
