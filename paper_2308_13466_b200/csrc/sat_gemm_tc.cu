// Dense contractions on the 5th-generation tensor cores (tcgen05.mma, accumulators in TMEM, operands staged in shared
// memory by TMA) with fp32-level accuracy from a split of either operand into two terms:
//     x = hi + lo                                               (kind::tf32: |x - hi - lo| <= 2^-21 |x|; kind::f16, scaled by powers of two: see split_f16)
//     A B ~= Ah Bh + Ah Bl + Al Bh                              (three MMAs per k-step, fp32 accumulate)
// Activations and weights stay plain fp32 in global memory: TMA brings the fp32 tiles into shared memory.  For TF32 terms
// the converter warps write the residual tiles next to them, element-wise, so the swizzled layout never has to be decoded
// (see "TF32 split of a shared-memory tile" below for the two variants); halves take the place of the raw values.  Weights
// are repacked into the K-major operand layout: once per call, for the layers of an epoch over several partitions once per
// epoch, for a predictor with a version once per version.
//
//   k_gemm_tc_k   C[M x N] = A[M x K] B[N x K]^T   both operands K-major, 64-byte swizzle, BLOCK_K = 16, persistent CTA pairs
//                 (layer transform, recurrent gates with two A operands, input projections, predictor output, input gradient)
//   k_gemm_tc_h   the same on half-precision pairs, 128-byte swizzle, BLOCK_K = 32, for long contractions (sat_tc_half)
//   k_lstm_seq    LSTM steps over cached input projections, half-precision pairs
//   k_gemm_tc_mn  C[M x N] = A[R x M]^T B[R x N]   both operands MN-major, 128-byte swizzle with 32-byte atoms, split over R
//                 (weight gradient)
// Warp roles of k_gemm_tc_k (512 threads): warp 0 = TMA producer, warp 1 = TMEM owner + MMA issuer, then 6 converter and
// 8 epilogue warps (two per TMEM lane quadrant), or 2 + 12 with a gathered residual (K = h).  k_gemm_tc_mn:
// warps 0 / 1 as above, warps 2..9 convert during the main loop and then run the epilogue.  Every mbarrier wait is
// bounded; a timeout raises a status word and lets the CTA drain (TMEM is freed, the kernel returns).
#include <cuda.h>
#include <cuda_fp16.h>

#include "sat_internal.h"

#include <algorithm>

#define TC_BM 128
#define TC_BK 16          /* fp32 elements per k-block: 64-byte rows */
#define TCH_BK 32         /* K-major kernel on half-precision pairs: elements per k-block, 128-byte rows of fp32 and of [hi | lo] halves alike */
#define TC_WAIT_LIMIT (1u << 22)

// =====================================================================================
// PTX wrappers
// =====================================================================================
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// bounded wait: returns false (and raises *dead) when the limit is hit or another thread already gave up.
// SLEEP_NS > 0 backs off between polls: a spinning warp otherwise takes issue slots from the warps doing the work
// (the epilogue shares its schedulers with the waiting converter warps).
template <int SLEEP_NS = 0>
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *dead, int *status)
{
    const uint32_t addr = smem_u32(bar);
    for (uint32_t it = 0; it < TC_WAIT_LIMIT; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t"
            ".reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t"
            "}"
            : "=r"(ok)
            : "r"(addr), "r"(parity)
            : "memory");
        if (ok) return true;
        if (*dead) return false;
        if (SLEEP_NS > 0) __nanosleep(SLEEP_NS);
    }
    *dead = 1;
    atomicOr(status, 1);
    return false;
}
// whole-warp wait: lane 0 polls, then every lane observes the completed phase itself (one immediate try_wait each), so
// that a waiting warp issues one poll per round instead of 32
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, volatile int *dead, int *status, int lane)
{
    int ok = 1;
    if (lane == 0) ok = mbar_wait<64>(bar, parity, dead, status) ? 1 : 0;
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (!ok) return false;
    return mbar_wait(bar, parity, dead, status);
}
// every lane waits; the result is that of the whole warp
__device__ __forceinline__ bool mbar_wait_all(uint64_t *bar, uint32_t parity, volatile int *dead, int *status)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, dead, status));
}
__device__ __forceinline__ void tma_load_2d(void *smem_dst, const CUtensorMap *map, uint64_t *bar, int32_t x, int32_t y)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
                     smem_u32(smem_dst)),
                 "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, const void *smem_src, int32_t x, int32_t y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"((uint64_t)map), "r"(smem_u32(smem_src)),
                 "r"(x), "r"(y)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// waits until at most `N` of this thread's bulk stores still read their shared-memory source
template <int N>
__device__ __forceinline__ void tma_store_wait_read()
{
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// One warp; GROUP = 2: one warp of each CTA of the pair, which get the same columns
template <int GROUP>
__device__ __forceinline__ void tc_alloc(uint32_t *base, uint32_t cols)
{
    if (GROUP == 2) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(base)), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(base)), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
}
template <int GROUP>
__device__ __forceinline__ void tc_dealloc(uint32_t base, uint32_t cols)
{
    if (GROUP == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// arrives on the barrier once this thread's MMAs so far have completed; GROUP = 2: on that of both CTAs of the pair
template <int GROUP>
__device__ __forceinline__ void tc_commit(uint64_t *bar)
{
    if (GROUP == 2)
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
                     "h"((uint16_t)3)
                     : "memory");
    else
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// D (+)= A B.  USE_A: what becomes of the A tile in the tensor core's operand collector -- 1: it stays, 2: it is taken from there for
// the last time.  (The two products with A hi read it from shared memory once: 1.3 % of a 179250 x 512 x 512 contraction.)
#define TC_MMA_ASM(G, KIND, COLLECTOR)                                                                 \
    asm volatile(                                                                                      \
        "{\n\t"                                                                                        \
        ".reg .pred p;\n\t"                                                                            \
        "setp.ne.b32 p, %4, 0;\n\t"                                                                    \
        "tcgen05.mma.cta_group::" G ".kind::" KIND COLLECTOR " [%0], %1, %2, %3, p;\n\t"                   \
        "}" ::"r"(tmem_d),                                                                             \
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)                                            \
        : "memory")
template <int USE_A, int GROUP>
__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    if (GROUP == 2) {
        if (USE_A == 1) TC_MMA_ASM("2", "tf32", ".collector::a::fill");
        else if (USE_A == 2) TC_MMA_ASM("2", "tf32", ".collector::a::lastuse");
        else TC_MMA_ASM("2", "tf32", "");
    } else {
        if (USE_A == 1) TC_MMA_ASM("1", "tf32", ".collector::a::fill");
        else if (USE_A == 2) TC_MMA_ASM("1", "tf32", ".collector::a::lastuse");
        else TC_MMA_ASM("1", "tf32", "");
    }
}
// the same with half-precision operands
template <int USE_A, int GROUP>
__device__ __forceinline__ void tc_mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    if (GROUP == 2) {
        if (USE_A == 1) TC_MMA_ASM("2", "f16", ".collector::a::fill");
        else if (USE_A == 2) TC_MMA_ASM("2", "f16", ".collector::a::lastuse");
        else TC_MMA_ASM("2", "f16", "");
    } else {
        if (USE_A == 1) TC_MMA_ASM("1", "f16", ".collector::a::fill");
        else if (USE_A == 2) TC_MMA_ASM("1", "f16", ".collector::a::lastuse");
        else TC_MMA_ASM("1", "f16", "");
    }
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t *r)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, "
        "%19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// shared-memory matrix descriptor: start address, leading / stride byte offsets (16-byte units), sm_100 version, swizzle mode
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes, uint32_t layout_type)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)layout_type << 61;
    return d;
}

// instruction descriptor for kind::tf32 (TF32 operands in 32-bit containers, fp32 accumulation)
__host__ __device__ inline uint32_t make_idesc(int m, int n, int a_mn_major, int b_mn_major)
{
    uint32_t d = 0;
    d |= 1u << 4;   // D format: f32
    d |= 2u << 7;   // A format: tf32
    d |= 2u << 10;  // B format: tf32
    d |= (uint32_t)a_mn_major << 15;
    d |= (uint32_t)b_mn_major << 16;
    d |= (uint32_t)(n >> 3) << 17;
    d |= (uint32_t)(m >> 4) << 24;
    return d;
}

// kind::f16 with half-precision operands, both K-major, fp32 accumulation
__host__ __device__ inline uint32_t make_idesc_f16(int m, int n) { return 1u << 4 | (uint32_t)(n >> 3) << 17 | (uint32_t)(m >> 4) << 24; }

// Two-term split into half precision, x s = hi + lo + e with |e| <= 2^-22 |x s| wherever |x s| is not small: both terms are rounded to nearest,
// and a power of two s brings the largest element of the operand's row to [2^14, 2^15), so that terms are subnormal (and e
// is at most 2^-25) only for elements 2^18 times smaller than that one.  Closer than the TF32 split (2^-21 |x|, and hi truncated) down to there, on
// operands of half the size and at twice the rate; below 2^-19 of its row's largest element the TF32 split keeps more of an element, which shows
// only in sums where that largest one meets a near-zero element of the other operand.  Two elements at a time: the first in the low half.
__device__ __forceinline__ void split_f16(float x0, float x1, uint32_t &hi, uint32_t &lo)
{
    const __half2 h = __floats2half2_rn(x0, x1);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(x0 - f.x, x1 - f.y);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}
// An accumulator is multiplied by the inverse scales of its column and of its row, one after the other: their product may lie outside of fp32.  2^SCALE_SHIFT goes
// over from the column's to the row's, so that the first product stays inside for columns up to 2^118.
#define SCALE_SHIFT 14
// biased exponent of the power of two that brings the elements of a row, the largest of which has this biased exponent, below 2^15; the
// inverse has 254 minus it.  One for zeros, infinities and NaN.
__device__ __forceinline__ uint32_t f16_scale_exponent(uint32_t largest)
{
    const int e = 268 - (int)largest;
    return largest == 0 || largest == 255 ? 127u : (uint32_t)(e > 253 ? 253 : e);
}

// (x s) s2 + y by packed operations (each component rounded as by itself)
__device__ __forceinline__ float4 scaled_add(const uint32_t *x, const float4 &s, const float4 &y, const float2 &s2)
{
    const float2 lo = __fmul2_rn(make_float2(__uint_as_float(x[0]), __uint_as_float(x[1])), make_float2(s.x, s.y));
    const float2 hi = __fmul2_rn(make_float2(__uint_as_float(x[2]), __uint_as_float(x[3])), make_float2(s.z, s.w));
    const float2 a = __ffma2_rn(lo, s2, make_float2(y.x, y.y)), b = __ffma2_rn(hi, s2, make_float2(y.z, y.w));
    return make_float4(a.x, a.y, b.x, b.y);
}

// =====================================================================================
// TF32 split of a shared-memory tile, element-wise (the swizzled layout never has to be decoded).
//
// The tensor core reads an fp32 container as TF32 by ignoring the low 13 mantissa bits.  split_tile_residual uses that:
// the raw tile already is the "hi" operand (hi = x with those bits cleared) and only lo = tf32_rn(x - hi) is written, to
// the second tile (x - hi is exact; rounding lo to nearest keeps the representation error |x - hi - lo| <= 2^-21 |x|
// free of bias).  split4 rounds hi to nearest as well and the weight gradient rewrites the raw tile in place: hi and lo are then
// symmetric around x, which matters for the weight gradient (a small difference of ~1e5 signed terms per element).
// =====================================================================================
__device__ __forceinline__ float tf32_round(float x)
{
    return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);  // round half away from zero to 10 mantissa bits
}
__device__ __forceinline__ float tf32_residual(float x) { return tf32_round(x - __uint_as_float(__float_as_uint(x) & 0xFFFFE000u)); }
__device__ __forceinline__ float4 residual4(const float4 &x)
{
    return make_float4(tf32_residual(x.x), tf32_residual(x.y), tf32_residual(x.z), tf32_residual(x.w));
}
__device__ __forceinline__ void split4(const float4 &x, float4 &h, float4 &l)
{
    h.x = tf32_round(x.x); l.x = tf32_round(x.x - h.x);
    h.y = tf32_round(x.y); l.y = tf32_round(x.y - h.y);
    h.z = tf32_round(x.z); l.z = tf32_round(x.z - h.z);
    h.w = tf32_round(x.w); l.w = tf32_round(x.w - h.w);
}
// two 16-byte chunks per thread and iteration, loads first (the loops are latency-bound otherwise)
__device__ __forceinline__ void split_tile_residual(const uint8_t *hi_tile, uint8_t *lo_tile, uint32_t bytes, int tid, int nthreads)
{
    const uint32_t step = (uint32_t)nthreads * 16;
    for (uint32_t off = (uint32_t)tid * 16; off < bytes; off += 2 * step) {
        const uint32_t off2 = off + step;
        const bool two = off2 < bytes;
        const float4 x1 = *reinterpret_cast<const float4 *>(hi_tile + off);
        float4 x2 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (two) x2 = *reinterpret_cast<const float4 *>(hi_tile + off2);
        *reinterpret_cast<float4 *>(lo_tile + off) = residual4(x1);
        if (two) *reinterpret_cast<float4 *>(lo_tile + off2) = residual4(x2);
    }
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// A warp's arrival on a barrier that the MMA issuer waits for.  CTAS = 1: every lane arrives.  2: lane 0 does, on the barrier at the same
// place in CTA 0 of the pair, without a scope, that is at CTA scope.  An assumption rests on that: that shared-memory writes in front of
// the proxy fence and TMEM reads in front of their wait are done for the pair's MMAs when the arrival is seen.  The memory model does not
// say so across two CTAs; it is the form in which CUTLASS's cluster barriers arrive at the other CTA of a pair, and
// tests/test_gpu_edges.py compares pair launches with single CTAs bit by bit.  (With .release.cluster the arrival also waits for
// everything else the SM has in flight, 1.4 us: a 179250 x 512 x 512 contraction took 490 us instead of 370; waits that acquire at
// cluster scope, which would be half of it, cost 0.3-0.5 % of an epoch.)
template <int CTAS>
__device__ __forceinline__ void mbar_arrive_warp(uint64_t *bar, int lane)
{
    if (CTAS == 1) {
        mbar_arrive(bar);
        return;
    }
    __syncwarp();
    if (lane == 0)
        asm volatile(
            "{\n\t"
            ".reg .b32 a;\n\t"
            "mapa.shared::cluster.u32 a, %0, 0;\n\t"
            "mbarrier.arrive.shared::cluster.b64 _, [a];\n\t"
            "}" ::"r"(smem_u32(bar))
            : "memory");
}
// lane 0's arrival on the same barriers with single CTAs too
template <int CTAS>
__device__ __forceinline__ void mbar_arrive_lane0(uint64_t *bar, int lane)
{
    __syncwarp();
    if (CTAS == 2) mbar_arrive_warp<CTAS>(bar, lane);
    else if (lane == 0) mbar_arrive(bar);
}
// make generic-proxy shared-memory writes visible to the tensor-core (async) proxy
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// =====================================================================================
// K-major kernel
// =====================================================================================
struct TcEpilogue {
    // (half-precision pairs)
    const uint32_t *row_max; // [row_parts][row_stride] bits of the largest magnitude in each part of a row of A
    int64_t row_stride;
    int32_t row_parts;
    uint32_t row_least;      // what the largest magnitude is taken to be at least (bits)
    int32_t k1, k2;          // terms of the A operands
    const float *unscale;    // inverse scale of every column of B, see TcWeights
    float *C;
    int64_t ldc;
    const float *bias;
    int relu;
    uint32_t *mask_out;
    int32_t mask_words;
    const uint32_t *mask_in;
    int32_t mask_in_words;
    const float *resid;  // C += resid[resid_idx[row]]  (row gather)
    const int32_t *resid_idx;
    int64_t ld_resid;
    int32_t lstm_h;      // > 0: fused recurrent cell, C = hidden state [M x lstm_h], lstm_c = cell state (LSTM only)
    int lstm_first;
    float *lstm_c;       // cell state in the blocked layout of sat_cell_offset
    int32_t proj_h;      // (EPI_PROJ) hidden units: C is a projection plane, see sat_proj_floats
    RowMaxOut push_max;  // (EPI_PUSH; or none) largest magnitude of every pushed row: part 2 (column tile) + (half of the epilogue warps), by slot
    float *push_dst;     // (EPI_PUSH) row i is also written to push_dst + push_slot[i] * ld_push when push_slot[i] >= 0
    const int32_t *push_slot;
    int64_t ld_push;
    const int32_t *tile_order;  // row tile walked at position i of the schedule (null: i itself)
};

// Row tile (of 128 rows per CTA of a unit) of schedule position t: the persistent CTAs or CTA pairs walk positions unit, unit + units, ...;
// a permutation lets the caller choose which row tiles run at the same time (results do not depend on it).
__device__ __forceinline__ int64_t tck_row_tile(const TcEpilogue &ep, int64_t t, int32_t n_tiles_n)
{
    const int64_t rt = t / n_tiles_n;
    return ep.tile_order ? (int64_t)__ldg(ep.tile_order + rt) : rt;
}

#define TCK_STAGES_MAX 8
struct TcShared {
    uint64_t full[TCK_STAGES_MAX];       // TMA bytes of the stage have landed
    uint64_t conv[TCK_STAGES_MAX];       // the converter threads have split the stage
    uint64_t empty[TCK_STAGES_MAX];      // the MMAs reading the stage have completed
    uint64_t acc_full[2];   // accumulator buffer holds a finished tile
    uint64_t acc_empty[2];  // accumulator buffer has been drained by the epilogue
    uint32_t tmem_base;
    int dead;
};

/* 512 threads, 128 registers each: warp 0 TMA, warp 1 MMA, then the converter warps, then the epilogue warps.  The split
 * between converters and epilogue depends on the epilogue variant (TckCfg): the one with a gathered residual has four
 * k-blocks per tile (K = h) and an epilogue bound by latency, so it runs 2 + 12 instead of 6 + 8.
 * The converter warps work in two groups on alternate k-blocks, so two stages are being split at any time.  The stage
 * count is even, hence a stage is always handled by the same group and each group meets the phases of its stages in
 * order (a parity wait must never be more than one phase ahead of its barrier). */
#define TCK_THREADS 512
#define TCK_CONV_GROUPS 2
/* The weights' residual plane is made once by k_split_weights and fetched by TMA next to the raw plane: B is the same for
 * every row tile, and splitting its tile again per k-block cost the converters twice what the A tile costs (measured:
 * K = 256 transform 132 -> 118 us, K = 64 LSTM step 98 -> 85 us) for 16 KB more L2 -> SM traffic per k-block. */
#define TCK_B_PRESPLIT 1

// Epilogue variants.  EPI_RESID streams a per-row side operand from global memory (gathered residual rows): a ring of 32 x 32 side tiles
// per epilogue warp in shared memory, filled by cp.async ahead of the consumer.  It contracts over a small K (the predictor width), so
// it gives up main-loop stages for the ring.  (Four slots with the results staged in place, which fits with eight epilogue
// warps: 1018 -> 1232 us at 612257 nodes; the twelve warps are worth more than the deeper ring.)
enum { EPI_PLAIN = 0, EPI_RESID = 1, EPI_LSTM = 2, EPI_PROJ = 3, EPI_PUSH = 4, EPI_GRU = 5 };   // EPI_PUSH = EPI_PLAIN + a second copy of the rows that have a cache slot
template <int EPI> struct TckCfg { static constexpr int ring = 0, conv_warps = 6, epi_warps = 8, out_bytes = epi_warps * 4096; };
template <> struct TckCfg<EPI_RESID> { static constexpr int ring = 1, conv_warps = 2, epi_warps = 12, out_bytes = epi_warps * 4096; };
template <> struct TckCfg<EPI_LSTM> { static constexpr int ring = 0, conv_warps = 6, epi_warps = 8, out_bytes = 0; };
template <> struct TckCfg<EPI_GRU> : TckCfg<EPI_LSTM> {};
template <> struct TckCfg<EPI_PROJ> : TckCfg<EPI_LSTM> {};

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gsrc, bool valid)
{
    // src-size 0 writes 16 zero bytes without reading the source
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(smem_dst)), "l"(gsrc), "r"(valid ? 16u : 0u) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Persistent: each CTA (CTAS = 1) or pair of CTAs (2) walks tiles unit, unit + units, ... of 128 or 256 rows.  A pair's MMA
// (cta_group::2) multiplies the 128 rows of either CTA with all columns of B, of which each CTA holds half: per k-block of 16 at 256
// columns the tensor core reads 24 KB and the TMA writes 16 KB less per SM than with single CTAs, where shared memory (128 KB per k-block
// at 128 B per clock) and not the tensor work (96 KB worth) was the bound; and the ring holds six stages instead of four.  Measured:
// 169343 x 256 x 256 117 -> 105 us, 179250 x 512 x 512 413 -> 370, 612257 x 256 x 256 415 -> 358.  The shared-memory ring of k-block stages
// and the two TMEM accumulator buffers let the TMA loads, the TF32 split, the MMAs and the epilogue of consecutive tiles
// overlap.  A and B arrive as raw fp32 tiles, which the tensor core reads as the hi operands; the converters write the
// residual tiles.  The epilogue is a template parameter (plain bias / ReLU / mask, gathered residual, fused LSTM cell)
// and runs on eight or twelve warps, two or three per TMEM lane quadrant taking 32-column chunks in turn: with one warp
// per scheduler the epilogue was bound by instruction issue and load latency (9 - 14 us per 128 x 256 tile, longer than
// the main loop of a K = 256 tile).
template <int EPI, int CTAS>
__global__ void __launch_bounds__(TCK_THREADS, 1)
k_gemm_tc_k(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapA2, const __grid_constant__ CUtensorMap mapB,
            const __grid_constant__ CUtensorMap mapBlo, const __grid_constant__ CUtensorMap mapC, int use_tma_store, uint32_t stages, int64_t M, int32_t N, int32_t nkb1, int32_t nkb2, int32_t bn, int32_t n_tiles_n, int64_t n_tiles, TcEpilogue ep, int *status)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t a_bytes = TC_BM * TC_BK * 4;  // one plane of the A tile: 128 rows x 64 B
    const uint32_t b_bytes = (uint32_t)bn / CTAS * TC_BK * 4;  // a CTA of a pair holds half of the columns
    const uint32_t stage_bytes = 2 * a_bytes + 2 * b_bytes;  // [A hi | A lo | B hi | B lo]
    const uint32_t rank = CTAS == 2 ? blockIdx.x & 1u : 0u;  // in the pair; CTA 0 issues the MMAs of both
    const int64_t unit = blockIdx.x / CTAS, units = gridDim.x / CTAS;
    constexpr int RING = TckCfg<EPI>::ring;
    uint8_t *out_stage = smem + (size_t)stages * stage_bytes;
    uint8_t *ring_base = out_stage + TckCfg<EPI>::out_bytes;
    constexpr int CONV_THREADS = TckCfg<EPI>::conv_warps * 32, CONV_GROUP_THREADS = CONV_THREADS / TCK_CONV_GROUPS;
    constexpr int EPI_WARPS = TckCfg<EPI>::epi_warps, EPI_WARP0 = 2 + TckCfg<EPI>::conv_warps;
    constexpr int CHUNK_STEP = 32 * (EPI_WARPS / 4);  // the EPI_WARPS / 4 warps of a TMEM lane quadrant take 32-column chunks in turn
    static_assert(64 + CONV_THREADS + EPI_WARPS * 32 == TCK_THREADS && EPI_WARP0 % 4 == 0 && EPI_WARPS % 4 == 0, "warp roles");
    TcShared *sh = (TcShared *)(ring_base + (size_t)EPI_WARPS * RING * 4096);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t nkb = nkb1 + nkb2;
    const uint32_t acc_cols = 256;  // column stride between the two accumulator buffers

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < stages; ++s) {
            mbar_init(&sh->full[s], 1);
            mbar_init(&sh->conv[s], CTAS == 2 ? 2 * (CONV_GROUP_THREADS / 32) : CONV_GROUP_THREADS);
            mbar_init(&sh->empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh->acc_full[i], 1);
            mbar_init(&sh->acc_empty[i], CTAS == 2 ? 2 * EPI_WARPS : EPI_WARPS * 32);
        }
        sh->dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        tc_alloc<CTAS>(&sh->tmem_base, 512u);
    }
    tc_fence_before();
    __syncthreads();
    if (CTAS == 2) cluster_sync();   // the other CTA's barriers are initialised and its TMEM is allocated
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    volatile int *dead = &sh->dead;
    sat_grid_wait();   // everything above is set-up of this block; no global memory has been touched

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            uint32_t s = 0, ph = 0;
            for (int64_t t = unit; t < n_tiles; t += units) {
                const int32_t m0 = ((int32_t)tck_row_tile(ep, t, n_tiles_n) * CTAS + (int32_t)rank) * TC_BM;   // CTA `rank` holds the rank-th 128 rows
                const int32_t n0 = (int32_t)(t % n_tiles_n) * bn + (int32_t)rank * (bn / CTAS);
                for (int32_t kb = 0; kb < nkb; ++kb) {
                    if (!mbar_wait(&sh->empty[s], ph ^ 1u, dead, status)) goto done;
                    uint8_t *st = smem + (size_t)s * stage_bytes;
                    mbar_expect_tx(&sh->full[s], a_bytes + (TCK_B_PRESPLIT ? 2 * b_bytes : b_bytes));
                    if (kb < nkb1) tma_load_2d(st, &mapA, &sh->full[s], kb * TC_BK, m0);
                    else tma_load_2d(st, &mapA2, &sh->full[s], (kb - nkb1) * TC_BK, m0);
                    tma_load_2d(st + 2 * a_bytes, &mapB, &sh->full[s], kb * TC_BK, n0);
                    if (TCK_B_PRESPLIT) tma_load_2d(st + 2 * a_bytes + b_bytes, &mapBlo, &sh->full[s], kb * TC_BK, n0);
                    if (++s == stages) s = 0, ph ^= 1u;
                }
            }
            // the pair's MMAs have signalled every stage: nothing arrives here any more once both CTAs may exit
            for (uint32_t i = 0; CTAS == 2 && i < stages; ++i) {
                if (!mbar_wait(&sh->empty[s], ph ^ 1u, dead, status)) goto done;
                if (++s == stages) s = 0, ph ^= 1u;
            }
        }
    } else if (warp == 1 && rank == 0) {
        // ---------------- MMA issuer ----------------
        // The whole warp walks the k-blocks and an elected lane issues: the operands of the instructions are then known to be uniform.
        // (One lane doing all of it took 0.4 us per k-block, which bound the narrow tiles: 169343 x 40, K = 256: 70 -> 62 us.)
        const uint32_t idesc = make_idesc(TC_BM * CTAS, bn, 0, 0);
        const uint64_t desc0 = make_desc(smem_u32(smem), 16, 512, 4);
        uint32_t s = 0, ph = 0, lt = 0;
        for (int64_t t = unit; t < n_tiles; t += units, ++lt) {
            const uint32_t buf = lt & 1u;
            if (!mbar_wait_all(&sh->acc_empty[buf], ((lt >> 1) & 1u) ^ 1u, dead, status)) goto done;
            tc_fence_after();
            const uint32_t acc = tmem + buf * acc_cols;
            for (int32_t kb = 0; kb < nkb; ++kb) {
                // the converters arrive on conv[s] only after they have seen full[s] (the TMA bytes) themselves
                if (!mbar_wait_all(&sh->conv[s], ph, dead, status)) goto done;
                tc_fence_after();
                // K-major, 64-byte swizzle: rows 64 B apart, 8-row groups 512 B apart; a k-step (8 values) is 32 B inside the
                // row.  Only the 14-bit start-address field (bytes >> 4) differs between the descriptors of a stage.
                const uint64_t a_hi0 = desc0 + (uint64_t)((s * stage_bytes) >> 4);
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < TC_BK / 8; ++ks) {
                        const uint64_t a_hi = a_hi0 + (uint64_t)(ks * 2);
                        const uint64_t a_lo = a_hi + (a_bytes >> 4);
                        const uint64_t b_hi = a_hi + (2 * a_bytes >> 4);
                        const uint64_t b_lo = b_hi + (b_bytes >> 4);
                        tc_mma<1, CTAS>(acc, a_hi, b_hi, idesc, (kb > 0 || ks > 0) ? 1u : 0u);
                        tc_mma<2, CTAS>(acc, a_hi, b_lo, idesc, 1u);
                        tc_mma<0, CTAS>(acc, a_lo, b_hi, idesc, 1u);
                    }
                    tc_commit<CTAS>(&sh->empty[s]);  // the stage is free once these MMAs have read it
                }
                if (++s == stages) s = 0, ph ^= 1u;
            }
            if (elect_one()) tc_commit<CTAS>(&sh->acc_full[buf]);
        }
    } else if (warp >= 2 && warp < EPI_WARP0) {
        // ---------------- converters: TF32 split of the A and B tiles of every k-block ----------------
        const int grp = (threadIdx.x - 64) / CONV_GROUP_THREADS;
        const int ctid = (threadIdx.x - 64) % CONV_GROUP_THREADS;
        const int64_t my_tiles = unit < n_tiles ? (n_tiles - 1 - unit) / units + 1 : 0;
        uint32_t s = grp, ph = 0;
        for (int64_t it = grp; it < my_tiles * nkb; it += TCK_CONV_GROUPS) {
            if (CTAS == 2 ? !mbar_wait_all(&sh->full[s], ph, dead, status) : !mbar_wait(&sh->full[s], ph, dead, status)) goto done;
            uint8_t *st = smem + (size_t)s * stage_bytes;
            split_tile_residual(st, st + a_bytes, a_bytes, ctid, CONV_GROUP_THREADS);
            if (!TCK_B_PRESPLIT) split_tile_residual(st + 2 * a_bytes, st + 2 * a_bytes + b_bytes, b_bytes, ctid, CONV_GROUP_THREADS);
            fence_async_smem();
            mbar_arrive_warp<CTAS>(&sh->conv[s], lane);
            s += TCK_CONV_GROUPS;
            if (s >= stages) s -= stages, ph ^= 1u;
        }
    } else if (warp >= EPI_WARP0) {
        // ---------------- epilogue ----------------
        // warp w reads TMEM lanes 32 (w % 4) .. +31 = rows of the tile, one row per thread; the warps of a lane quadrant
        // take alternate 32-column chunks.
        constexpr bool LSTM = EPI == EPI_LSTM || EPI == EPI_GRU;   // a recurrent cell
        const int e = warp - EPI_WARP0;
        const int q = warp & 3;
        const int c_first = 32 * (e >> 2);
        uint8_t *obuf = out_stage + e * 4096;
        const bool vec = ((ep.ldc & 3) == 0) && ((((uintptr_t)ep.C) & 15u) == 0);
        const int32_t n4 = (N + 3) & ~3;
        const bool lstm_full = LSTM && (ep.lstm_h & 3) == 0;
        const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);

        // Side-operand ring (RING slots of 32 rows x 128 B, 128-byte swizzle like the store staging tile), private to the
        // warp: cp.async group counting plus __syncwarp is all the synchronisation needed.  The prefetch cursor (pf_*)
        // walks this warp's (tile, chunk) sequence RING chunks ahead of the consumer.
        uint8_t *ring = ring_base + (size_t)e * RING * 4096;
        int64_t pf_t = unit;
        int pf_c = c_first;
        const float *pf_srow = nullptr;
        int32_t pf_lim = 0;
        int32_t pf_idx_next = -1;   // (gathered residual) row index for the tile after the cursor's, fetched a tile early
        uint32_t pf_slot = 0, rd_slot = 0;
        auto tile_row = [&](int64_t t) { return (tck_row_tile(ep, t, n_tiles_n) * CTAS + rank) * TC_BM + q * 32; };   // first row of this warp
        auto pf_enter_tile = [&](int32_t idx_now) {
            // called when the cursor enters tile pf_t; idx_now = gathered row index for this thread's row, or -1
            pf_srow = nullptr;
            if (pf_t < n_tiles) {
                const int64_t prow = tile_row(pf_t) + lane;
                const int32_t pn0 = (int32_t)(pf_t % n_tiles_n) * bn;
                if (prow < M && idx_now >= 0) pf_srow = ep.resid + (int64_t)idx_now * ep.ld_resid + pn0;  // rows padded to 4 floats
                pf_lim = n4 - pn0;
                const int64_t nt = pf_t + units;
                const int64_t nrow = nt < n_tiles ? tile_row(nt) + lane : M;
                pf_idx_next = nrow < M ? __ldg(ep.resid_idx + nrow) : -1;
            }
        };
        auto pf_issue = [&]() {
            // one group per call (possibly empty), so that the consumer's wait count is uniform.  Lane L copies 16-byte
            // piece (L & 7) of rows (L >> 3) + 4 i: an instruction touches 4 rows (4 cache lines) instead of 32, which
            // matters because the load/store unit handles one line per cycle.
            if (pf_t < n_tiles && pf_c < bn) {
                uint8_t *slot = ring + pf_slot * 4096;
                const int piece = lane & 7;
                const bool col_ok = pf_c + 4 * piece < pf_lim;
#pragma unroll
                for (int i = 0; i < 8; ++i) {  // the row pointer lives in the lane that owns the row
                    const int rr = (lane >> 3) + 4 * i;
                    const float *rowp = reinterpret_cast<const float *>(__shfl_sync(0xffffffffu, (unsigned long long)(uintptr_t)pf_srow, rr));
                    const bool valid = rowp != nullptr && col_ok;
                    cp_async16(slot + rr * 128 + ((piece ^ (rr & 7)) << 4), (valid ? rowp : ep.resid) + pf_c + 4 * piece, valid);
                }
                pf_c += CHUNK_STEP;
                if (pf_c >= bn) {
                    pf_c = c_first;
                    pf_t += units;
                    pf_enter_tile(pf_idx_next);
                }
            }
            cp_async_commit();
            pf_slot = pf_slot + 1 == RING ? 0 : pf_slot + 1;
        };
        if (RING > 0 && c_first < bn) {
            int32_t idx0 = -1;
            if (pf_t < n_tiles) {
                const int64_t prow = tile_row(pf_t) + lane;
                if (prow < M) idx0 = __ldg(ep.resid_idx + prow);
            }
            pf_enter_tile(idx0);
#pragma unroll
            for (int i = 0; i < RING; ++i) pf_issue();
        }

        uint32_t lt = 0;
        for (int64_t t = unit; t < n_tiles; t += units, ++lt) {
            const int64_t m0 = tile_row(t) - q * 32;
            const int32_t n0 = (int32_t)(t % n_tiles_n) * bn;
            const uint32_t buf = lt & 1u;
            const int64_t row = m0 + q * 32 + lane;
            const bool row_ok = row < M;
            float *crow = ep.C + row * ep.ldc;
            float *prow = nullptr;   // (EPI_PUSH) this row's home in the cache ring, if it has one
            const int32_t push_slot = EPI == EPI_PUSH && row_ok ? __ldg(ep.push_slot + row) : -1;
            if (EPI == EPI_PUSH && !use_tma_store && push_slot >= 0) prow = ep.push_dst + (int64_t)push_slot * ep.ld_push;
            float4 side[8], cside[2];
            float largest = 0.f;   // (EPI_PUSH) of this thread's chunks
            // previous cell state (GRU: hidden state) of the next chunk, fetched one chunk ahead (two 128-bit loads per thread)
            auto load_cell = [&](int c0) {
                if (LSTM) {
                    cside[0] = cside[1] = zero4;
                    const int32_t j0 = (n0 + c0) >> 2;
                    if (row_ok && lstm_full && !ep.lstm_first && j0 + 7 < ep.lstm_h) {
                        const float *cp = EPI == EPI_GRU ? crow + j0 : ep.lstm_c + sat_cell_offset(row, j0, ep.lstm_h);
                        cside[0] = *reinterpret_cast<const float4 *>(cp);
                        cside[1] = *reinterpret_cast<const float4 *>(cp + 4);
                    }
                }
            };
            if (c_first < bn) load_cell(c_first);
            if (!mbar_wait_warp(&sh->acc_full[buf], (lt >> 1) & 1u, dead, status, lane)) goto done;
            tc_fence_after();
            for (int c0 = c_first; c0 < bn; c0 += CHUNK_STEP) {
                uint32_t r[32];
                tc_ld32(tmem + buf * acc_cols + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, r);
                if (RING > 0) {
                    cp_async_wait<(RING > 0 ? RING - 1 : 0)>();  // every lane's copies of the oldest chunk in the ring have landed ...
                    __syncwarp();                                // ... and are visible to the lane that owns the row
                    const uint8_t *src = ring + rd_slot * 4096 + lane * 128;
#pragma unroll
                    for (int u = 0; u < 8; ++u) side[u] = *reinterpret_cast<const float4 *>(src + ((u ^ (lane & 7)) << 4));
                    rd_slot = rd_slot + 1 == RING ? 0 : rd_slot + 1;
                    __syncwarp();  // all lanes have read the slot: refill it with the chunk RING steps ahead
                    pf_issue();
                }
                if (LSTM) {
                    // packed columns 4 j .. 4 j + 3 are the (i, f, g, o) pre-activations of hidden unit j
                    if (row_ok) {
                        const int32_t j0 = (n0 + c0) >> 2;
                        const bool full = lstm_full && j0 + 7 < ep.lstm_h;
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            float4 b4 = zero4;
                            if (ep.bias) {
                                const float4 bb = __ldg(reinterpret_cast<const float4 *>(ep.bias + n0 + c0) + u);
                                b4.x += bb.x; b4.y += bb.y; b4.z += bb.z; b4.w += bb.w;
                            }
                            r[4 * u] = __float_as_uint(__uint_as_float(r[4 * u]) + b4.x);
                            r[4 * u + 1] = __float_as_uint(__uint_as_float(r[4 * u + 1]) + b4.y);
                            r[4 * u + 2] = __float_as_uint(__uint_as_float(r[4 * u + 2]) + b4.z);
                            r[4 * u + 3] = __float_as_uint(__uint_as_float(r[4 * u + 3]) + b4.w);
                        }
                        float cprev[8];
                        cprev[0] = cside[0].x; cprev[1] = cside[0].y; cprev[2] = cside[0].z; cprev[3] = cside[0].w;
                        cprev[4] = cside[1].x; cprev[5] = cside[1].y; cprev[6] = cside[1].z; cprev[7] = cside[1].w;
                        if (!ep.lstm_first && !full) {
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                if (j0 + u < ep.lstm_h) cprev[u] = EPI == EPI_GRU ? crow[j0 + u] : ep.lstm_c[sat_cell_offset(row, j0 + u, ep.lstm_h)];
                        }
                        if (c0 + CHUNK_STEP < bn) load_cell(c0 + CHUNK_STEP);
                        float sv[8], cv[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            if (EPI == EPI_GRU) {   // (r, z, n from the input, n from the state)
                                const float gr = 1.f / (1.f + expf(-__uint_as_float(r[4 * u])));
                                const float gz = 1.f / (1.f + expf(-__uint_as_float(r[4 * u + 1])));
                                const float gn = tanhf(__uint_as_float(r[4 * u + 2]) + gr * __uint_as_float(r[4 * u + 3]));
                                sv[u] = (1.f - gz) * gn + gz * cprev[u];
                                continue;
                            }
                            const float gi = sigmoid_fast(__uint_as_float(r[4 * u]));
                            const float gf = sigmoid_fast(__uint_as_float(r[4 * u + 1]));
                            const float gg = tanh_fast(__uint_as_float(r[4 * u + 2]));
                            const float go = sigmoid_fast(__uint_as_float(r[4 * u + 3]));
                            cv[u] = gf * cprev[u] + gi * gg;
                            sv[u] = go * tanh_fast(cv[u]);
                        }
                        if (full) {
                            float4 *sd = reinterpret_cast<float4 *>(ep.C + row * ep.ldc + j0);
                            if (EPI != EPI_GRU) {
                                float4 *cd = reinterpret_cast<float4 *>(ep.lstm_c + sat_cell_offset(row, j0, ep.lstm_h));
                                cd[0] = make_float4(cv[0], cv[1], cv[2], cv[3]);
                                cd[1] = make_float4(cv[4], cv[5], cv[6], cv[7]);
                            }
                            sd[0] = make_float4(sv[0], sv[1], sv[2], sv[3]);
                            sd[1] = make_float4(sv[4], sv[5], sv[6], sv[7]);
                        } else {
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                if (j0 + u < ep.lstm_h) {
                                    if (EPI != EPI_GRU) ep.lstm_c[sat_cell_offset(row, j0 + u, ep.lstm_h)] = cv[u];
                                    ep.C[row * ep.ldc + j0 + u] = sv[u];
                                }
                        }
                    }
                    continue;
                }
                uint32_t bits = 0;
                if (row_ok) {
                    // bias is padded with zeros to the tile width and the accumulators of padded columns are exactly zero,
                    // so no column predicate is needed (the stores clip)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float4 b4 = EPI == EPI_RESID ? side[j] : zero4;
                        if (ep.bias) {
                            const float4 bb = __ldg(reinterpret_cast<const float4 *>(ep.bias + n0 + c0) + j);
                            b4.x += bb.x; b4.y += bb.y; b4.z += bb.z; b4.w += bb.w;
                        }
                        r[4 * j] = __float_as_uint(__uint_as_float(r[4 * j]) + b4.x);
                        r[4 * j + 1] = __float_as_uint(__uint_as_float(r[4 * j + 1]) + b4.y);
                        r[4 * j + 2] = __float_as_uint(__uint_as_float(r[4 * j + 2]) + b4.z);
                        r[4 * j + 3] = __float_as_uint(__uint_as_float(r[4 * j + 3]) + b4.w);
                    }
                    if ((EPI == EPI_PLAIN || EPI == EPI_PUSH) && ep.mask_out) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) bits |= (__uint_as_float(r[j]) > 0.f ? 1u : 0u) << j;
                    }
                    if (ep.relu) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(fmaxf(__uint_as_float(r[j]), 0.f));
                    }
                    if (EPI == EPI_PUSH && ep.push_max.p) {
#pragma unroll
                        for (int j = 0; j < 32; j += 2) largest = fmaxf(largest, fmaxf(fabsf(__uint_as_float(r[j])), fabsf(__uint_as_float(r[j + 1]))));
                    }
                    if (EPI == EPI_PLAIN && ep.mask_in) {
                        const int32_t word = (n0 + c0) >> 5;
                        const uint32_t keep = word < ep.mask_in_words ? __ldg(ep.mask_in + row * ep.mask_in_words + word) : 0u;
#pragma unroll
                        for (int j = 0; j < 32; ++j) r[j] = keep >> j & 1u ? r[j] : 0u;
                    }
                }
                if (EPI == EPI_PROJ) {   // a warp's store of a unit is 512 contiguous bytes
                    if (row_ok) {
                        const int32_t j0 = (n0 + c0) >> 2;
                        float4 *dst = reinterpret_cast<float4 *>(ep.C) + ((row >> 7) * ep.proj_h + j0) * 128 + (row & 127);
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (j0 + u < ep.proj_h)
                                dst[u * 128] = make_float4(__uint_as_float(r[4 * u]), __uint_as_float(r[4 * u + 1]), __uint_as_float(r[4 * u + 2]),
                                                           __uint_as_float(r[4 * u + 3]));
                    }
                    continue;
                }
                if (EPI == EPI_PUSH && prow) {   // one full 128-byte line per thread and chunk
#pragma unroll
                    for (int j4 = 0; j4 < 32; j4 += 4) {
                        const int32_t colb = n0 + c0 + j4;
                        if (colb + 3 < N) {
                            *reinterpret_cast<uint4 *>(prow + colb) = make_uint4(r[j4], r[j4 + 1], r[j4 + 2], r[j4 + 3]);
                        } else {
#pragma unroll
                            for (int jj = 0; jj < 4; ++jj)
                                if (colb + jj < N) prow[colb + jj] = __uint_as_float(r[j4 + jj]);
                        }
                    }
                }
                if (use_tma_store) {
                    // stage the 32 x 32 block (128-byte swizzle: 16-byte chunk j of row r sits at chunk j ^ (r & 7)) and
                    // let the TMA write it as whole 128-byte row segments; rows / columns past the matrix are clipped
                    if (lane == 0) tma_store_wait_read<0>();  // the previous block has left the staging tile
                    __syncwarp();
                    uint8_t *dst = obuf + lane * 128;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        *reinterpret_cast<uint4 *>(dst + ((j ^ (lane & 7)) << 4)) = make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) tma_store_2d(&mapC, obuf, n0 + c0, (int32_t)(m0 + q * 32));
                    if (EPI == EPI_PUSH) {
                        // the boundary rows also go to the cache ring, read back from the staged block: every instruction
                        // writes whole 128-byte row segments (the per-thread form touches 32 different lines per instruction)
                        const int piece = lane & 7;
                        const int32_t colb = n0 + c0 + 4 * piece;
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int rr = (lane >> 3) + 4 * i;
                            const int32_t slot = __shfl_sync(0xffffffffu, push_slot, rr);
                            if (slot < 0 || colb >= N) continue;
                            float *pr = ep.push_dst + (int64_t)slot * ep.ld_push;
                            const uint4 x = *reinterpret_cast<const uint4 *>(obuf + rr * 128 + ((piece ^ (rr & 7)) << 4));
                            if (colb + 3 < N) {
                                *reinterpret_cast<uint4 *>(pr + colb) = x;
                            } else {
                                pr[colb] = __uint_as_float(x.x);
                                if (colb + 1 < N) pr[colb + 1] = __uint_as_float(x.y);
                                if (colb + 2 < N) pr[colb + 2] = __uint_as_float(x.z);
                            }
                        }
                    }
                } else if (row_ok) {
#pragma unroll
                    for (int j4 = 0; j4 < 32; j4 += 4) {
                        const int32_t colb = n0 + c0 + j4;
                        if (vec && colb + 3 < N) {
                            *reinterpret_cast<uint4 *>(crow + colb) = make_uint4(r[j4], r[j4 + 1], r[j4 + 2], r[j4 + 3]);
                        } else {
#pragma unroll
                            for (int jj = 0; jj < 4; ++jj)
                                if (colb + jj < N) crow[colb + jj] = __uint_as_float(r[j4 + jj]);
                        }
                    }
                }
                if ((EPI == EPI_PLAIN || EPI == EPI_PUSH) && ep.mask_out && row_ok) {
                    const int32_t word = (n0 + c0) >> 5;
                    if (word < ep.mask_words) ep.mask_out[row * ep.mask_words + word] = bits;
                }
            }
            tc_fence_before();
            mbar_arrive_warp<CTAS>(&sh->acc_empty[buf], lane);  // the accumulator buffer may be overwritten by the tile after next
            if (EPI == EPI_PUSH && ep.push_max.p) {
                if (push_slot >= 0) ep.push_max.p[(2 * (t % n_tiles_n) + (e >> 2)) * ep.push_max.stride + push_slot] = __float_as_uint(largest);
            }
        }
        if (use_tma_store && lane == 0) tma_store_wait_all();
        if (RING > 0) cp_async_wait<0>();
    }
done:
    tc_fence_before();
    __syncthreads();
    if (CTAS == 2) cluster_sync();   // neither CTA's shared memory or TMEM is in use by the other any more
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tc_dealloc<CTAS>(tmem, 512u);
    }
}

// =====================================================================================
// K-major kernel on half-precision pairs, for contractions of many terms (sat_tc_half)
// =====================================================================================
#define TCH_STAGES_MAX 8
#define TCH_A_BYTES (TC_BM * 128)      /* a k-block of A, raw or split */
struct TchShared {
    uint64_t full[TCH_STAGES_MAX];       // TMA bytes of the stage have landed
    uint64_t conv[TCH_STAGES_MAX];       // the converter threads have split the stage
    uint64_t empty[TCH_STAGES_MAX];      // the MMAs reading the stage have completed
    uint64_t acc_full[2];   // accumulator buffer holds a finished tile
    uint64_t acc_empty[2];  // accumulator buffer has been drained by the epilogue
    uint64_t b_full, b_ready;   // a resident B has landed in this CTA; in all of them
    uint32_t tmem_base;
    int dead;
};

/* 640 threads.  Warps 0-7 convert, in two groups on alternate k-blocks, 8 is the TMA producer, 9 owns the TMEM and issues the MMAs: 72
 * registers each (10 and 11 fill their warpgroup).  12-19 are the epilogue, which holds whole chunks of columns: 128. */
#define TCH_THREADS 640
#define TCH_EPI_WARPS 8

template <int EPI> struct TchCfg { static constexpr int out_bytes = TCH_EPI_WARPS * 4096; };
template <> struct TchCfg<EPI_LSTM> { static constexpr int out_bytes = 0; };
template <> struct TchCfg<EPI_GRU> : TchCfg<EPI_LSTM> {};
template <> struct TchCfg<EPI_PROJ> : TchCfg<EPI_LSTM> {};

// Persistent: each CTA (CTAS = 1) or pair of CTAs (2) walks tiles unit, unit + units, ... of 128 or 256 rows.  A pair's MMA
// (cta_group::2) multiplies the 128 rows of either CTA with all columns of B, of which each CTA holds half.  The shared-memory ring of
// k-block stages and the two TMEM accumulator buffers let the TMA loads, the split, the MMAs and the epilogue of consecutive tiles
// overlap.
//
// A arrives as raw fp32 rows of 128 bytes (32 values).  A converter thread owns a row: it reads 16 of its values, scales and splits them
// (split_f16) and puts the 16 hi and 16 lo halves in their place, so that a k-step's operands are 32 bytes of every row of a K-major
// tile.  B was packed like that once (k_pack_half), so a k-block is one TMA load of each.
//
// The scale is that of the whole row: the kernel is told the largest element of every row (RowMax) by whoever wrote the matrix, since looking for it
// here meant fetching A twice.  The epilogue takes the scales back out (powers of two: exact).
//
// The form with TF32 terms takes in 48 KB of A, B and B's second plane per 32 terms; here it is 32 KB, and 16 where B stays in shared memory.  At
// 164833 x 512, K = 512 (208 us) that is 29 bytes per clock and SM with the tensor pipe active for 75 % of the time; with B resident (256 -> 128,
// 55 us) 13 bytes, tensor pipe 32 %, DRAM 4 TB/s: bound by the chain of a k-block (arrival, split, product) there.
// 169343 rows, TF32 terms -> pairs, us: 256 -> 256 88 -> 70, 256 -> 40 57 -> 42, projections 256 -> 256 89 -> 72; 179250 rows: 512 -> 512
// 320 -> 195, projections 512 -> 256 185 -> 119, 512 -> 512 with the push 378 -> 280.  Errors against 64 bits are half of the TF32 form's
// (embeddings of the first layer of 169343 nodes 1.2e-6 -> 5.7e-7).  (Rows pushed by the two idle warps instead of the epilogue: 120 -> 193.)
// The epilogue is that of k_gemm_tc_k without the gathered residual, on eight warps.
template <int EPI, int CTAS>
__global__ void __launch_bounds__(TCH_THREADS, 1)
k_gemm_tc_h(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapA2, const __grid_constant__ CUtensorMap mapB,
            const __grid_constant__ CUtensorMap mapC, int use_tma_store, uint32_t stages, uint32_t out_tiles, int b_resident,
            int64_t M, int32_t N, int32_t nkb1, int32_t nkb2, int32_t bn, int32_t n_tiles_n, int64_t n_tiles, TcEpilogue ep, int *status)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    constexpr uint32_t a_bytes = TCH_A_BYTES;                // a k-block of A: 128 rows x 128 B, raw or split
    const uint32_t b_bytes = (uint32_t)bn / CTAS * 128;      // of B: [hi | lo], a CTA of a pair holds half of the columns
    const uint32_t stage_bytes = a_bytes + (b_resident ? 0 : b_bytes);
    const uint32_t rank = CTAS == 2 ? blockIdx.x & 1u : 0u;  // in the pair; CTA 0 issues the MMAs of both
    const int64_t unit = blockIdx.x / CTAS, units = gridDim.x / CTAS;
    uint8_t *b_all = smem + (size_t)stages * stage_bytes;       // (b_resident) B's k-blocks of this CTA's columns
    uint8_t *out_stage = b_all + (b_resident ? (nkb1 + nkb2) * b_bytes : 0);   // staging blocks of the epilogue
    constexpr int CONV_WARPS = 8, TMA_WARP = 8, MMA_WARP = 9, EPI_WARP0 = 12, EPI_WARPS = TCH_EPI_WARPS;
    constexpr int CHUNK_STEP = 32 * (EPI_WARPS / 4);  // the EPI_WARPS / 4 warps of a TMEM lane quadrant take 32-column chunks in turn
    TchShared *sh = (TchShared *)(out_stage + TchCfg<EPI>::out_bytes * out_tiles);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t nkb = nkb1 + nkb2;
    const uint32_t acc_cols = 256;  // column stride between the two accumulator buffers

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < stages; ++s) {
            mbar_init(&sh->full[s], 1);
            mbar_init(&sh->conv[s], CTAS * (CONV_WARPS / 2));
            mbar_init(&sh->empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh->acc_full[i], 1);
            mbar_init(&sh->acc_empty[i], CTAS * EPI_WARPS);
        }
        mbar_init(&sh->b_full, 1);
        mbar_init(&sh->b_ready, CTAS);
        sh->dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == MMA_WARP) {
        tc_alloc<CTAS>(&sh->tmem_base, 512u);
    }
    tc_fence_before();
    __syncthreads();
    if (CTAS == 2) cluster_sync();   // the other CTA's barriers are initialised and its TMEM is allocated
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    volatile int *dead = &sh->dead;
    sat_grid_wait();   // everything above is set-up of this block; no global memory has been touched
    // exponent of the scale of a row of A (past the matrix: any)
    auto row_scale = [&](int64_t row) {
        uint32_t m = ep.row_least;
        for (int32_t p = 0; p < ep.row_parts; ++p) m = max(m, __ldg(ep.row_max + p * ep.row_stride + (row < M ? row : M - 1)));
        return f16_scale_exponent(m >> 23);
    };
    auto tile_row0 = [&](int64_t t) { return (tck_row_tile(ep, t, n_tiles_n) * CTAS + rank) * TC_BM; };   // first row of this CTA

    if (warp < EPI_WARP0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");   // 384 x 72 + 256 x 128 of the 640 x 96 registers at launch
    if (warp == TMA_WARP) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            uint32_t s = 0, ph = 0;
            if (b_resident) {   // (every tile of the CTA has the same columns)
                mbar_expect_tx(&sh->b_full, (uint32_t)nkb * b_bytes);
                for (int32_t kb = 0; kb < nkb; ++kb)
                    tma_load_2d(b_all + kb * b_bytes, &mapB, &sh->b_full, kb * 2 * TCH_BK, (int32_t)(unit % n_tiles_n) * bn + (int32_t)rank * (bn / CTAS));
            }
            for (int64_t t = unit; t < n_tiles; t += units) {
                const int32_t m0 = (int32_t)tile_row0(t);
                const int32_t n0 = (int32_t)(t % n_tiles_n) * bn + (int32_t)rank * (bn / CTAS);
                for (int32_t kb = 0; kb < nkb; ++kb) {
                    if (!mbar_wait(&sh->empty[s], ph ^ 1u, dead, status)) goto done;
                    uint8_t *st = smem + (size_t)s * stage_bytes;
                    mbar_expect_tx(&sh->full[s], stage_bytes);
                    if (kb < nkb1) tma_load_2d(st, &mapA, &sh->full[s], kb * TCH_BK, m0);
                    else tma_load_2d(st, &mapA2, &sh->full[s], (kb - nkb1) * TCH_BK, m0);
                    if (!b_resident) tma_load_2d(st + a_bytes, &mapB, &sh->full[s], kb * 2 * TCH_BK, n0);
                    if (++s == stages) s = 0, ph ^= 1u;
                }
            }
            // the pair's MMAs have signalled every stage: nothing arrives here any more once both CTAs may exit
            for (uint32_t i = 0; CTAS == 2 && i < stages; ++i) {
                if (!mbar_wait(&sh->empty[s], ph ^ 1u, dead, status)) goto done;
                if (++s == stages) s = 0, ph ^= 1u;
            }
        }
    } else if (warp == MMA_WARP && rank == 0) {
        // ---------------- MMA issuer ----------------
        // The whole warp walks the k-blocks and an elected lane issues: the operands of the instructions are then known to be uniform.
        // (One lane doing all of it took 0.4 us per k-block, which bound the narrow tiles: 169343 x 40, K = 256: 70 -> 62 us.)
        const uint32_t idesc = make_idesc_f16(TC_BM * CTAS, bn);
        const uint64_t desc0 = make_desc(smem_u32(smem), 16, 1024, 2);
        uint32_t s = 0, ph = 0, lt = 0;
        if (b_resident && !mbar_wait_all(&sh->b_ready, 0, dead, status)) goto done;
        for (int64_t t = unit; t < n_tiles; t += units, ++lt) {
            const uint32_t buf = lt & 1u;
            if (!mbar_wait_all(&sh->acc_empty[buf], ((lt >> 1) & 1u) ^ 1u, dead, status)) goto done;
            tc_fence_after();
            const uint32_t acc = tmem + buf * acc_cols;
            for (int32_t kb = 0; kb < nkb; ++kb) {
                // the converters arrive on conv[s] only after they have seen full[s] (the TMA bytes) themselves
                if (!mbar_wait_all(&sh->conv[s], ph, dead, status)) goto done;
                tc_fence_after();
                // K-major, 128-byte swizzle: rows 128 B apart, 8-row groups 1024 B; a k-step (16 terms) takes 64 B of the row, its hi halves
                // and then its lo halves.  Only the 14-bit start-address field (bytes >> 4) differs between the descriptors of a stage.
                const uint64_t a_hi0 = desc0 + (uint64_t)((s * stage_bytes) >> 4);
                const uint64_t b_hi0 = b_resident ? desc0 + (uint64_t)((stages * stage_bytes + (uint32_t)kb * b_bytes) >> 4) : a_hi0 + (a_bytes >> 4);
                const int32_t left = kb < nkb1 ? ep.k1 - kb * TCH_BK : ep.k2 - (kb - nkb1) * TCH_BK;   // terms from here on (the rest of the block is zero)
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks) {
                        if (ks == 1 && left <= 16) break;
                        const uint64_t a_hi = a_hi0 + (uint64_t)(ks * 4), a_lo = a_hi + 2;
                        const uint64_t b_hi = b_hi0 + (uint64_t)(ks * 4), b_lo = b_hi + 2;
                        tc_mma_f16<1, CTAS>(acc, a_hi, b_hi, idesc, (kb > 0 || ks > 0) ? 1u : 0u);
                        tc_mma_f16<2, CTAS>(acc, a_hi, b_lo, idesc, 1u);
                        tc_mma_f16<0, CTAS>(acc, a_lo, b_hi, idesc, 1u);
                    }
                    tc_commit<CTAS>(&sh->empty[s]);  // the stage is free once these MMAs have read it
                }
                if (++s == stages) s = 0, ph ^= 1u;
            }
            if (elect_one()) tc_commit<CTAS>(&sh->acc_full[buf]);
        }
    } else if (warp < CONV_WARPS) {
        // ---------------- converters: the two-term split of the A tile of every k-block ----------------
        const uint32_t grp = warp / (CONV_WARPS / 2);
        const int r = threadIdx.x & (TC_BM - 1), sw = r & 7;   // this thread's row; 16-byte piece c of it sits at c ^ sw
        if (b_resident && warp == 0) {
            if (!mbar_wait_all(&sh->b_full, 0, dead, status)) goto done;
            mbar_arrive_lane0<CTAS>(&sh->b_ready, lane);
        }
        uint32_t s = grp, ph = 0, odd = 0;    // next own stage; parity of the k-blocks before this tile
        uint32_t next = unit < n_tiles ? row_scale(tile_row0(unit) + r) : 0;
        for (int64_t t = unit; t < n_tiles; t += units) {
            const float scale = __uint_as_float(next << 23);
            if (t + units < n_tiles) next = row_scale(tile_row0(t + units) + r);   // a tile early
            for (int32_t kb = (int32_t)(grp ^ odd); kb < nkb; kb += 2) {
                if (!mbar_wait_all(&sh->full[s], ph, dead, status)) goto done;
                uint8_t *const row = smem + s * stage_bytes + r * 128;
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {   // 16 values, whose 64 bytes the halves take
                    float4 x[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) x[c] = *reinterpret_cast<const float4 *>(row + (((4 * ks + c) ^ sw) << 4));
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const float4 u = x[2 * c], v = x[2 * c + 1];
                        uint4 hi, lo;
                        split_f16(u.x * scale, u.y * scale, hi.x, lo.x);
                        split_f16(u.z * scale, u.w * scale, hi.y, lo.y);
                        split_f16(v.x * scale, v.y * scale, hi.z, lo.z);
                        split_f16(v.z * scale, v.w * scale, hi.w, lo.w);
                        *reinterpret_cast<uint4 *>(row + (((4 * ks + c) ^ sw) << 4)) = hi;
                        *reinterpret_cast<uint4 *>(row + (((4 * ks + c + 2) ^ sw) << 4)) = lo;
                    }
                }
                fence_async_smem();
                mbar_arrive_lane0<CTAS>(&sh->conv[s], lane);
                s += 2;
                if (s >= stages) s -= stages, ph ^= 1u;
            }
            odd ^= (uint32_t)nkb & 1u;
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 128;");
        // ---------------- epilogue ----------------
        // warp w reads TMEM lanes 32 (w % 4) .. +31 = rows of the tile, one row per thread; the warps of a lane quadrant
        // take alternate 32-column chunks.
        constexpr bool LSTM = EPI == EPI_LSTM || EPI == EPI_GRU;   // a recurrent cell
        const int e = warp - EPI_WARP0;
        const int q = warp & 3;
        const int c_first = 32 * (e >> 2);
        uint32_t staged = 0;   // blocks staged so far
        const bool vec = ((ep.ldc & 3) == 0) && ((((uintptr_t)ep.C) & 15u) == 0);
        const bool lstm_full = LSTM && (ep.lstm_h & 3) == 0;
        const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);

        uint32_t lt = 0;
        for (int64_t t = unit; t < n_tiles; t += units, ++lt) {
            const int64_t m0 = tile_row0(t);
            const int32_t n0 = (int32_t)(t % n_tiles_n) * bn;
            const uint32_t buf = lt & 1u;
            const int64_t row = m0 + q * 32 + lane;
            const bool row_ok = row < M;
            float *crow = ep.C + row * ep.ldc;
            float *prow = nullptr;   // (EPI_PUSH) this row's home in the cache ring, if it has one
            const int32_t push_slot = EPI == EPI_PUSH && row_ok ? __ldg(ep.push_slot + row) : -1;
            if (EPI == EPI_PUSH && !use_tma_store && push_slot >= 0) prow = ep.push_dst + (int64_t)push_slot * ep.ld_push;
            float4 cside[2];
            float largest = 0.f;   // (EPI_PUSH) of this thread's chunks
            // previous cell state (GRU: hidden state) of the next chunk, fetched one chunk ahead (two 128-bit loads per thread)
            auto load_cell = [&](int c0) {
                if (LSTM) {
                    cside[0] = cside[1] = zero4;
                    const int32_t j0 = (n0 + c0) >> 2;
                    if (row_ok && lstm_full && !ep.lstm_first && j0 + 7 < ep.lstm_h) {
                        const float *cp = EPI == EPI_GRU ? crow + j0 : ep.lstm_c + sat_cell_offset(row, j0, ep.lstm_h);
                        cside[0] = *reinterpret_cast<const float4 *>(cp);
                        cside[1] = *reinterpret_cast<const float4 *>(cp + 4);
                    }
                }
            };
            if (c_first < bn) load_cell(c_first);
            const float unscale = __uint_as_float((254u + SCALE_SHIFT - row_scale(row)) << 23);
            if (!mbar_wait_warp(&sh->acc_full[buf], (lt >> 1) & 1u, dead, status, lane)) goto done;
            tc_fence_after();
            for (int c0 = c_first; c0 < bn; c0 += CHUNK_STEP) {
                // inverse scales of the chunk's columns: ahead of the accumulators for the cells (84671 rows, GRU step of 320 terms 67.0 -> 66.2 us), with them
                // for the others (169343 rows, masked 256 -> 256 75.0 -> 73.5)
                auto load_unscale = [&](int u) { return __ldg(reinterpret_cast<const float4 *>(ep.unscale + n0 + c0) + u); };
                float4 us8[8];
#pragma unroll
                for (int u = 0; LSTM && u < 8; ++u) us8[u] = load_unscale(u);
                uint32_t r[32];
                tc_ld32(tmem + buf * acc_cols + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, r);
                // takes the scales out and adds the bias to four columns
                auto finish = [&](uint32_t *x, int u) {
                    const float4 us = LSTM ? us8[u] : load_unscale(u);
                    const float4 b4 = ep.bias ? __ldg(reinterpret_cast<const float4 *>(ep.bias + n0 + c0) + u) : zero4;
                    const float4 y = scaled_add(x, us, b4, make_float2(unscale, unscale));
                    x[0] = __float_as_uint(y.x);
                    x[1] = __float_as_uint(y.y);
                    x[2] = __float_as_uint(y.z);
                    x[3] = __float_as_uint(y.w);
                };
                if (LSTM) {
                    // packed columns 4 j .. 4 j + 3 are the (i, f, g, o) pre-activations of hidden unit j
                    if (row_ok) {
                        const int32_t j0 = (n0 + c0) >> 2;
                        const bool full = lstm_full && j0 + 7 < ep.lstm_h;
#pragma unroll
                        for (int u = 0; u < 8; ++u) finish(r + 4 * u, u);
                        float cprev[8];
                        cprev[0] = cside[0].x; cprev[1] = cside[0].y; cprev[2] = cside[0].z; cprev[3] = cside[0].w;
                        cprev[4] = cside[1].x; cprev[5] = cside[1].y; cprev[6] = cside[1].z; cprev[7] = cside[1].w;
                        if (!ep.lstm_first && !full) {
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                if (j0 + u < ep.lstm_h) cprev[u] = EPI == EPI_GRU ? crow[j0 + u] : ep.lstm_c[sat_cell_offset(row, j0 + u, ep.lstm_h)];
                        }
                        if (c0 + CHUNK_STEP < bn) load_cell(c0 + CHUNK_STEP);
                        float sv[8], cv[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            if (EPI == EPI_GRU) {   // (r, z, n from the input, n from the state)
                                const float gr = 1.f / (1.f + expf(-__uint_as_float(r[4 * u])));
                                const float gz = 1.f / (1.f + expf(-__uint_as_float(r[4 * u + 1])));
                                const float gn = tanhf(__uint_as_float(r[4 * u + 2]) + gr * __uint_as_float(r[4 * u + 3]));
                                sv[u] = (1.f - gz) * gn + gz * cprev[u];
                                continue;
                            }
                            const float gi = sigmoid_fast(__uint_as_float(r[4 * u]));
                            const float gf = sigmoid_fast(__uint_as_float(r[4 * u + 1]));
                            const float gg = tanh_fast(__uint_as_float(r[4 * u + 2]));
                            const float go = sigmoid_fast(__uint_as_float(r[4 * u + 3]));
                            cv[u] = gf * cprev[u] + gi * gg;
                            sv[u] = go * tanh_fast(cv[u]);
                        }
                        if (full) {
                            float4 *sd = reinterpret_cast<float4 *>(ep.C + row * ep.ldc + j0);
                            if (EPI != EPI_GRU) {
                                float4 *cd = reinterpret_cast<float4 *>(ep.lstm_c + sat_cell_offset(row, j0, ep.lstm_h));
                                cd[0] = make_float4(cv[0], cv[1], cv[2], cv[3]);
                                cd[1] = make_float4(cv[4], cv[5], cv[6], cv[7]);
                            }
                            sd[0] = make_float4(sv[0], sv[1], sv[2], sv[3]);
                            sd[1] = make_float4(sv[4], sv[5], sv[6], sv[7]);
                        } else {
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                if (j0 + u < ep.lstm_h) {
                                    if (EPI != EPI_GRU) ep.lstm_c[sat_cell_offset(row, j0 + u, ep.lstm_h)] = cv[u];
                                    ep.C[row * ep.ldc + j0 + u] = sv[u];
                                }
                        }
                    }
                    continue;
                }
                uint32_t bits = 0;
                if (row_ok) {
                    // bias is padded with zeros to the tile width and the accumulators of padded columns are exactly zero,
                    // so no column predicate is needed (the stores clip)
#pragma unroll
                    for (int j = 0; j < 8; ++j) finish(r + 4 * j, j);
                    if ((EPI == EPI_PLAIN || EPI == EPI_PUSH) && ep.mask_out) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) bits |= (__uint_as_float(r[j]) > 0.f ? 1u : 0u) << j;
                    }
                    if (ep.relu) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(fmaxf(__uint_as_float(r[j]), 0.f));
                    }
                    if (EPI == EPI_PUSH && ep.push_max.p) {
#pragma unroll
                        for (int j = 0; j < 32; j += 2) largest = fmaxf(largest, fmaxf(fabsf(__uint_as_float(r[j])), fabsf(__uint_as_float(r[j + 1]))));
                    }
                    if (EPI == EPI_PLAIN && ep.mask_in) {
                        const int32_t word = (n0 + c0) >> 5;
                        const uint32_t keep = word < ep.mask_in_words ? __ldg(ep.mask_in + row * ep.mask_in_words + word) : 0u;
#pragma unroll
                        for (int j = 0; j < 32; ++j) r[j] = keep >> j & 1u ? r[j] : 0u;
                    }
                }
                if (EPI == EPI_PROJ) {   // a warp's store of a unit is 512 contiguous bytes
                    if (row_ok) {
                        const int32_t j0 = (n0 + c0) >> 2;
                        float4 *dst = reinterpret_cast<float4 *>(ep.C) + ((row >> 7) * ep.proj_h + j0) * 128 + (row & 127);
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (j0 + u < ep.proj_h)
                                dst[u * 128] = make_float4(__uint_as_float(r[4 * u]), __uint_as_float(r[4 * u + 1]), __uint_as_float(r[4 * u + 2]),
                                                           __uint_as_float(r[4 * u + 3]));
                    }
                    continue;
                }
                if (EPI == EPI_PUSH && prow) {   // one full 128-byte line per thread and chunk
#pragma unroll
                    for (int j4 = 0; j4 < 32; j4 += 4) {
                        const int32_t colb = n0 + c0 + j4;
                        if (colb + 3 < N) {
                            *reinterpret_cast<uint4 *>(prow + colb) = make_uint4(r[j4], r[j4 + 1], r[j4 + 2], r[j4 + 3]);
                        } else {
#pragma unroll
                            for (int jj = 0; jj < 4; ++jj)
                                if (colb + jj < N) prow[colb + jj] = __uint_as_float(r[j4 + jj]);
                        }
                    }
                }
                if (use_tma_store) {
                    // stage the 32 x 32 block (128-byte swizzle: 16-byte chunk j of row r sits at chunk j ^ (r & 7)) and
                    // let the TMA write it as whole 128-byte row segments; rows / columns past the matrix are clipped
                    // the block before, or the one before that, has left its staging tile
                    if (lane == 0) {
                        if (out_tiles == 2) tma_store_wait_read<1>();
                        else tma_store_wait_read<0>();
                    }
                    uint8_t *const obuf = out_stage + (e * out_tiles + (staged++ & (out_tiles - 1))) * 4096;
                    __syncwarp();
                    uint8_t *dst = obuf + lane * 128;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        *reinterpret_cast<uint4 *>(dst + ((j ^ (lane & 7)) << 4)) = make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) tma_store_2d(&mapC, obuf, n0 + c0, (int32_t)(m0 + q * 32));
                    if (EPI == EPI_PUSH) {
                        // the boundary rows also go to the cache ring, read back from the staged block: every instruction
                        // writes whole 128-byte row segments (the per-thread form touches 32 different lines per instruction)
                        // (lane L writes 16-byte piece L & 7 of rows (L >> 3) + 4 i)
                        const int piece = lane & 7;
                        const int32_t colb = n0 + c0 + 4 * piece;
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int rr = (lane >> 3) + 4 * i;
                            const int32_t slot = __shfl_sync(0xffffffffu, push_slot, rr);
                            if (slot < 0 || colb >= N) continue;
                            float *pr = ep.push_dst + (int64_t)slot * ep.ld_push;
                            const uint4 x = *reinterpret_cast<const uint4 *>(obuf + rr * 128 + ((piece ^ (rr & 7)) << 4));
                            if (colb + 3 < N) {
                                *reinterpret_cast<uint4 *>(pr + colb) = x;
                            } else {
                                pr[colb] = __uint_as_float(x.x);
                                if (colb + 1 < N) pr[colb + 1] = __uint_as_float(x.y);
                                if (colb + 2 < N) pr[colb + 2] = __uint_as_float(x.z);
                            }
                        }
                    }
                } else if (row_ok) {
#pragma unroll
                    for (int j4 = 0; j4 < 32; j4 += 4) {
                        const int32_t colb = n0 + c0 + j4;
                        if (vec && colb + 3 < N) {
                            *reinterpret_cast<uint4 *>(crow + colb) = make_uint4(r[j4], r[j4 + 1], r[j4 + 2], r[j4 + 3]);
                        } else {
#pragma unroll
                            for (int jj = 0; jj < 4; ++jj)
                                if (colb + jj < N) crow[colb + jj] = __uint_as_float(r[j4 + jj]);
                        }
                    }
                }
                if ((EPI == EPI_PLAIN || EPI == EPI_PUSH) && ep.mask_out && row_ok) {
                    const int32_t word = (n0 + c0) >> 5;
                    if (word < ep.mask_words) ep.mask_out[row * ep.mask_words + word] = bits;
                }
            }
            tc_fence_before();
            mbar_arrive_lane0<CTAS>(&sh->acc_empty[buf], lane);  // the accumulator buffer may be overwritten by the tile after next
            if (EPI == EPI_PUSH && ep.push_max.p) {
                if (push_slot >= 0) ep.push_max.p[(2 * (t % n_tiles_n) + (e >> 2)) * ep.push_max.stride + push_slot] = __float_as_uint(largest);
            }
        }
        if (use_tma_store && lane == 0) tma_store_wait_all();
    }
done:
    tc_fence_before();
    __syncthreads();
    if (CTAS == 2) cluster_sync();   // neither CTA's shared memory or TMEM is in use by the other any more
    if (warp == MMA_WARP) {
        __syncwarp();
        tc_fence_after();
        tc_dealloc<CTAS>(tmem, 512u);
    }
}

// =====================================================================================
// LSTM steps over cached input projections, all in one kernel: z = proj_t + s Uh, c = f c + i g, s = o tanh(c) for consecutive steps t.
//
// One launch per step moved the state s and c through memory every time and fetched Uh for every tile: 345 MB a step at 169343 rows and
// h = 64, half of it the projection (83 us a step, and 54 for the first one).  Here a row tile stays on the SM for all steps: s as the
// A operand in shared memory, c in registers, Uh resident; a step reads its projection and nothing else.
//
// A CTA works on two slots of 128 rows so that one slot's product runs under the other's cell arithmetic.  The operands are half-precision
// pairs (split_f16; the state lies in [-1, 1], its scale is 2^14), rows of 128 bytes with 16 hi and 16 lo halves per k-step: 32 KB a slot
// and 64 KB for Uh at h = 64, half of what TF32 terms take, which leaves 96 KB for the projections.  Those are stored [row tile of 128][unit][row]
// float4 (sat_proj_floats); a thread copies its own row's 64 bytes of a quad of units by cp.async, SEQ_RING of its quads ahead, so
// that nobody else has to be waited for.  Eight warps per slot, two per lane quadrant with alternate quads, one row per thread; accumulator
// columns are fetched a quad ahead.  The slot's first warp also issues its products.
//
// 164833 rows, h = 64, four steps (675 MB of projections): 198 -> 158 us; 612257 rows 660 -> 504; 179250 rows and eight steps 393 -> 310.  Before, a
// CTA pair held TF32 terms and the projections came through registers, two quads ahead; that form was bound by its latencies with every
// unit below 45 %.  What did it: the copies' depth and their .cg (.ca: 184 us) and the accumulator columns a quad ahead.  (Bulk copies
// by a warp of their own per slot, which leaves 96 registers: 192 us.)  The errors are what they were (relative 1.6e-6 of the
// state at K = 256).  The inverse scales of a quad's sixteen columns come out of shared memory too, next to projections and state: 164833 rows 161 -> 180 us with
// one for every column, so eight neighbours (a pair of units) share theirs where they are of a size (k_pack_half), and only a matrix where they are not
// takes that form, which costs the other 6 us by its call.
// =====================================================================================
#define SEQ_THREADS 512   /* 128 registers a thread */
#define SEQ_RING 3        /* quads of projections in flight per thread */
struct SeqSteps {
    const float *proj[SAT_SEQ_MAX];
};
struct SeqShared {
    float4 unscale[64];                              // inverse scales of a unit's gate columns, the state's taken along
    float2 pair_unscale[16];                         // of the pairs of units of a quad, whose columns share them unless
    int own_scales;                                  // ... somewhere the columns of a pair have scales of their own
    uint64_t b_full;                                 // Uh has landed
    uint64_t a_ready[2], acc_full[2];                // per slot: the state is in place; the product is done
    uint32_t tmem_base;
    int dead;
};

// 16 accumulator columns, to be waited for by tc_wait16 before their use
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tc_wait16(uint32_t *r)   // (the registers are operands so that nothing reads them earlier)
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]),
                   "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])::"memory");
}
// One LSTM cell: gates (i, f, g, o) and the cell state; returns the hidden state.  The quotients share reciprocals, since the transcendental unit
// (16 lanes per clock, two operations per sigmoid or tanh by themselves) would take as long as the memory:
//   i g = (e^{2 zg} - 1) / ((1 + e^{-zi}) (1 + e^{2 zg})),  o tanh(c) = (e^{2c} - 1) / ((1 + e^{-zo}) (1 + e^{2c})):
// eight operations instead of ten.  Exponents are capped at 2^60, where both quotients have reached their limits in fp32, so that the products
// do not overflow.
__device__ __forceinline__ float lstm_cell(const float4 &z, float &c)
{
    auto capped = [](float x) {   // 2^min(x, 60), NaN for NaN
        asm("min.NaN.f32 %0, %0, 0f42700000;" : "+f"(x));
        return ex2_fast(x);
    };
    const float L = 1.4426950408889634f;
    const float ei = capped(-L * z.x), ef = ex2_fast(-L * z.y), eg = capped(2.f * L * z.z), eo = capped(-L * z.w);
    c = fmaf(rcp_fast(1.f + ef), c, (eg - 1.f) * rcp_fast((1.f + ei) * (1.f + eg)));
    const float ec = capped(2.f * L * c);
    return (ec - 1.f) * rcp_fast((1.f + eo) * (1.f + ec));
}

// The row tiles of a slot.  SHARED: the columns of a pair of units have one scale.
template <bool SHARED>
__device__ __forceinline__ void
lstm_tiles(uint8_t *smem, uint8_t *Bs, uint8_t *Ps, SeqShared *sh, uint32_t tmem, const SeqSteps &steps, int32_t n_steps, int first, int64_t rows, int32_t h,
           int32_t bn, int32_t nkb, int32_t mine, float *S, float *cell, int write_cell, int *status)
{
    constexpr uint32_t a_block = TC_BM * 128;
    const uint32_t b_block = (uint32_t)bn * 128, slot_bytes = (uint32_t)nkb * a_block;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t nq = h >> 2;                       // quads of four units
    volatile int *dead = &sh->dead;
    const int slot = warp >> 3, q = warp & 3, half = (warp >> 2) & 1;
    const bool issuer = (warp & 7) == 0;   // of its slot's products
    const uint32_t idesc = make_idesc_f16(TC_BM, bn), acc = tmem + (uint32_t)slot * 256u;
    const uint64_t a0 = make_desc(smem_u32(smem) + (uint32_t)slot * slot_bytes, 16, 1024, 2), b0 = make_desc(smem_u32(Bs), 16, 1024, 2);
    const int32_t nks = (h + 15) / 16;               // k-steps of 16
    const int r_in = q * 32 + lane;                  // this thread's row of the tile
    uint8_t *A = smem + (uint32_t)slot * slot_bytes + r_in * 128;
    const uint32_t swz = (uint32_t)r_in & 7u;        // 16-byte piece c of row r sits at c ^ (r & 7)
    uint8_t *const ring = Ps + threadIdx.x * 16;
    const uint32_t mine_acc = acc + ((uint32_t)(q * 32) << 16);
    auto put = [&](int qd, const float4 &v) {   // a quad is half a piece
        uint2 hi, lo;
        split_f16(v.x * 0x1p14f, v.y * 0x1p14f, hi.x, lo.x);
        split_f16(v.z * 0x1p14f, v.w * 0x1p14f, hi.y, lo.y);
        uint8_t *d = A + ((uint32_t)qd >> 3) * a_block + (((uint32_t)qd & 1u) << 3);
        const uint32_t piece = ((uint32_t)qd & 4u) | (((uint32_t)qd & 3u) >> 1);
        *reinterpret_cast<uint2 *>(d + ((piece ^ swz) << 4)) = hi;
        *reinterpret_cast<uint2 *>(d + (((piece + 2) ^ swz) << 4)) = lo;
    };
    // this thread's quads in the order in which they are taken: (tile, step, quad); the copies run SEQ_RING of them ahead
    const int32_t my_quads = (nq - half + 1) / 2;
    int32_t pf_k = slot, pf_t = 0, pf_i = 0;
    uint32_t pf_at = 0, at = 0;
    auto copy_next = [&]() {   // a group a call, empty at the end
        if (pf_k < mine && my_quads > 0) {
            const float4 *src = reinterpret_cast<const float4 *>(steps.proj[pf_t]) +
                                ((blockIdx.x + (int64_t)pf_k * gridDim.x) * h + 4 * (half + 2 * pf_i)) * TC_BM + r_in;
#pragma unroll
            for (int u = 0; u < 4; ++u) cp_async16(ring + (pf_at * 4 + u) * (SEQ_THREADS * 16), src + u * TC_BM, true);
            if (++pf_i == my_quads) {
                pf_i = 0;
                if (++pf_t == n_steps) pf_t = 0, pf_k += 2;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        pf_at = pf_at + 1 == SEQ_RING ? 0 : pf_at + 1;
    };
#pragma unroll
    for (int i = 0; i < SEQ_RING; ++i) copy_next();
    if (issuer && mine > slot && !mbar_wait_all(&sh->b_full, 0, dead, status)) return;
    uint32_t ph = 0;
    for (int32_t k = slot; k < mine; k += 2) {
        const int64_t row = (blockIdx.x + (int64_t)k * gridDim.x) * TC_BM + r_in;
        const bool row_ok = row < rows;
        float4 c[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int32_t qd = half + 2 * i;
            c[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (!first && qd < nq) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row_ok) {
                    v = *reinterpret_cast<const float4 *>(S + row * h + 4 * qd);
                    c[i] = *reinterpret_cast<const float4 *>(cell + sat_cell_offset(row, 4 * qd, h));
                }
                put(qd, v);
            }
        }
        for (int32_t t = 0; t < n_steps; ++t) {
            const bool product = t > 0 || !first, last = t + 1 == n_steps;
            if (product) {
                fence_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh->a_ready[slot]);
                if (issuer) {
                    if (!mbar_wait_all(&sh->a_ready[slot], ph, dead, status)) return;
                    tc_fence_after();
                    if (elect_one()) {
                        for (int32_t ks = 0; ks < nks; ++ks) {
                            const uint64_t a_hi = a0 + (uint64_t)((ks >> 1) * (a_block >> 4) + (ks & 1) * 4), a_lo = a_hi + 2;
                            const uint64_t b_hi = b0 + (uint64_t)((ks >> 1) * (b_block >> 4) + (ks & 1) * 4), b_lo = b_hi + 2;
                            tc_mma_f16<1, 1>(acc, a_hi, b_hi, idesc, ks > 0 ? 1u : 0u);
                            tc_mma_f16<2, 1>(acc, a_hi, b_lo, idesc, 1u);
                            tc_mma_f16<0, 1>(acc, a_lo, b_hi, idesc, 1u);
                        }
                        tc_commit<1>(&sh->acc_full[slot]);
                    }
                    __syncwarp();
                }
                if (!mbar_wait_all(&sh->acc_full[slot], ph, dead, status)) return;
                ph ^= 1u;
                tc_fence_after();
            }
            uint32_t r[2][16];   // accumulator columns of this quad and the next
            if (product && half < nq) tc_ld16(mine_acc + 16u * (uint32_t)half, r[0]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int32_t qd = half + 2 * i;
                if (qd < nq) {
                    asm volatile("cp.async.wait_group %0;" ::"n"(SEQ_RING - 1) : "memory");   // this thread's own copies
                    float4 z[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) z[u] = *reinterpret_cast<const float4 *>(ring + (at * 4 + u) * (SEQ_THREADS * 16));
                    at = at + 1 == SEQ_RING ? 0 : at + 1;
                    if (product) {
                        uint32_t(&a)[16] = r[i & 1];
                        const float2 us2 = SHARED ? sh->pair_unscale[qd] : make_float2(0.f, 0.f);
                        tc_wait16(a);
                        if (i < 7 && qd + 2 < nq) tc_ld16(mine_acc + 16u * (uint32_t)(qd + 2), r[(i + 1) & 1]);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            float4 us = make_float4(u < 2 ? us2.x : us2.y, 0.f, 0.f, 0.f);
                            if (SHARED) us.y = us.z = us.w = us.x;
                            else us = sh->unscale[4 * qd + u];
                            z[u].x = fmaf(__uint_as_float(a[4 * u]), us.x, z[u].x);
                            z[u].y = fmaf(__uint_as_float(a[4 * u + 1]), us.y, z[u].y);
                            z[u].z = fmaf(__uint_as_float(a[4 * u + 2]), us.z, z[u].z);
                            z[u].w = fmaf(__uint_as_float(a[4 * u + 3]), us.w, z[u].w);
                        }
                    }
                    copy_next();   // (into the place just read)
                    float4 sv;
                    float *cf = reinterpret_cast<float *>(&c[i]), *sf = reinterpret_cast<float *>(&sv);
#pragma unroll
                    for (int u = 0; u < 4; ++u) sf[u] = lstm_cell(z[u], cf[u]);   // unit 4 qd + u
                    if (!last) {
                        put(qd, sv);
                    } else if (row_ok) {
                        *reinterpret_cast<float4 *>(S + row * h + 4 * qd) = sv;
                        if (write_cell) *reinterpret_cast<float4 *>(cell + sat_cell_offset(row, 4 * qd, h)) = c[i];
                    }
                }
            }
        }
    }
}
// (with registers of its own: in line with the other form it made that one spill, 161 -> 178 us)
__device__ __noinline__ void
lstm_tiles_own_scales(uint8_t *smem, uint8_t *Bs, uint8_t *Ps, SeqShared *sh, uint32_t tmem, const SeqSteps &steps, int32_t n_steps, int first, int64_t rows, int32_t h,
                      int32_t bn, int32_t nkb, int32_t mine, float *S, float *cell, int write_cell, int *status)
{
    lstm_tiles<false>(smem, Bs, Ps, sh, tmem, steps, n_steps, first, rows, h, bn, nkb, mine, S, cell, write_cell, status);
}

__global__ void __launch_bounds__(SEQ_THREADS, 1)
k_lstm_seq(const __grid_constant__ CUtensorMap mapB, const float *__restrict__ unscale, const __grid_constant__ SeqSteps steps, int32_t n_steps, int first,
           int64_t rows, int32_t h, int32_t bn, int32_t nkb, float *S, float *cell, int write_cell,
           int *status)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    constexpr uint32_t a_block = TC_BM * 128;                     // a k-block: rows of two k-steps of 16 hi and 16 lo halves, 128-byte swizzle
    const uint32_t b_block = (uint32_t)bn * 128, slot_bytes = (uint32_t)nkb * a_block;
    uint8_t *Bs = smem + 2 * slot_bytes;
    uint8_t *Ps = Bs + (uint32_t)nkb * b_block;                   // projections: [SEQ_RING][unit of the quad][thread] float4
    SeqShared *sh = (SeqShared *)(Ps + SEQ_RING * 4 * SEQ_THREADS * 16);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n_rt = (rows + TC_BM - 1) / TC_BM;
    const int32_t mine = blockIdx.x < n_rt ? (int32_t)((n_rt - 1 - blockIdx.x) / gridDim.x + 1) : 0;   // row tiles of the CTA, alternately in slot 0 and 1

    for (uint32_t o = threadIdx.x * 16; o < 2 * slot_bytes; o += SEQ_THREADS * 16) *reinterpret_cast<float4 *>(smem + o) = make_float4(0.f, 0.f, 0.f, 0.f);
    fence_async_smem();   // (the columns from h on stay zero)
    if (threadIdx.x == 0) {
        mbar_init(&sh->b_full, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh->a_ready[i], 8);
            mbar_init(&sh->acc_full[i], 1);
        }
        sh->dead = sh->own_scales = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tc_alloc<1>(&sh->tmem_base, 512u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    volatile int *dead = &sh->dead;
    sat_grid_wait();
    if ((int)threadIdx.x < bn) {
        const float us = __ldg(unscale + threadIdx.x);   // (with the inverse of the state's scale, 2^-SCALE_SHIFT, in it)
        reinterpret_cast<float *>(sh->unscale)[threadIdx.x] = us;
        if (us != __shfl_sync(0xffffffffu, us, lane & 24)) sh->own_scales = 1;   // (whole warps: bn is a multiple of 32)
        if ((lane & 7) == 0) reinterpret_cast<float *>(sh->pair_unscale)[threadIdx.x >> 3] = us;
    }
    __syncthreads();

    if (warp == 0 && mine > 0) {
        if (lane == 0) {
            mbar_expect_tx(&sh->b_full, (uint32_t)nkb * b_block);
            for (int32_t kb = 0; kb < nkb; ++kb) tma_load_2d(Bs + (uint32_t)kb * b_block, &mapB, &sh->b_full, kb * 2 * TCH_BK, 0);
        }
        if (!mbar_wait_all(&sh->b_full, 0, dead, status)) goto done;
    }
    if (sh->own_scales) lstm_tiles_own_scales(smem, Bs, Ps, sh, tmem, steps, n_steps, first, rows, h, bn, nkb, mine, S, cell, write_cell, status);
    else lstm_tiles<true>(smem, Bs, Ps, sh, tmem, steps, n_steps, first, rows, h, bn, nkb, mine, S, cell, write_cell, status);
done:
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        tc_dealloc<1>(tmem, 512u);
    }
}

// =====================================================================================
// MN-major kernel (weight gradient): block (x, y, z) = tile (x, y) of A^T B over rows [z' * rps, (z' + 1) * rps) of segment z / seg_splits,
// z' = z % seg_splits (several products of the same shape summed into one result: the steps of the predictor); the blocks with x == 0
// also leave the column sums of their rows of B (the bias gradient) in part_cs [z x N] when it is given: the converters hold every
// value of B in registers anyway, which saves a pass over it (34 us for 169 k x 256).
//
// Tile: up to 256 columns of A (two accumulators of 128 TMEM lanes) by up to 256 of B, one CTA per SM (two where m <= 128).  Both operands are activations
// and have to be split in the kernel; a 256-column tile of A converts and fetches B once where two 128-column CTAs did it twice, and the
// ring holds three stages of 64 KB instead of two per CTA.  Per k-block of 16 rows at 256 x 256 the TMA writes 32 KB, eight converter
// warps read 32 and write 64 KB and the MMAs read 144 KB: 1.1 us at 128 B per clock, as much as the tensor work (1.1 us).
// =====================================================================================
#define MN_STAGES_MAX 6
struct MnMaps {   // operands of the segments: C = sum over segments of A^T B
    CUtensorMap a[SAT_TN_SEGMENTS], b[SAT_TN_SEGMENTS];
};
#define MN_CONV_THREADS 256
#define MN_THREADS (64 + MN_CONV_THREADS)
#define MN_SMEM_MAX (227 * 1024)
#define MN_TURN_BYTES (8u * 32 * 33 * 4)   /* the epilogue turns eight 32 x 32 blocks around in the stages */
struct MnShared {
    uint64_t full[MN_STAGES_MAX], conv[MN_STAGES_MAX], empty[MN_STAGES_MAX];
    uint64_t accum;
    uint32_t tmem_base;
    int dead;
};

__global__ void __launch_bounds__(MN_THREADS, 2)
k_gemm_tc_mn(const __grid_constant__ MnMaps maps, int32_t seg_splits, int32_t Mdim, int32_t N, int64_t rps, int64_t rows,
             int32_t mt_max, int32_t bn, int32_t stages, uint32_t tmem_cols, float *part_C, float *part_cs, int *status)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    constexpr uint32_t blk_bytes = TC_BK * 128;            // one 32-column block of a k-block: 16 rows x 128 B
    constexpr uint32_t sub_bytes = (TC_BM / 32) * blk_bytes;  // one plane of 128 columns of A
    const int n_blks_b = (bn + 31) / 32;
    const uint32_t a_bytes = (uint32_t)mt_max * sub_bytes, b_bytes = (uint32_t)n_blks_b * blk_bytes;
    const uint32_t stage_bytes = 2 * a_bytes + 2 * b_bytes;  // [A hi | A lo | B hi | B lo]
    const uint32_t stage_area = (uint32_t)stages * stage_bytes > MN_TURN_BYTES ? (uint32_t)stages * stage_bytes : MN_TURN_BYTES;
    MnShared *sh = (MnShared *)(smem + stage_area);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t m0 = blockIdx.x * (mt_max * TC_BM), n0 = blockIdx.y * bn;
    const int32_t mt = (Mdim - m0 + TC_BM - 1) / TC_BM < mt_max ? (Mdim - m0 + TC_BM - 1) / TC_BM : mt_max;   // 128-column sub-tiles in use
    const int32_t seg = (int32_t)blockIdx.z / seg_splits;
    const int64_t r0 = (int64_t)((int32_t)blockIdx.z - seg * seg_splits) * rps, r1 = r0 + rps < rows ? r0 + rps : rows;
    const int32_t nkb = (int32_t)((r1 - r0 + TC_BK - 1) / TC_BK);

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&sh->full[s], 1);
            mbar_init(&sh->conv[s], MN_CONV_THREADS);
            mbar_init(&sh->empty[s], 1);
        }
        mbar_init(&sh->accum, 1);
        sh->dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        tc_alloc<1>(&sh->tmem_base, tmem_cols);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    volatile int *dead = &sh->dead;
    sat_grid_wait();   // everything above is set-up of this block; no global memory has been touched

    if (warp == 0) {
        if (lane == 0) {
            for (int32_t kb = 0; kb < nkb; ++kb) {
                const int s = kb % stages;
                const uint32_t ph = (uint32_t)(kb / stages) & 1u;
                if (!mbar_wait(&sh->empty[s], ph ^ 1u, dead, status)) break;
                uint8_t *st = smem + (size_t)s * stage_bytes;
                const int32_t r = (int32_t)(r0 + (int64_t)kb * TC_BK);
                mbar_expect_tx(&sh->full[s], (uint32_t)mt * sub_bytes + b_bytes);
                for (int bl = 0; bl < mt * (TC_BM / 32); ++bl) tma_load_2d(st + bl * blk_bytes, &maps.a[seg], &sh->full[s], m0 + bl * 32, r);
                for (int bl = 0; bl < n_blks_b; ++bl) tma_load_2d(st + 2 * a_bytes + bl * blk_bytes, &maps.b[seg], &sh->full[s], n0 + bl * 32, r);
            }
        }
    } else if (warp == 1) {
        const uint32_t idesc = make_idesc(TC_BM, bn, 1, 1);
        // MN-major 32-bit operands use the 128-byte swizzle with 32-byte atoms (the only layout the tensor core accepts for them):
        // 32-column blocks blk_bytes apart (leading offset), groups of 4 k-rows 512 B apart (stride offset); a k-step is 8 rows =
        // 1024 B.  Only the 14-bit start-address field (bytes >> 4) differs between the descriptors.
        const uint64_t desc0 = make_desc(smem_u32(smem), blk_bytes, 512, 1);
        for (int32_t kb = 0; kb < nkb; ++kb) {
            const int s = kb % stages;
            const uint32_t ph = (uint32_t)(kb / stages) & 1u;
            // the converters arrive on conv[s] only after they have seen full[s] (the TMA bytes) themselves
            if (!mbar_wait_all(&sh->conv[s], ph, dead, status)) break;
            tc_fence_after();
            const uint64_t st = desc0 + (uint64_t)(((uint32_t)s * stage_bytes) >> 4);
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < TC_BK / 8; ++ks) {
                    const uint64_t b_hi = st + (uint64_t)((2 * a_bytes + ks * 1024) >> 4), b_lo = b_hi + (b_bytes >> 4);
                    for (int i = 0; i < mt; ++i) {
                        const uint64_t a_hi = st + (uint64_t)(((uint32_t)i * sub_bytes + ks * 1024) >> 4), a_lo = a_hi + (a_bytes >> 4);
                        const uint32_t acc = tmem + (uint32_t)i * 256u;
                        tc_mma<1, 1>(acc, a_hi, b_hi, idesc, (kb > 0 || ks > 0) ? 1u : 0u);
                        tc_mma<2, 1>(acc, a_hi, b_lo, idesc, 1u);
                        tc_mma<0, 1>(acc, a_lo, b_hi, idesc, 1u);
                    }
                }
                tc_commit<1>(&sh->empty[s]);
            }
        }
        if (elect_one()) tc_commit<1>(&sh->accum);
    } else {
        const int ctid = threadIdx.x - 64;
        const bool want_cs = part_cs != nullptr && blockIdx.x == 0;
        // thread t takes 16-byte piece t % 128 of every second 32-column block; row (t % 128) / 8 of each k-block
        const uint32_t off = (uint32_t)(ctid & 127) * 16, half = (uint32_t)(ctid >> 7);
        // column sums in two levels (sixteen k-blocks, then their sums): in one, a long split's sum carried 3.3e-7 instead of 2.2e-7
        float4 cs[4], cs_sum[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) cs[i] = cs_sum[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        auto fold = [&]() {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                cs_sum[i].x += cs[i].x;
                cs_sum[i].y += cs[i].y;
                cs_sum[i].z += cs[i].z;
                cs_sum[i].w += cs[i].w;
                cs[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        };
        bool alive = true;
        for (int32_t kb = 0; kb < nkb && alive; ++kb) {
            const int s = kb % stages;
            const uint32_t ph = (uint32_t)(kb / stages) & 1u;
            alive = mbar_wait(&sh->full[s], ph, dead, status);
            if (!alive) break;
            uint8_t *ah = smem + (size_t)s * stage_bytes + off + half * blk_bytes, *bh = ah + 2 * a_bytes;
            float4 x[4];
            // loads first, four 16-byte pieces at a time (the loop is latency-bound otherwise)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if ((int)half + 2 * i < n_blks_b) x[i] = *reinterpret_cast<const float4 *>(bh + 2 * i * blk_bytes);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if ((int)half + 2 * i < n_blks_b) {
                    float4 h, l;
                    split4(x[i], h, l);
                    *reinterpret_cast<float4 *>(bh + 2 * i * blk_bytes) = h;
                    *reinterpret_cast<float4 *>(bh + 2 * i * blk_bytes + b_bytes) = l;
                    cs[i].x += x[i].x;
                    cs[i].y += x[i].y;
                    cs[i].z += x[i].z;
                    cs[i].w += x[i].w;
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < 2 * mt) x[i] = *reinterpret_cast<const float4 *>(ah + 2 * i * blk_bytes);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i < 2 * mt) {
                    float4 h, l;
                    split4(x[i], h, l);
                    *reinterpret_cast<float4 *>(ah + 2 * i * blk_bytes) = h;
                    *reinterpret_cast<float4 *>(ah + 2 * i * blk_bytes + a_bytes) = l;
                }
            }
            fence_async_smem();
            mbar_arrive(&sh->conv[s]);
            if ((kb & 15) == 15) fold();
        }
        fold();
        const int q = warp & 3, e = (warp - 2) >> 2;
        const bool ok = alive && mbar_wait(&sh->accum, 0, dead, status);   // every MMA has completed: the stages are free
        tc_fence_after();
        if (ok) {
            // two warps per TMEM lane quadrant: one per sub-tile, or alternate chunks of the only one.  Each turns its 32 x 32 blocks
            // around in shared memory and writes whole row segments: with one row per lane a store instruction touched 32 lines, and
            // the partial sums of a tile took 35 us
            float *tb = reinterpret_cast<float *>(smem) + (warp - 2) * (32 * 33);
            float *pc = part_C + (int64_t)blockIdx.z * Mdim * N;
            const int sub = mt > 1 ? e : 0;
            const int32_t row0 = m0 + sub * TC_BM + q * 32;
            for (int c0 = mt > 1 ? 0 : 32 * e; c0 < bn; c0 += mt > 1 ? 32 : 64) {
                uint32_t r[32];
                tc_ld32(tmem + (uint32_t)sub * 256u + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, r);
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 32; ++j) tb[lane * 33 + j] = __uint_as_float(r[j]);
                __syncwarp();
                const int32_t col = n0 + c0 + lane;
                if (col < N) {
#pragma unroll 8
                    for (int i = 0; i < 32; ++i)
                        if (row0 + i < Mdim) pc[(int64_t)(row0 + i) * N + col] = tb[i * 33 + lane];
                }
            }
        }
        if (want_cs) {
            // the 16 rows of a k-block lie in 16 groups of eight threads; the 32-byte atoms of a row are exchanged by its low two bits
            asm volatile("bar.sync 1, 256;" ::: "memory");
            float *cb = reinterpret_cast<float *>(smem);   // [16][n_blks_b * 32]
            const int rr = (ctid & 127) >> 3, piece = (ctid & 7) ^ ((rr & 3) << 1), w = n_blks_b * 32;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int bl = (int)half + 2 * i;
                if (bl < n_blks_b && ok) *reinterpret_cast<float4 *>(cb + rr * w + bl * 32 + piece * 4) = cs_sum[i];
            }
            asm volatile("bar.sync 1, 256;" ::: "memory");
            for (int c = ctid; c < w; c += MN_CONV_THREADS) {
                float t = cb[c];
                for (int g = 1; g < 16; ++g) t += cb[g * w + c];
                if (n0 + c < N && c < bn) part_cs[(int64_t)blockIdx.z * N + n0 + c] = t;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tc_dealloc<1>(tmem, tmem_cols);
    }
}

// =====================================================================================
// element-wise helpers
// =====================================================================================
// D = src o mask (written only when `dst` is non-null) and per-block column sums of it for the bias gradient.
// A block covers MASK_ROWS_PER_BLOCK rows; TPR threads (a power of two >= d / 4) walk one row with 128-bit accesses,
// 256 / TPR rows per pass; each thread keeps the running sum of its four columns, the row groups are added through
// shared memory in fixed order.
#define MASK_ROWS_PER_BLOCK 256
__global__ void __launch_bounds__(256)
k_mask_rows(const float *__restrict__ src, int64_t ld, int64_t rows, int32_t d, int32_t tpr, const uint32_t *__restrict__ mask,
            int32_t mask_words, const float *__restrict__ act, int64_t ld_act, int act_vec, float *__restrict__ dst, int64_t ld_dst,
            float *__restrict__ colsum_part)
{
    sat_grid_wait();
    __shared__ float4 red[256];
    const int c4 = threadIdx.x % tpr, rg = threadIdx.x / tpr, n_rg = 256 / tpr;
    const int64_t r0 = (int64_t)blockIdx.x * MASK_ROWS_PER_BLOCK;
    const int64_t r1 = (r0 + MASK_ROWS_PER_BLOCK < rows) ? r0 + MASK_ROWS_PER_BLOCK : rows;
    const int d4 = (d + 3) / 4;
    for (int cb = 0; cb < d4; cb += tpr) {  // column blocks (one unless d > 1024)
        const int c = cb + c4;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < d4) {
            // four rows in flight per thread (the loop is latency-bound otherwise); the sums are taken in row order
            for (int64_t r = r0 + rg; r < r1; r += 4 * n_rg) {
                float4 x[4];
                uint32_t w[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t rr = r + (int64_t)u * n_rg;
                    x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    w[u] = 0xFu;
                    if (rr < r1) {
                        x[u] = __ldg(reinterpret_cast<const float4 *>(src + rr * ld) + c);
                        if (mask) w[u] = __ldg(mask + rr * mask_words + (c >> 3)) >> ((c & 7) * 4);
                        if (act) {
                            const float *ar = act + rr * ld_act + 4 * c;
                            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (act_vec) a = __ldg(reinterpret_cast<const float4 *>(ar));
                            else {
                                a.x = ar[0];
                                if (4 * c + 1 < d) a.y = ar[1];
                                if (4 * c + 2 < d) a.z = ar[2];
                                if (4 * c + 3 < d) a.w = ar[3];
                            }
                            w[u] = (a.x > 0.f ? 1u : 0u) | (a.y > 0.f ? 2u : 0u) | (a.z > 0.f ? 4u : 0u) | (a.w > 0.f ? 8u : 0u);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t rr = r + (int64_t)u * n_rg;
                    if (rr >= r1) break;
                    if (!(w[u] & 1u)) x[u].x = 0.f;
                    if (!(w[u] & 2u)) x[u].y = 0.f;
                    if (!(w[u] & 4u)) x[u].z = 0.f;
                    if (!(w[u] & 8u)) x[u].w = 0.f;
                    if (4 * c + 3 >= d) {  // ragged tail: keep the padding columns out of the sums
                        if (4 * c + 1 >= d) x[u].y = 0.f;
                        if (4 * c + 2 >= d) x[u].z = 0.f;
                        x[u].w = 0.f;
                    }
                    if (dst) *(reinterpret_cast<float4 *>(dst + rr * ld_dst) + c) = x[u];
                    s.x += x[u].x; s.y += x[u].y; s.z += x[u].z; s.w += x[u].w;
                }
            }
        }
        if (colsum_part) {
            red[threadIdx.x] = s;
            __syncthreads();
            if (rg == 0 && c < d4) {
                float4 t = red[c4];
                for (int g = 1; g < n_rg; ++g) {
                    const float4 y = red[g * tpr + c4];
                    t.x += y.x; t.y += y.y; t.z += y.z; t.w += y.w;
                }
                float *o = colsum_part + (int64_t)blockIdx.x * d + 4 * c;
                o[0] = t.x;
                if (4 * c + 1 < d) o[1] = t.y;
                if (4 * c + 2 < d) o[2] = t.z;
                if (4 * c + 3 < d) o[3] = t.w;
            }
            __syncthreads();
        }
    }
}

// zero-padded bias for the tile width (optionally with the same gate interleave as the weights)
__global__ void k_pack_bias(const float *__restrict__ bias, int32_t n, int32_t n_pad, int32_t gate_h, float *__restrict__ out)
{
    sat_grid_wait();
    const int32_t np = blockIdx.x * blockDim.x + threadIdx.x;
    if (np >= n_pad) return;
    const int32_t nn = gate_h > 0 ? (np & 3) * gate_h + (np >> 2) : np;
    out[np] = np < n ? bias[nn] : 0.f;
}

// B operand [n_pad x k_pad] (K-major fp32, zero padded) from fp32 weights; the TF32 split happens in the GEMM kernel.
//   transpose = 1: W is [K x N] row-major (ldw) -> B[n][k] = W[k][n]          (C = A W)
//   transpose = 0: W is [N x K] row-major (ldw) -> B[n][k] = W[n][k]          (C = A W^T)
// A second source W2 (same orientation, k2 rows) continues along K at column offset k1_pad.
// A bias [n] is packed alike, zero padded (four gates with gates = 3 too).
// gate_h > 0: packed column 4 j + g is gate g of hidden unit j.  gates = 4: the sources have the columns i | f | g | o.  gates = 3 (GRU,
// sources r | z | n): the candidate's two parts stay apart, column 4 j + 2 takes n of the first source only and 4 j + 3 n of the second.
__global__ void k_split_weights(const float *__restrict__ W, int64_t ldw, int32_t k1, int32_t k1_pad, const float *__restrict__ W2,
                                int64_t ldw2, int32_t k2, int32_t n, int32_t n_pad, int32_t k_pad, int transpose, int32_t gate_h, int gates,
                                float *__restrict__ hi, float *__restrict__ lo, const float *__restrict__ bias, float *__restrict__ bias_out)
{
    sat_grid_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (bias && i < n_pad) bias_out[i] = i < n ? bias[gate_h > 0 ? ((int32_t)i & 3) * gate_h + ((int32_t)i >> 2) : (int32_t)i] : 0.f;
    if (i >= (int64_t)n_pad * k_pad) return;
    const int32_t np = (int32_t)(i / k_pad), kk = (int32_t)(i - (int64_t)np * k_pad);
    const int32_t g = np & 3;
    const int32_t nn = gate_h > 0 ? (gates == 3 && g == 3 ? 2 : g) * gate_h + (np >> 2) : np;  // packed row -> logical column
    float x = 0.f;
    if (np < n && !(gates == 3 && g == (kk < k1 ? 3 : 2))) {
        if (kk < k1) x = transpose ? W[(int64_t)kk * ldw + nn] : W[(int64_t)nn * ldw + kk];
        else if (kk >= k1_pad && kk - k1_pad < k2) x = transpose ? W2[(int64_t)(kk - k1_pad) * ldw2 + nn] : W2[(int64_t)nn * ldw2 + (kk - k1_pad)];
    }
    hi[i] = x;
    lo[i] = tf32_residual(x);  // second plane: read by the variants that do not split B in the kernel
}

// B operand from fp32 weights: per packed column the k-steps of 16 one after the other, each 16 hi and 16 lo halves (split_f16), zero padded to
// k-blocks of two k-steps, and the inverse of the column's scale.
//   transpose = 1: W is [K x N] row-major (ldw) -> B[n][k] = W[k][n]          (C = A W)
//   transpose = 0: W is [N x K] row-major (ldw) -> B[n][k] = W[n][k]          (C = A W^T)
// A second source W2 (same orientation, k2 rows) continues along K with a k-block of its own.
// A bias [n] is packed alike, zero padded (four gates with gates = 3 too).
// gate_h > 0: packed column 4 j + g is gate g of hidden unit j.  gates = 4: the sources have the columns i | f | g | o.  gates = 3 (GRU,
// sources r | z | n): the candidate's two parts stay apart, column 4 j + 2 takes n of the first source only and 4 j + 3 n of the second.
// Every column has its own scale, so that none loses bits to (or is overrun by) a larger neighbour; it is at most 2^100, so that an accumulator times its
// inverse (and 2^-SCALE_SHIFT) stays normal.  share: the eight columns of a block have one where their largest elements lie within 2^PACK_SHARE of each other
// (k_lstm_seq).  A block takes eight columns.  Its threads keep their pairs of terms in registers between the search for the largest and the
// split, PACK_PAIRS of them (a latency of the memory each time otherwise: 256 x 256 12 us -> 4), and look again at what is beyond.
#define PACK_COLS 8
#define PACK_SHARE 2
#define PACK_PAIRS 8
__global__ void __launch_bounds__(256)
k_pack_half(const float *__restrict__ W, int64_t ldw, int32_t k1, int32_t nkb1, const float *__restrict__ W2, int64_t ldw2, int32_t k2, int32_t nkb,
                int32_t n, int transpose, int32_t gate_h, int gates, int share, __half *__restrict__ out, float *__restrict__ unscale, const float *__restrict__ bias,
                float *__restrict__ bias_out)
{
    sat_grid_wait();
    __shared__ uint32_t largest[PACK_COLS];
    __shared__ float scale[PACK_COLS];
    const int32_t np0 = blockIdx.x * PACK_COLS, pairs = nkb * (TCH_BK / 2);
    auto value = [&](int32_t np, int32_t kk) {   // kk: term, the second source's from nkb1 k-blocks on
        const int32_t g = np & 3, nn = gate_h > 0 ? (gates == 3 && g == 3 ? 2 : g) * gate_h + (np >> 2) : np;   // packed row -> logical column
        const bool second = kk >= nkb1 * TCH_BK;
        const int32_t k = second ? kk - nkb1 * TCH_BK : kk;
        if (np >= n || k >= (second ? k2 : k1) || (gates == 3 && g == (second ? 2 : 3))) return 0.f;
        const float *w = second ? W2 : W;
        const int64_t ld = second ? ldw2 : ldw;
        return __ldg(transpose ? w + k * ld + nn : w + nn * ld + k);
    };
    // consecutive threads along the rows of the sources: pair p of column c
    const int32_t step_c = transpose ? 0 : 256 / pairs, step_p = transpose ? 32 : 256 % pairs;
    int32_t c = transpose ? threadIdx.x % PACK_COLS : threadIdx.x / pairs, p = transpose ? threadIdx.x / PACK_COLS : threadIdx.x - c * pairs;
    const int32_t c_first = c, p_first = p;
    auto advance = [&]() {
        c += step_c;
        p += step_p;
        if (!transpose && p >= pairs) p -= pairs, ++c;
    };
    auto inside = [&]() { return c < PACK_COLS && p < pairs; };
    if (threadIdx.x < PACK_COLS) {
        largest[threadIdx.x] = 0;
        const int32_t np = np0 + (int32_t)threadIdx.x;
        if (bias) bias_out[np] = np < n ? bias[gate_h > 0 ? (np & 3) * gate_h + (np >> 2) : np] : 0.f;
    }
    __syncthreads();
    float x[PACK_PAIRS][2];
#pragma unroll
    for (int i = 0; i < PACK_PAIRS; ++i) {
        const bool in = inside();
        x[i][0] = in ? value(np0 + c, 2 * p) : 0.f;
        x[i][1] = in ? value(np0 + c, 2 * p + 1) : 0.f;
        advance();
    }
    const int lane = threadIdx.x & 31;
    if (transpose) {   // a thread keeps to its column, and lanes eight apart share one
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < PACK_PAIRS; ++i) m = fmaxf(m, fmaxf(fabsf(x[i][0]), fabsf(x[i][1])));
        for (; inside(); advance()) m = fmaxf(m, fmaxf(fabsf(value(np0 + c, 2 * p)), fabsf(value(np0 + c, 2 * p + 1))));
        uint32_t b = __float_as_uint(m);
        b = max(b, __shfl_xor_sync(0xffffffffu, b, 8));
        b = max(b, __shfl_xor_sync(0xffffffffu, b, 16));
        if (lane < PACK_COLS) atomicMax(&largest[lane], b);
    } else {   // half a warp has pairs of one column: their number is a multiple of 16
        for (; inside(); advance()) atomicMax(&largest[c], __float_as_uint(fmaxf(fabsf(value(np0 + c, 2 * p)), fabsf(value(np0 + c, 2 * p + 1)))));
        c = c_first;
        p = p_first;
#pragma unroll
        for (int i = 0; i < PACK_PAIRS; ++i) {
            uint32_t b = __float_as_uint(fmaxf(fabsf(x[i][0]), fabsf(x[i][1])));
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
            if ((lane & 15) == 0 && inside()) atomicMax(&largest[c], b);
            advance();
        }
    }
    __syncthreads();
    if (threadIdx.x < PACK_COLS) {
        uint32_t l = largest[threadIdx.x] >> 23;
        if (share) {
            uint32_t least = 255, most = 0;
#pragma unroll
            for (int i = 0; i < PACK_COLS; ++i) {
                const uint32_t li = largest[i] >> 23;
                if (li > 0) least = min(least, li), most = max(most, li);
            }
            if (most < 255 && most <= least + PACK_SHARE) l = most;
        }
        const uint32_t e = min(f16_scale_exponent(l), 227u);
        scale[threadIdx.x] = __uint_as_float(e << 23);
        unscale[np0 + threadIdx.x] = __uint_as_float((254u - SCALE_SHIFT - e) << 23);
    }
    __syncthreads();
    auto put = [&](float x0, float x1) {
        uint32_t h, l;
        split_f16(x0 * scale[c], x1 * scale[c], h, l);
        uint32_t *o = reinterpret_cast<uint32_t *>(out + ((int64_t)(np0 + c) * (pairs / 8) + p / 8) * 32 + 2 * (p % 8));
        o[0] = h;
        o[8] = l;
    };
    c = c_first;
    p = p_first;
#pragma unroll
    for (int i = 0; i < PACK_PAIRS; ++i) {
        if (inside()) put(x[i][0], x[i][1]);
        advance();
    }
    for (; inside(); advance()) put(value(np0 + c, 2 * p), value(np0 + c, 2 * p + 1));
}

// out[r] = bits of the largest magnitude in row r of A: a warp per row (for matrices whose writer did not leave it)
__global__ void __launch_bounds__(256)
k_row_max(const float *__restrict__ A, int64_t lda, int32_t d, int64_t rows, uint32_t *__restrict__ out)
{
    sat_grid_wait();
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    float m = 0.f;
#pragma unroll 4
    for (int32_t c = 4 * lane; c < d; c += 128) {   // rows are padded to four floats; what stands there is not part of them
        const float4 x = __ldg(reinterpret_cast<const float4 *>(A + r * lda + c));
        m = fmaxf(m, fabsf(x.x));
        if (c + 1 < d) m = fmaxf(m, fabsf(x.y));
        if (c + 2 < d) m = fmaxf(m, fabsf(x.z));
        if (c + 3 < d) m = fmaxf(m, fabsf(x.w));
    }
    const uint32_t b = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if (lane == 0) out[r] = b;
}

// =====================================================================================
// host side
// =====================================================================================
typedef CUresult (*PFN_encodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                    const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static PFN_encodeTiled get_encode()
{
    static PFN_encodeTiled fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = (PFN_encodeTiled)p;
    }
    return fn;
}

// 2-D fp32 tensor map: `inner` contiguous elements per row, `outer` rows `ld` elements apart
static sat_status make_map(sat_ctx *ctx, CUtensorMap *map, const void *base, int64_t inner, int64_t outer, int64_t ld, int box_inner,
                           int box_outer, CUtensorMapSwizzle swz)
{
    PFN_encodeTiled enc = get_encode();
    if (!enc) return sat_fail(ctx, SAT_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
    cuuint64_t gdim[2] = {(cuuint64_t)(inner > 0 ? inner : 1), (cuuint64_t)(outer > 0 ? outer : 1)};
    cuuint64_t gstr[1] = {(cuuint64_t)ld * 4};
    cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_outer};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void *>(base), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return sat_fail(ctx, SAT_EINVAL, "cuTensorMapEncodeTiled failed (%d): base %p inner %lld outer %lld ld %lld", (int)r, base,
                                           (long long)inner, (long long)outer, (long long)ld);
    return SAT_OK;
}

// packed weights, a k-block of `box_cols` columns at a time
static sat_status make_map_weights(sat_ctx *ctx, CUtensorMap *map, const TcWeights &B, int box_cols)
{
    PFN_encodeTiled enc = get_encode();
    if (!enc) return sat_fail(ctx, SAT_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
    const cuuint64_t gdim[2] = {(cuuint64_t)B.ld, (cuuint64_t)B.n_pad}, gstr[1] = {(cuuint64_t)B.ld * 2};
    const cuuint32_t box[2] = {2 * TCH_BK, (cuuint32_t)box_cols}, estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, B.planes, gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return sat_fail(ctx, SAT_EINVAL, "cuTensorMapEncodeTiled failed (%d) for packed weights", (int)r);
    return SAT_OK;
}

// output columns per tile: as few tiles of at most 256 as possible, of equal width (a multiple of 32)
static int tile_n_for(int n)
{
    const int tiles = (n + 255) / 256;
    return ((n + tiles - 1) / tiles + 31) / 32 * 32;
}

bool sat_use_tc(int32_t n, int32_t k)
{
    static int no_tc = -1;
    if (no_tc < 0) {
        const char *e = getenv("SAT_NO_TC");
        no_tc = (e && e[0] == '1') ? 1 : 0;
    }
    return !no_tc && k >= 16 && n >= 16;
}

// The two forms of the K-major kernel.  Pairs pay where the contraction is long and the launch has more than a wave of row tiles; a short launch
// takes as long either way and its weights take 4 us to pack instead of 2 (epoch of 12,833 nodes, 192-200-200-83 with a GRU of 8 units: 393 us
// with TF32 terms, 424 with pairs), unless the contraction is very long (2,151 nodes, 21-512-512-35: 688 and 644).  A short
// contraction is bound by its output, and the epilogue with TF32 terms is the shorter one (169343 x 256, K = 40: 47.5 and 50.7
// us, K = 128 with the push 92 and 104).  The number of nodes stands for the rows of a launch, so that one partition and all of
// them in one launch give the same bits.
bool sat_tc_half(const sat_ctx *ctx, int32_t k) { return (k >= 384 || (k >= 192 && ctx->n >= 32768)) && sat_use_tc(16, k); }

sat_status sat_mask_rows(sat_ctx *ctx, const float *src, int32_t ld, int64_t rows, int32_t d, const uint32_t *mask, int32_t mask_words,
                         float *dst, int32_t ld_dst, float *colsum, int accumulate, const float *act, int32_t ld_act)
{
    if (rows == 0 || d == 0) return SAT_OK;
    if (!dst && !colsum) return SAT_OK;
    ProfScope prof(ctx, SATK_SPLIT, (dst ? 8.0 : 4.0) * (double)rows * d, 0.0);
    const int64_t blocks = cdiv64(rows, MASK_ROWS_PER_BLOCK);
    float *part = nullptr;
    if (colsum) {
        SAT_TRY(sat_ensure(ctx, ctx->buf_colsum, (size_t)blocks * d * sizeof(float)));
        part = (float *)ctx->buf_colsum.p;
    }
    int tpr = 1;
    while (tpr < (d + 3) / 4 && tpr < 256) tpr <<= 1;
    sat_pdl(ctx->stream, k_mask_rows, (unsigned)blocks, 256, 0)(src, ld, rows, d, tpr, mask, mask_words, act, ld_act, aligned16(act) && !(ld_act & 3),
                                                            dst, ld_dst, part);
    SAT_LAUNCHED(ctx);
    if (colsum) SAT_TRY(sat_splitk_reduce(ctx, part, d, (int32_t)blocks, accumulate, colsum, d, d));
    return SAT_OK;
}

// where weights packed as half-precision pairs with `nkb` k-blocks and n outputs lie in a buffer, and the bytes they take
static size_t half_layout(int32_t nkb, int32_t n, void *base, TcWeights *out)
{
    const int32_t bn = tile_n_for(n);
    out->n_pad = (n + bn - 1) / bn * bn;
    out->ld = nkb * 2 * TCH_BK;
    const size_t planes = (size_t)out->n_pad * out->ld * sizeof(__half);   // a multiple of 4 KB
    out->planes = base;
    out->unscale = (float *)((char *)base + planes);
    out->bias = out->unscale + out->n_pad;   // 16-byte aligned: n_pad is a multiple of 32
    return planes + 2 * (size_t)out->n_pad * sizeof(float);
}

sat_status sat_tc_weights(sat_ctx *ctx, const float *W, int32_t ldw, int32_t k1, const float *W2, int32_t ldw2, int32_t k2, int32_t n,
                          int transpose, DevBuf &buf, TcWeights *out, int32_t gate_h, int gates, const float *bias)
{
    if (out->half) {
        const int32_t nkb1 = (int32_t)cdiv64(k1, TCH_BK), nkb = nkb1 + (W2 ? (int32_t)cdiv64(k2, TCH_BK) : 0);
        SAT_TRY(sat_ensure(ctx, buf, half_layout(nkb, n, nullptr, out)));
        half_layout(nkb, n, buf.p, out);
        if (!bias) out->bias = nullptr;
        sat_pdl(ctx->stream, k_pack_half, (unsigned)(out->n_pad / PACK_COLS), 256, 0)(W, ldw, k1, nkb1, W2, ldw2, k2, nkb, n, transpose, gate_h, gates,
                                                                                  out->share, (__half *)out->planes, out->unscale, bias, out->bias);
        SAT_LAUNCHED(ctx);
        return SAT_OK;
    }
    const int32_t k1_pad = W2 ? (k1 + TC_BK - 1) / TC_BK * TC_BK : k1;
    const int32_t k_tot = k1_pad + (W2 ? k2 : 0);
    const int32_t k_pad = (k_tot + TC_BK - 1) / TC_BK * TC_BK;
    const int32_t bn = tile_n_for(n);
    const int32_t n_pad = (n + bn - 1) / bn * bn;
    const size_t plane = ((size_t)n_pad * k_pad * sizeof(float) + 255) & ~(size_t)255;
    SAT_TRY(sat_ensure(ctx, buf, 2 * plane + (bias ? (size_t)n_pad * sizeof(float) : 0)));
    out->hi = (float *)buf.p;
    out->lo = (float *)((char *)buf.p + plane);
    out->ld = k_pad;
    out->n_pad = n_pad;
    out->bias = bias ? (float *)((char *)buf.p + 2 * plane) : nullptr;
    sat_pdl(ctx->stream, k_split_weights, (unsigned)cdiv64((int64_t)n_pad * k_pad, 256), 256, 0)(W, ldw, k1, k1_pad, W2, ldw2, k2, n, n_pad, k_pad,
                                                                                          transpose, gate_h, gates, out->hi, out->lo, bias, out->bias);
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

// the description of planes that an earlier sat_tc_weights call (single source, k terms, n outputs, `bias`: with one) left in `buf`
sat_status sat_tc_weights_layout(int32_t k, int32_t n, const DevBuf &buf, TcWeights *out, bool bias)
{
    if (out->half) {
        if (!buf.p || buf.bytes < half_layout((int32_t)cdiv64(k, TCH_BK), n, buf.p, out)) return SAT_ESTATE;
        if (!bias) out->bias = nullptr;
        return SAT_OK;
    }
    const int32_t k_pad = (k + TC_BK - 1) / TC_BK * TC_BK;
    const int32_t bn = tile_n_for(n);
    const int32_t n_pad = (n + bn - 1) / bn * bn;
    const size_t plane = ((size_t)n_pad * k_pad * sizeof(float) + 255) & ~(size_t)255;
    if (!buf.p || buf.bytes < 2 * plane + (bias ? (size_t)n_pad * sizeof(float) : 0)) return SAT_ESTATE;
    out->hi = (float *)buf.p;
    out->lo = (float *)((char *)buf.p + plane);
    out->ld = k_pad;
    out->n_pad = n_pad;
    out->bias = bias ? (float *)((char *)buf.p + 2 * plane) : nullptr;
    return SAT_OK;
}

static PerDeviceOnce g_attr_mn;

struct TckLaunch {
    CUtensorMap mA, mA2, mB, mBlo, mC;
    int use_tma_store;
    int64_t m;
    int32_t n, nkb1, nkb2, bn, n_tiles_n;
    int64_t n_tiles;
    unsigned grid;
    uint32_t stage_bytes, b_resident;   // (half-precision pairs) bytes of a resident B
};

template <int EPI, int CTAS>
static sat_status launch_tck(sat_ctx *ctx, const TckLaunch &L, const TcEpilogue &ep)
{
    static PerDeviceOnce attr_set;
    // As many stages as fit, since the bytes in flight bound the narrow contractions (169343 x 128, K = 256: 86 us with 4 stages, 77 with
    // 6), but no more than the longest CTA has k-blocks, so that a small launch leaves room on the SM for its successor; an even number
    const size_t fixed = TckCfg<EPI>::out_bytes + (size_t)TckCfg<EPI>::epi_warps * TckCfg<EPI>::ring * 4096 + sizeof(TcShared) + 1024;
    const int64_t blocks = cdiv64(L.n_tiles, L.grid / CTAS) * (L.nkb1 + L.nkb2), fit = (227 * 1024 - (int64_t)fixed) / L.stage_bytes;
    uint32_t stages = TCK_STAGES_MAX;
    while (stages > 2 && (stages > fit || stages - 2 >= blocks)) stages -= 2;
    const size_t smem = (size_t)stages * L.stage_bytes + fixed;
    if (smem > 227 * 1024) return sat_fail(ctx, SAT_EINVAL, "tensor-core GEMM: shared-memory layout of %zu bytes does not fit", smem);
    if (attr_set.need(ctx->device)) {
        SAT_CUDA(ctx, cudaFuncSetAttribute(k_gemm_tc_k<EPI, CTAS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        attr_set.mark(ctx->device);
    }
    sat_pdl(ctx->stream, k_gemm_tc_k<EPI, CTAS>, L.grid, TCK_THREADS, smem, CTAS)(L.mA, L.mA2, L.mB, L.mBlo, L.mC, L.use_tma_store, stages, L.m, L.n, L.nkb1, L.nkb2, L.bn, L.n_tiles_n,
                                                                L.n_tiles, ep, ctx->d_flag + 1);
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

template <int EPI, int CTAS>
static sat_status launch_tch(sat_ctx *ctx, const TckLaunch &L, const TcEpilogue &ep)
{
    static PerDeviceOnce attr_set;
    // As many stages as fit, since the bytes in flight bound the narrow contractions, but no more than the longest CTA has k-blocks, so that a
    // small launch leaves room on the SM for its successor; an even number.
    const int64_t cta_tiles = cdiv64(L.n_tiles, L.grid / CTAS), blocks = cta_tiles * (L.nkb1 + L.nkb2);
    size_t fixed = TchCfg<EPI>::out_bytes + L.b_resident + sizeof(TchShared) + 1024;
    // two staging tiles per epilogue warp where they leave room for six stages 
    const uint32_t out_tiles = TchCfg<EPI>::out_bytes && cta_tiles > 1 && fixed + TchCfg<EPI>::out_bytes + 6 * L.stage_bytes <= 227 * 1024 ? 2 : 1;
    fixed += (out_tiles - 1) * TchCfg<EPI>::out_bytes;
    const int64_t fit = (227 * 1024 - (int64_t)fixed) / L.stage_bytes;
    uint32_t stages = TCH_STAGES_MAX;
    while (stages > 2 && (stages > fit || stages - 2 >= blocks)) stages -= 2;
    const size_t smem = (size_t)stages * L.stage_bytes + fixed;
    if (smem > 227 * 1024) return sat_fail(ctx, SAT_EINVAL, "tensor-core GEMM: shared-memory layout of %zu bytes does not fit", smem);
    if (attr_set.need(ctx->device)) {
        SAT_CUDA(ctx, cudaFuncSetAttribute(k_gemm_tc_h<EPI, CTAS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        attr_set.mark(ctx->device);
    }
    sat_pdl(ctx->stream, k_gemm_tc_h<EPI, CTAS>, L.grid, TCH_THREADS, smem, CTAS)(L.mA, L.mA2, L.mB, L.mC, L.use_tma_store, stages, out_tiles, L.b_resident > 0, L.m, L.n, L.nkb1, L.nkb2, L.bn, L.n_tiles_n,
                                                                L.n_tiles, ep, ctx->d_flag + 1);
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

sat_status sat_row_max(sat_ctx *ctx, const float *A, int32_t lda, int32_t d, int64_t rows, uint32_t *out)
{
    if (rows == 0) return SAT_OK;
    sat_pdl(ctx->stream, k_row_max, (unsigned)cdiv64(rows, 8), 256, 0)(A, lda, d, rows, out);
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

// C[m x n] = [A | A2] B^T with B = packed weights [n_pad x k_pad]
sat_status sat_gemm_tc(sat_ctx *ctx, int64_t m, int32_t n, const float *A, int32_t lda, int32_t k1, const float *A2, int32_t lda2, int32_t k2,
                       const TcWeights &Bw, const TcEpilogueHost &eh, int family)
{
    if (m == 0 || n == 0) return SAT_OK;
    const bool half = Bw.half;
    const int32_t bk = half ? TCH_BK : TC_BK, nkb1 = (int32_t)cdiv64(k1, bk), nkb2 = A2 ? (int32_t)cdiv64(k2, bk) : 0;
    const int32_t bn = tile_n_for(n);
    // CTA pairs for launches of more than one wave of single CTAs (below, the pair only adds its synchronisation: 6000 x 72, K = 50: 12.0
    // -> 12.9 us), except with a gathered residual: that contracts over the predictor width and is bound by the residual's
    // stream, which the pair holds up (145 -> 161 us at 169343 rows)
    const int32_t n_tiles_n = (int32_t)cdiv64(n, bn);
    const bool pair = !eh.resid_idx && cdiv64(m, TC_BM) * n_tiles_n > ctx->sms;
    const int ctas = pair ? 2 : 1;
    // a B of half-precision pairs of at most 128 KB per CTA stays in shared memory, where there are as many CTAs (or pairs) as column tiles: it is
    // loaded once, for the columns of the CTA's first tile, so the number of CTAs has to be a multiple of the number of column tiles
    int64_t units = ctx->sms / ctas;
    const uint32_t b_bytes = (uint32_t)bn / ctas * 128;
    const int64_t b_all = (int64_t)b_bytes * (nkb1 + nkb2);
    const uint32_t b_resident = half && b_all <= 131072 && n_tiles_n <= units ? (uint32_t)b_all : 0;
    if (b_resident) units -= units % n_tiles_n;
    const uint32_t stage_bytes = half ? TCH_A_BYTES + (b_resident ? 0 : b_bytes) : 2 * (TC_BM * TC_BK * 4) + b_bytes;
    // algorithmic bytes: operands once, results once.  Plain: A, B, C.  Gathered residual: + the residual rows.  LSTM cell:
    // the output is the hidden state [m x h] plus the cell state read and written, and the cached projection if it is added.
    double alg_bytes = 4.0 * ((double)m * (k1 + k2) + (double)(k1 + k2) * n);
    if (eh.lstm_h > 0) alg_bytes += 4.0 * (double)m * eh.lstm_h * (eh.gru ? 1.0 : eh.lstm_first ? 2.0 : 3.0);
    else alg_bytes += 4.0 * (double)m * n * (eh.resid_idx ? 2.0 : 1.0);
    ProfScope prof(ctx, family, alg_bytes, 2.0 * (double)m * n * (k1 + k2));
    CUtensorMap mA, mA2, mB, mBlo, mC;
    const int use_tma_store = eh.lstm_h == 0 && eh.proj_h == 0 && ((eh.ldc & 3) == 0) && ((((uintptr_t)eh.C) & 15u) == 0);
    if (use_tma_store) SAT_TRY(make_map(ctx, &mC, eh.C, n, m, eh.ldc, 32, 32, CU_TENSOR_MAP_SWIZZLE_128B));
    else memset(&mC, 0, sizeof(mC));
    const CUtensorMapSwizzle swz = half ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    SAT_TRY(make_map(ctx, &mA, A, k1, m, lda, bk, TC_BM, swz));
    if (A2) SAT_TRY(make_map(ctx, &mA2, A2, k2, m, lda2, bk, TC_BM, swz));
    else mA2 = mA;
    if (half) {
        SAT_TRY(make_map_weights(ctx, &mB, Bw, bn / ctas));
        mBlo = mB;
    } else {
        SAT_TRY(make_map(ctx, &mB, Bw.hi, Bw.ld, Bw.n_pad, Bw.ld, TC_BK, bn / ctas, swz));
        SAT_TRY(make_map(ctx, &mBlo, Bw.lo, Bw.ld, Bw.n_pad, Bw.ld, TC_BK, bn / ctas, swz));
    }
    TcEpilogue ep;
    if (half && (!eh.rows.p || eh.resid_idx)) return sat_fail(ctx, SAT_EINVAL, "a contraction on half-precision pairs needs the largest magnitudes of its rows and has no residual");
    ep.row_max = eh.rows.p;
    ep.row_stride = eh.rows.stride;
    ep.row_parts = eh.rows.parts;
    ep.row_least = A2 ? 0x3f800000u : 0u;   // a second operand is a hidden state, which lies in [-1, 1]
    ep.k1 = k1;
    ep.k2 = A2 ? k2 : 0;
    ep.unscale = Bw.unscale;
    ep.push_max = eh.push_max;
    ep.C = eh.C;
    ep.ldc = eh.ldc;
    ep.bias = nullptr;
    if (eh.bias && Bw.bias) {
        ep.bias = Bw.bias;   // packed with the weights
    } else if (eh.bias) {  // zero-padded copy so that the epilogue can read whole 128-bit vectors
        const size_t padded = (size_t)cdiv64(n, bn) * bn;
        DevBuf &home = eh.bias_home ? *eh.bias_home : ctx->buf_bias;
        if (!(eh.bias_home && eh.bias_ready && home.bytes >= padded * sizeof(float))) {
            SAT_TRY(sat_ensure(ctx, home, padded * sizeof(float)));
            sat_pdl(ctx->stream, k_pack_bias, (unsigned)cdiv64(padded, 256), 256, 0)(eh.bias, n, (int32_t)padded, eh.lstm_h > 0 ? eh.lstm_h : eh.proj_h,
                                                                                (float *)home.p);
            SAT_LAUNCHED(ctx);
        }
        ep.bias = (const float *)home.p;
    }
    ep.push_dst = eh.push_dst;
    ep.push_slot = eh.push_slot;
    ep.ld_push = eh.ld_push;
    if (eh.push_dst && (eh.lstm_h > 0 || eh.resid_idx || !eh.push_slot || (eh.ld_push & 3) || (((uintptr_t)eh.push_dst) & 15u)))
        return sat_fail(ctx, SAT_EINVAL, "push epilogue needs a slot map, an aligned destination and the plain epilogue");
    ep.lstm_h = eh.lstm_h;
    ep.lstm_first = eh.lstm_first;
    ep.lstm_c = eh.lstm_c;
    ep.proj_h = eh.proj_h;
    if (eh.lstm_h > 0 && (!eh.bias || (!eh.gru && !eh.lstm_c) || n != 4 * eh.lstm_h))
        return sat_fail(ctx, SAT_EINVAL, "fused recurrent epilogue needs bias, cell state (LSTM) and n = 4h");
    if (eh.resid_idx && (eh.mask_out || eh.lstm_h > 0))
        return sat_fail(ctx, SAT_EINVAL, "gathered-residual epilogue cannot be combined with a mask output or the LSTM cell");
    ep.relu = eh.relu;
    ep.mask_out = eh.mask_out;
    ep.mask_words = eh.mask_words;
    ep.mask_in = eh.mask_in;
    ep.mask_in_words = eh.mask_in_words;
    if (eh.mask_in && (eh.lstm_h > 0 || eh.proj_h > 0 || eh.resid_idx || eh.push_dst)) return sat_fail(ctx, SAT_EINVAL, "an input mask needs the plain epilogue");
    ep.resid = eh.resid;
    ep.resid_idx = eh.resid_idx;
    ep.ld_resid = eh.ld_resid;
    ep.tile_order = eh.tile_order;
    const int64_t n_tiles = cdiv64(m, TC_BM * ctas) * n_tiles_n;
    const unsigned grid = (unsigned)(n_tiles < units ? n_tiles : units) * ctas;
    TckLaunch L;
    L.mA = mA; L.mA2 = mA2; L.mB = mB; L.mBlo = mBlo; L.mC = mC;
    L.use_tma_store = use_tma_store;
    L.m = m; L.n = n; L.nkb1 = nkb1; L.nkb2 = nkb2; L.bn = bn; L.n_tiles_n = n_tiles_n; L.n_tiles = n_tiles;
    L.grid = grid;
    L.stage_bytes = stage_bytes;
    L.b_resident = b_resident;
    if (half) {
        if (eh.gru) return pair ? launch_tch<EPI_GRU, 2>(ctx, L, ep) : launch_tch<EPI_GRU, 1>(ctx, L, ep);
        if (ep.proj_h > 0) return pair ? launch_tch<EPI_PROJ, 2>(ctx, L, ep) : launch_tch<EPI_PROJ, 1>(ctx, L, ep);
        if (ep.lstm_h > 0) return pair ? launch_tch<EPI_LSTM, 2>(ctx, L, ep) : launch_tch<EPI_LSTM, 1>(ctx, L, ep);
        if (ep.push_dst) return pair ? launch_tch<EPI_PUSH, 2>(ctx, L, ep) : launch_tch<EPI_PUSH, 1>(ctx, L, ep);
        return pair ? launch_tch<EPI_PLAIN, 2>(ctx, L, ep) : launch_tch<EPI_PLAIN, 1>(ctx, L, ep);
    }
    if (eh.gru) return pair ? launch_tck<EPI_GRU, 2>(ctx, L, ep) : launch_tck<EPI_GRU, 1>(ctx, L, ep);
    if (ep.proj_h > 0) return pair ? launch_tck<EPI_PROJ, 2>(ctx, L, ep) : launch_tck<EPI_PROJ, 1>(ctx, L, ep);
    if (ep.lstm_h > 0) return pair ? launch_tck<EPI_LSTM, 2>(ctx, L, ep) : launch_tck<EPI_LSTM, 1>(ctx, L, ep);
    if (ep.resid_idx) return launch_tck<EPI_RESID, 1>(ctx, L, ep);
    if (ep.push_dst) return pair ? launch_tck<EPI_PUSH, 2>(ctx, L, ep) : launch_tck<EPI_PUSH, 1>(ctx, L, ep);
    return pair ? launch_tck<EPI_PLAIN, 2>(ctx, L, ep) : launch_tck<EPI_PLAIN, 1>(ctx, L, ep);
}

sat_status sat_lstm_seq(sat_ctx *ctx, int64_t rows, int32_t h, const TcWeights &Uh, const float *const *proj, int32_t n_steps, int first, float *S,
                        float *cell, int write_cell)
{
    if (rows == 0 || n_steps == 0) return SAT_OK;
    if (n_steps > SAT_SEQ_MAX || h > 64 || (h & 3)) return sat_fail(ctx, SAT_EINVAL, "sat_lstm_seq: at most %d steps and 64 units", SAT_SEQ_MAX);
    ProfScope prof(ctx, SATK_GEMM_SIDE, 4.0 * (double)rows * h * (4.0 * n_steps + 1.0 + (first ? 0.0 : 2.0)), 8.0 * (double)rows * h * h * (n_steps - (first ? 1 : 0)));
    const int32_t bn = tile_n_for(4 * h), nkb = (h + TCH_BK - 1) / TCH_BK;
    const size_t smem = (size_t)nkb * (2 * TC_BM + bn) * 128 + (size_t)SEQ_RING * 4 * SEQ_THREADS * 16 + sizeof(SeqShared) + 1024;
    static PerDeviceOnce attr_set;
    if (attr_set.need(ctx->device)) {
        SAT_CUDA(ctx, cudaFuncSetAttribute(k_lstm_seq, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        attr_set.mark(ctx->device);
    }
    CUtensorMap mB;
    SAT_TRY(make_map_weights(ctx, &mB, Uh, bn));
    SeqSteps st;
    for (int32_t t = 0; t < SAT_SEQ_MAX; ++t) st.proj[t] = t < n_steps ? proj[t] : nullptr;
    const int64_t tiles = cdiv64(rows, TC_BM);
    sat_pdl(ctx->stream, k_lstm_seq, (unsigned)(tiles < ctx->sms ? tiles : ctx->sms), SEQ_THREADS, smem)(mB, Uh.unscale, st, n_steps, first, rows, h, bn, nkb, S, cell,
                                                                                              write_cell, ctx->d_flag + 1);
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

// C[m x n] (+)= sum_i A[i]^T B[i] over `rows` rows each: A fp32 [rows x m] (lda), B fp32 [rows x n] (ldb)
sat_status sat_gemm_tc_tn(sat_ctx *ctx, int64_t rows, int32_t m, int32_t n, const float *const *A, int32_t lda, const float *const *B, int32_t ldb,
                          int32_t segments, float *C, int32_t ldc, int accumulate, float *colsum, int32_t reserve)
{
    if (m == 0 || n == 0) return SAT_OK;
    if (segments < 1 || segments > SAT_TN_SEGMENTS) return sat_fail(ctx, SAT_EINVAL, "sat_gemm_tc_tn: 1 to %d segments", SAT_TN_SEGMENTS);
    ProfScope prof(ctx, SATK_GEMM_TN, 4.0 * ((double)rows * segments * (m + n) + (double)m * n), 2.0 * (double)rows * segments * m * n);
    // Tiles of 256 columns of A where they are all full, else of 128 with two CTAs per SM (256 of the 512 TMEM columns each): 179250 x
    // 300 x 512 376 -> 370 us, 58241 x 602 x 256 119 -> 136 us with the splits below.
    const int32_t bn = tile_n_for(n), subs = (int32_t)cdiv64(m, TC_BM), mt = subs % 2 == 0 ? 2 : 1;
    const uint32_t stage_bytes = 2 * (uint32_t)mt * (TC_BM / 32) * TC_BK * 128 + 2 * (uint32_t)((bn + 31) / 32) * TC_BK * 128;
    const int64_t r1 = rows > 0 ? rows : 1, kblocks = cdiv64(r1, TC_BK);
    const int per_sm = mt == 1 ? 2 : 1;
    const int64_t col_tiles = cdiv64(n, bn), tiles = cdiv64(m, mt * TC_BM) * col_tiles;
    // Row splits of a segment, in whole waves.  The accumulation truncates, so the error of a split's sum grows with its length, while the
    // partial sums are added with rounding: a split is not longer than with two 128-column tiles per SM, whatever the tile and however many
    // segments share the launch (one wave over all segments: relative error of the predictor's gradients 8e-6 -> 6e-5 at 512 columns and
    // eight steps; one wave of 256-column tiles over 300 columns 7.2e-5 -> 8.7e-5).  Not less than six k-blocks each: the m x n partial
    // sums of a split, written and read again, cost about as much as that.
    const int64_t least = cdiv64(2 * ctx->sms, (int64_t)subs * col_tiles), slots = (int64_t)ctx->sms * per_sm;
    auto splits_of = [&](int32_t segs) {
        const int64_t per_split = tiles * segs, waves = cdiv64(least * per_split, slots);
        return std::min<int64_t>(per_split < slots * waves ? slots * waves / per_split : 1, cdiv64(kblocks, 6));
    };
    int64_t splits = splits_of(segments);
    const int64_t kpb = cdiv64(kblocks, splits), rps = kpb * TC_BK;
    splits = cdiv64(r1, rps);
    int64_t stages = (MN_SMEM_MAX / per_sm - 1024 - (int)sizeof(MnShared) - 1024) / stage_bytes;
    if (stages > MN_STAGES_MAX) stages = MN_STAGES_MAX;
    if (stages > kpb) stages = kpb;
    const size_t need = (size_t)stages * stage_bytes, turn = MN_TURN_BYTES;
    const size_t smem = (need > turn ? need : turn) + sizeof(MnShared) + 1024;
    // room for `reserve` segments at once: a window that fills epoch by epoch would grow it in each of them
    const int64_t parts = std::max<int64_t>(splits * segments, reserve > segments ? splits_of(reserve) * reserve : 0);
    SAT_TRY(sat_ensure(ctx, ctx->buf_splitk, (size_t)parts * ((size_t)m * n + n) * sizeof(float)));
    float *part = (float *)ctx->buf_splitk.p;
    float *part_cs = colsum ? part + (size_t)(splits * segments) * m * n : nullptr;
    MnMaps maps;
    for (int32_t i = 0; i < segments; ++i) {
        SAT_TRY(make_map(ctx, &maps.a[i], A[i], m, rows, lda, 32, TC_BK, CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B));
        SAT_TRY(make_map(ctx, &maps.b[i], B[i], n, rows, ldb, 32, TC_BK, CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B));
    }
    for (int32_t i = segments; i < SAT_TN_SEGMENTS; ++i) maps.a[i] = maps.a[0], maps.b[i] = maps.b[0];
    if (g_attr_mn.need(ctx->device)) {
        SAT_CUDA(ctx, cudaFuncSetAttribute(k_gemm_tc_mn, cudaFuncAttributeMaxDynamicSharedMemorySize, MN_SMEM_MAX));
        g_attr_mn.mark(ctx->device);
    }
    dim3 grid((unsigned)cdiv64(m, mt * TC_BM), (unsigned)cdiv64(n, bn), (unsigned)(splits * segments));
    sat_pdl(ctx->stream, k_gemm_tc_mn, grid, MN_THREADS, smem)(maps, (int32_t)splits, m, n, rps, r1, mt, bn, (int32_t)stages, mt == 1 ? 256u : 512u, part, part_cs,
                                                       ctx->d_flag + 1);
    SAT_LAUNCHED(ctx);
    return sat_splitk_reduce(ctx, part, (int64_t)m * n, (int32_t)(splits * segments), accumulate, C, n, ldc, part_cs, n, colsum);
}

sat_status sat_gemm_tc_tn(sat_ctx *ctx, int64_t rows, int32_t m, int32_t n, const float *A, int32_t lda, const float *B, int32_t ldb, float *C,
                          int32_t ldc, int accumulate, float *colsum)
{
    return sat_gemm_tc_tn(ctx, rows, m, n, &A, lda, &B, ldb, 1, C, ldc, accumulate, colsum, 0);
}
