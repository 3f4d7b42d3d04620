// Lossy storage of historical embeddings (Supplement, "Data Compression for Historical Embedding Storage"): the
// encoded-polyline scheme applied to every row of an fp32 matrix.
//   q_j = round-half-away-from-zero(x_j * 10^p)   (fp64: the product of an fp32 value and 10^p, p <= 7, is exact)
//   e_0 = q_0, e_j = q_j - q_{j-1};  v = e << 1, bitwise inverted when e < 0
//   5-bit groups of v, least significant first, bit 0x20 on all but the last, each + 63 -> one byte
// One warp per row in all three kernels; a lane owns four consecutive values.  The code length of an element depends only on x_j and
// x_{j-1}, so sizes and bytes are produced element-parallel (warp prefix sums give the byte positions); the bytes of 128 values
// meet in shared memory and leave as 16-byte words.  Decoding takes 512 bytes at a time: a byte below 0x20 (after the -63) ends a
// value, the values are then assembled one per lane, and a warp prefix sum turns the deltas into values.
// Instruction issue is what bounds all three (86 % of the slots, DRAM below a third), so the usual case runs in 32 bits: a quantised
// value below 2^22 comes from an exact two-term fp32 product, and a decoded one below 2^24 is one reciprocal product and one
// remainder step away from the correctly rounded quotient (both operands are 24-bit integers, and a double quotient has more than twice
// their bits, so this is what rounding the double quotient gives).  Anything larger takes the same steps in 64 bits.  164,833 x 256
// ReLU outputs at p = 3: sizes 119 -> 66, encode 198 -> 158, decode 628 -> 257 us.
#include "sat_internal.h"

#define CODEC_MAX_GROUPS 13  /* 64 bits / 5 */
#define CODEC_CHUNK 128      /* values per warp and step */

__device__ __forceinline__ int64_t codec_quantise(float x, double scale) { return llround((double)x * scale); }
// the same for products below 2^22: x s = hi + lo exactly; adding 2^23 rounds |hi| to the nearest integer m (kept in the low bits of the
// sum), and m moves by one where what is left, lo included, reaches one half or falls below minus one half (every difference here
// is exact where it decides: |lo| is at most half an ulp of hi).  No conversion instruction: they run at an eighth of the rate.
__device__ __forceinline__ bool codec_quantise32(float x, float s, int32_t *q)
{
    const float hi = x * s, lo = fmaf(x, s, -hi), a = fabsf(hi), r = a + 8388608.f, rest = a - (r - 8388608.f);
    const float l = __int_as_float(__float_as_int(lo) ^ (__float_as_int(hi) & (int)0x80000000u));   // lo with the sign of hi taken out
    const int32_t m = (__float_as_int(r) & 0x7fffff) + (rest - 0.5f >= -l ? 1 : 0) - (rest + 0.5f < -l ? 1 : 0);
    *q = hi < 0.f ? -m : m;
    return a < 4194304.f;   // false for NaN as well
}
__device__ __forceinline__ uint64_t codec_fold(int64_t e)
{
    const uint64_t v = (uint64_t)e << 1;
    return e < 0 ? ~v : v;
}
__device__ __forceinline__ uint32_t codec_fold(int32_t e) { return ((uint32_t)e << 1) ^ (uint32_t)(e >> 31); }
__device__ __forceinline__ int codec_len(uint64_t v) { return v == 0 ? 1 : (64 - __clzll((long long)v) + 4) / 5; }
__device__ __forceinline__ int codec_len(uint32_t v) { return (int)(((uint32_t)(36 - __clz((int)(v | 1u))) * 205u) >> 10); }   // (bits + 4) / 5

__device__ __forceinline__ void codec_load(const float *__restrict__ row, int32_t d, int32_t j, bool vec, float (&x)[4])
{
    if (vec && j + 3 < d) {
        const float4 t = __ldg(reinterpret_cast<const float4 *>(row + j));
        x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = j + k < d ? row[j + k] : 0.f;
    }
}
__device__ __forceinline__ bool codec_quantise4(const float (&x)[4], float s, int32_t (&q)[4])
{
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) ok &= codec_quantise32(x[k], s, &q[k]);
    return ok;
}
template <typename Q>
__device__ __forceinline__ Q codec_pick(const Q (&q)[4], int k) { return k == 0 ? q[0] : k == 1 ? q[1] : k == 2 ? q[2] : q[3]; }
// deltas against the value before: the lane below's last one, `carry` (the last value of the chunk before, 0 at the start) for lane 0;
// carry becomes the last value of this chunk of `cnt` values
template <typename Q>
__device__ __forceinline__ void codec_deltas(Q (&q)[4], int lane, int32_t cnt, Q &carry)
{
    Q prev = __shfl_up_sync(0xffffffffu, q[3], 1);
    if (lane == 0) prev = carry;
    carry = cnt == CODEC_CHUNK ? __shfl_sync(0xffffffffu, q[3], 31) : __shfl_sync(0xffffffffu, codec_pick(q, (cnt - 1) & 3), (cnt - 1) >> 2);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const Q t = q[k];
        q[k] = t - prev;
        prev = t;
    }
}
// whether a carry lets the next chunk run in 32 bits (it is kept in 64 from chunk to chunk)
__device__ __forceinline__ bool codec_small(int64_t carry) { return carry > -(1 << 22) && carry < (1 << 22); }

template <typename Q>
__device__ __forceinline__ Q codec_scan(Q x, int lane, Q *total)
{
    Q incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Q up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
    }
    *total = __shfl_sync(0xffffffffu, incl, 31);
    return incl;
}

__global__ void __launch_bounds__(256)
k_codec_sizes(const float *__restrict__ x, int64_t ld, int64_t rows, int32_t d, int vec, float scale32, double scale, int32_t *__restrict__ row_bytes)
{
    sat_grid_wait();
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    int32_t total = 0;
    int64_t carry = 0;
    for (int32_t j0 = 0; j0 < d; j0 += CODEC_CHUNK) {
        const int32_t cnt = d - j0 < CODEC_CHUNK ? d - j0 : CODEC_CHUNK, left = cnt - 4 * lane;
        float v[4];
        int32_t q[4];
        codec_load(x + r * ld, d, j0 + 4 * lane, vec, v);
        if (__all_sync(0xffffffffu, codec_quantise4(v, scale32, q)) && codec_small(carry)) {
            int32_t c = (int32_t)carry;
            codec_deltas(q, lane, cnt, c);
            carry = c;
#pragma unroll
            for (int k = 0; k < 4; ++k) total += k < left ? codec_len(codec_fold(q[k])) : 0;
        } else {
            int64_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = codec_quantise(v[k], scale);
            codec_deltas(w, lane, cnt, carry);
#pragma unroll
            for (int k = 0; k < 4; ++k) total += k < left ? codec_len(codec_fold(w[k])) : 0;
        }
    }
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    if (lane == 0) row_bytes[r] = total;
}

// the bytes of a folded value below 2^20 (at most four): five bits per byte, 63 added, 0x20 on every byte but the last
__device__ __forceinline__ uint32_t codec_bytes(uint32_t v, int len)
{
    uint32_t t = (v & 0x3ffu) | ((v & 0xffc00u) << 6);
    t = (t & 0x001f001fu) | ((t & 0x03e003e0u) << 3);
    t += 0x3f3f3f3fu + (0x20202020u & ((1u << (8 * (len - 1))) - 1u));
    return len == 4 ? t : t & ((1u << (8 * len)) - 1u);
}

#define CODEC_BUF ((16 + CODEC_CHUNK * CODEC_MAX_GROUPS + 15) / 16 * 16)
__global__ void __launch_bounds__(256)
k_codec_encode(const float *__restrict__ x, int64_t ld, int64_t rows, int32_t d, int vec, float scale32, double scale,
               const int64_t *__restrict__ offsets, uint8_t *__restrict__ out)
{
    sat_grid_wait();
    __shared__ __align__(16) uint8_t bufs[8][CODEC_BUF + 16];
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    uint8_t *buf = bufs[threadIdx.x >> 5];
    uint4 *buf16 = reinterpret_cast<uint4 *>(buf);
    uint32_t *buf4 = reinterpret_cast<uint32_t *>(buf);
    // buf[i] goes to base[i]; base is 16-byte aligned, the first `skip` bytes of the first word belong to the row before
    uint8_t *base = out + offsets[r];
    int32_t skip = (int32_t)((uintptr_t)base & 15u), fill = skip;
    base -= skip;
    int64_t carry = 0;
    if (lane == 0) buf16[0] = make_uint4(0, 0, 0, 0);
    __syncwarp();   // a chunk of large values writes its bytes without another wait
    for (int32_t j0 = 0; j0 < d; j0 += CODEC_CHUNK) {
        const int32_t cnt = d - j0 < CODEC_CHUNK ? d - j0 : CODEC_CHUNK, left = cnt - 4 * lane;
        float v[4];
        int32_t q[4];
        codec_load(x + r * ld, d, j0 + 4 * lane, vec, v);
        // the usual chunk: every value fits four bytes
        bool four = codec_quantise4(v, scale32, q) && codec_small(carry);
        if (__all_sync(0xffffffffu, four)) {
            int32_t c = (int32_t)carry;
            codec_deltas(q, lane, cnt, c);
            uint32_t f[4];
            four = true;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                f[k] = codec_fold(q[k]);
                four &= k >= left || f[k] < (1u << 20);
            }
            four = __all_sync(0xffffffffu, four);
            if (four) {
                carry = c;
                int len[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) len[k] = k < left ? codec_len(f[k]) : 0;
                const int ln = len[0] + len[1], total = ln + len[2] + len[3];   // bytes of the first two, and of all
                int32_t sum;
                const int32_t at = fill + codec_scan<int32_t>(total, lane, &sum) - total;
                fill += sum;
                // the lane's bytes as a 128-bit string, or-ed into the zeroed buffer word by word
                for (int32_t w = 1 + lane; w <= fill >> 4; w += 32) buf16[w] = make_uint4(0, 0, 0, 0);
                __syncwarp();
                if (total > 0) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) f[k] = len[k] ? codec_bytes(f[k], len[k]) : 0u;
                    const uint64_t lo = (uint64_t)f[0] | ((uint64_t)f[1] << (8 * len[0])), hi = (uint64_t)f[2] | ((uint64_t)f[3] << (8 * len[2]));
                    const uint64_t s0 = ln < 8 ? lo | (hi << (8 * ln)) : lo, s1 = hi >> (64 - 8 * ln);   // ln >= 1
                    const uint32_t w0 = (uint32_t)s0, w1 = (uint32_t)(s0 >> 32), w2 = (uint32_t)s1, w3 = (uint32_t)(s1 >> 32);
                    const int sh = 8 * (at & 3), n_words = ((at & 3) + total + 3) >> 2;
                    uint32_t *dst = buf4 + (at >> 2);
                    atomicOr(dst, w0 << sh);
                    if (n_words > 1) atomicOr(dst + 1, __funnelshift_l(w0, w1, sh));
                    if (n_words > 2) atomicOr(dst + 2, __funnelshift_l(w1, w2, sh));
                    if (n_words > 3) atomicOr(dst + 3, __funnelshift_l(w2, w3, sh));
                    if (n_words > 4) atomicOr(dst + 4, __funnelshift_l(w3, 0u, sh));
                }
            }
        } else {
            four = false;
        }
        if (!four) {
            int64_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = codec_quantise(v[k], scale);
            codec_deltas(w, lane, cnt, carry);
            int total = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) total += k < left ? codec_len(codec_fold(w[k])) : 0;
            int32_t sum;
            uint8_t *dst = buf + fill + codec_scan<int32_t>(total, lane, &sum) - total;
            fill += sum;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                uint64_t u = codec_fold(w[k]);
                const int len = k < left ? codec_len(u) : 0;
                for (int g = 0; g < len; ++g, u >>= 5) *dst++ = (uint8_t)((g + 1 < len ? 0x20u : 0u) + ((uint32_t)u & 0x1fu) + 63u);
            }
        }
        const int32_t words = fill >> 4;
        __syncwarp();
        // whole words leave; the tail moves to the front of the buffer
        for (int32_t w = lane; w < words; w += 32) {
            if (w == 0 && skip > 0) {
                for (int k = skip; k < 16; ++k) base[k] = buf[k];
            } else {
                *reinterpret_cast<uint4 *>(base + 16 * w) = buf16[w];
            }
        }
        const int32_t tail = fill & 15;
        const uint8_t t = lane < tail ? buf[16 * words + lane] : 0;
        __syncwarp();
        if (lane < 16) buf[lane] = t;   // zeros behind the tail: the next chunk ors into this word
        if (words > 0) skip = 0;
        base += 16 * words;
        fill = tail;
        __syncwarp();
    }
    if (lane >= skip && lane < fill) base[lane] = buf[lane];
}

// status bit 2: a row does not hold exactly d well-formed values.
// 512 bytes per step, sixteen per lane (1,024: 15 % slower).  The lanes mark the bytes that end a value and write their positions, in
// order, to a list in shared memory; then the values are taken 32 at a time, one per lane, whatever their length: bytes from shared
// memory, delta, warp prefix sum, and a coalesced store.  (With the values assembled where their last byte happened to lie, less than
// half of the lanes had one, and a 128-byte step took 870 instructions.)
#define CODEC_WIN 512
#define CODEC_LANE (CODEC_WIN / 32)   /* bytes per lane and step */
// five bits of each byte, low byte first
__device__ __forceinline__ uint32_t codec_gather(uint32_t t)
{
    t &= 0x1f1f1f1fu;
    t = (t & 0x001f001fu) | ((t >> 3) & 0x03e003e0u);
    return (t & 0x3ffu) | ((t >> 6) & 0xffc00u);
}

__global__ void __launch_bounds__(256)
k_codec_decode(const uint8_t *__restrict__ in, int64_t in_bytes, const int64_t *__restrict__ offsets, int64_t rows, int32_t d, float scale32,
               double scale, float *__restrict__ x, int64_t ld, int *__restrict__ status)
{
    sat_grid_wait();
    __shared__ __align__(16) uint8_t wins[8][16 + CODEC_WIN + 16];   // the last 16 bytes of the window before, the window (63 subtracted)
    __shared__ uint16_t lists[8][CODEC_WIN];
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    const int64_t b0 = offsets[r], b1 = offsets[r + 1];
    // an offset pair that does not lie inside the byte buffer is a malformed row: flagged and skipped, never dereferenced
    if (b0 < 0 || b1 > in_bytes || b1 < b0) {
        if (lane == 0) atomicOr(status, 2);
        return;
    }
    uint8_t *win = wins[threadIdx.x >> 5] + 16;
    uint16_t *list = lists[threadIdx.x >> 5];
    float *row = x + r * ld;
    // windows start at 4-byte aligned addresses; a word that lies partly outside the row is put together from the row's own bytes
    const int64_t a0 = b0 - (int64_t)((uintptr_t)(in + b0) & 3u);
    const float inv32 = 1.f / scale32;
    int64_t q_run = 0;
    int32_t elem = 0, prev_end = (int32_t)(b0 - a0) - 1;   // position of the last byte of the value before, in the window's coordinates
    bool bad = false;
    for (int64_t pos = a0; pos < b1; pos += CODEC_WIN) {
        const uint8_t *src = in + pos;
        const int32_t n_in = b1 - pos < CODEC_WIN ? (int32_t)(b1 - pos) : CODEC_WIN, head = pos == a0 ? (int32_t)(b0 - a0) : 0;
        uint32_t raw[CODEC_LANE / 4], term = 0;
#pragma unroll
        for (int k = 0; k < CODEC_LANE / 4; ++k) {
            const int32_t p = CODEC_LANE * lane + 4 * k;
            // bit 7 of each byte: 63 <= byte, byte <= 126, byte < 95 (a terminator).  Bytes above 190 carry into their neighbour, but
            // they are outside the alphabet themselves and flag the row.
            uint32_t inside = 0x80808080u;
            if (p >= head && p + 3 < n_in) {
                raw[k] = *reinterpret_cast<const uint32_t *>(src + p);
            } else {
                raw[k] = 0x3f3f3f3fu;   // outside: no borrow into the row's bytes when 63 is subtracted
                inside = 0;
#pragma unroll 1
                for (int i = max(head - p, 0); i < min(n_in - p, 4); ++i) {
                    raw[k] ^= (0x3fu ^ (uint32_t)src[p + i]) << (8 * i);
                    inside |= 0x80u << (8 * i);
                }
            }
            const uint32_t alpha = (raw[k] + 0x41414141u) & ~(raw[k] + 0x01010101u);
            if ((alpha & inside) != inside) bad = true;
            const uint32_t t = ~(raw[k] + 0x21212121u) & inside;
            // the four flags as four bits
            term |= (((t >> 7) & 0x01010101u) * 0x01020408u >> 24 & 0xfu) << (4 * k);
        }
        // the tail of the window before, then this one
        uint32_t keep = 0;
        if (lane < 4) keep = reinterpret_cast<const uint32_t *>(win + CODEC_WIN - 16)[lane];
        __syncwarp();
        if (lane < 4) reinterpret_cast<uint32_t *>(win - 16)[lane] = keep;
#pragma unroll
        for (int k = 0; k < CODEC_LANE / 16; ++k)
            *reinterpret_cast<uint4 *>(win + CODEC_LANE * lane + 16 * k) = make_uint4(raw[4 * k] - 0x3f3f3f3fu, raw[4 * k + 1] - 0x3f3f3f3fu,
                                                                                      raw[4 * k + 2] - 0x3f3f3f3fu, raw[4 * k + 3] - 0x3f3f3f3fu);
        int32_t n_val;
        const int32_t mine = __popc(term);
        int32_t at = codec_scan<int32_t>(mine, lane, &n_val) - mine;
        for (uint32_t t = term; t; t &= t - 1) list[at++] = (uint16_t)(CODEC_LANE * lane + __ffs((int)t) - 1);
        __syncwarp();
        for (int32_t i0 = 0; i0 < n_val; i0 += 32) {
            const int32_t i = i0 + lane;
            const bool ok = i < n_val;
            const int32_t end = ok ? (int32_t)list[i] : 0;
            const int32_t before = __shfl_up_sync(0xffffffffu, end, 1);
            const int32_t groups = ok ? end - (lane == 0 ? prev_end : before) : 1;
            prev_end = __shfl_sync(0xffffffffu, end, min(31, n_val - 1 - i0));
            if (groups > CODEC_MAX_GROUPS) bad = true;   // longer than 64 bits
            float y;
            if (__all_sync(0xffffffffu, groups <= 4) && q_run > -(1 << 30) && q_run < (1 << 30)) {
                // the four bytes that end at `end`; at most 32 deltas below 2^19 on top of |q_run| < 2^30: no 32-bit overflow
                const int32_t first = end - 3;
                const uint32_t *wp = reinterpret_cast<const uint32_t *>(win + (first & ~3));
                const uint32_t v = codec_gather(__funnelshift_r(wp[0], wp[1], 8 * (first & 3)) >> (32 - 8 * groups));
                const int32_t e = ok ? (int32_t)((v >> 1) ^ (0u - (v & 1u))) : 0;
                int32_t sum;
                const int32_t q = (int32_t)q_run + codec_scan<int32_t>(e, lane, &sum);
                q_run = (int32_t)q_run + sum;
                if (__all_sync(0xffffffffu, q > -(1 << 24) && q < (1 << 24))) {
                    // q / 10^p, correctly rounded: product with the rounded reciprocal and one exact remainder step (Markstein);
                    // checked for every q and p of this range
                    const float f = (float)q, y0 = f * inv32;
                    y = fmaf(fmaf(-y0, scale32, f), inv32, y0);
                } else {
                    y = (float)((double)q / scale);
                }
            } else {
                uint64_t v = 0;
                for (int g = 0; g < groups && g < CODEC_MAX_GROUPS; ++g) v = (v << 5) | (win[end - g] & 0x1fu);
                const int64_t e = !ok ? 0 : (v & 1) ? ~(int64_t)(v >> 1) : (int64_t)(v >> 1);
                int64_t sum;
                const int64_t q = q_run + codec_scan<int64_t>(e, lane, &sum);
                q_run += sum;
                y = (float)((double)q / scale);
            }
            if (ok) {
                if (elem + i < d) row[elem + i] = y;
                else bad = true;
            }
        }
        elem += n_val;
        prev_end -= CODEC_WIN;
        __syncwarp();
    }
    // the last byte of the row must end a value, and the row must hold exactly d values
    if (lane == 0 && b1 > b0 && (uint32_t)in[b1 - 1] - 63u >= 0x20u) bad = true;
    if (elem != d) bad = true;
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, 2);
}

static double codec_scale(int32_t precision)
{
    double s = 1.0;
    for (int32_t i = 0; i < precision; ++i) s *= 10.0;
    return s;
}

static int codec_vec(const float *x, int32_t ld) { return aligned16(x) && !(ld & 3); }   // rows allow 16-byte loads

static sat_status codec_check(sat_ctx *ctx, const char *who, const void *x, int32_t ld, int64_t rows, int32_t d, int32_t precision)
{
    if (rows < 0 || d <= 0 || ld < d || precision < 0 || precision > 7 || (rows > 0 && !x))
        return sat_fail(ctx, SAT_EINVAL, "%s: null tensor, bad shape or precision outside 0..7", who);
    return SAT_OK;
}

// through pinned memory: a copy to pageable memory is staged by the driver
static sat_status codec_read_total(sat_ctx *ctx, const int64_t *dev, int64_t *host)
{
    int64_t *pinned = (int64_t *)(ctx->h_flag + 2);
    SAT_CUDA(ctx, cudaMemcpyAsync(pinned, dev, sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
    SAT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    *host = *pinned;
    return SAT_OK;
}

static sat_status codec_plan(sat_ctx *ctx, const float *x, int32_t ld, int64_t rows, int32_t d, int32_t precision, int64_t *row_offsets,
                             int64_t *total_bytes)
{
    SAT_TRY(sat_ensure(ctx, ctx->buf_codec_sizes, (size_t)(rows > 0 ? rows : 1) * sizeof(int32_t)));
    int32_t *sizes = (int32_t *)ctx->buf_codec_sizes.p;
    if (rows > 0) {
        ProfScope prof(ctx, SATK_CODEC, 4.0 * (double)rows * d + 12.0 * (double)rows, 0.0);
        sat_pdl(ctx->stream, k_codec_sizes, (unsigned)cdiv64(rows * 32, 256), 256, 0)(x, ld, rows, d, codec_vec(x, ld), (float)codec_scale(precision),
                                                                             codec_scale(precision), sizes);
        SAT_LAUNCHED(ctx);
    }
    SAT_TRY(sat_scan_i32(ctx, sizes, rows, row_offsets));
    if (total_bytes) {
        SAT_TRY(codec_read_total(ctx, row_offsets + rows, total_bytes));
    }
    return SAT_OK;
}

extern "C" sat_status sat_codec_plan(sat_ctx *ctx, const float *x, int32_t ld, int64_t rows, int32_t d, int32_t precision,
                                     int64_t *row_offsets, int64_t *total_bytes)
{
    CHECK_CTX(ctx);
    SAT_TRY(codec_check(ctx, "sat_codec_plan", x, ld, rows, d, precision));
    if (!row_offsets || !total_bytes) return sat_fail(ctx, SAT_EINVAL, "sat_codec_plan: null row_offsets / total_bytes");
    return codec_plan(ctx, x, ld, rows, d, precision, row_offsets, total_bytes);
}

static sat_status codec_encode(sat_ctx *ctx, const float *x, int32_t ld, int64_t rows, int32_t d, int32_t precision,
                               const int64_t *row_offsets, uint8_t *out, int64_t total)
{
    if (rows == 0) return SAT_OK;
    ProfScope prof(ctx, SATK_CODEC, 4.0 * (double)rows * d + 8.0 * (double)rows + (double)total, 0.0);
    sat_pdl(ctx->stream, k_codec_encode, (unsigned)cdiv64(rows * 32, 256), 256, 0)(x, ld, rows, d, codec_vec(x, ld), (float)codec_scale(precision), codec_scale(precision),
                                                                             row_offsets, out);
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

extern "C" sat_status sat_codec_encode(sat_ctx *ctx, const float *x, int32_t ld, int64_t rows, int32_t d, int32_t precision,
                                       const int64_t *row_offsets, uint8_t *out, int64_t out_capacity)
{
    CHECK_CTX(ctx);
    SAT_TRY(codec_check(ctx, "sat_codec_encode", x, ld, rows, d, precision));
    if (!row_offsets || out_capacity < 0 || (rows > 0 && !out)) return sat_fail(ctx, SAT_EINVAL, "sat_codec_encode: null row_offsets / out");
    int64_t total = 0;
    SAT_TRY(codec_read_total(ctx, row_offsets + rows, &total));
    if (total > out_capacity)
        return sat_fail(ctx, SAT_EINVAL, "sat_codec_encode: the rows need %lld bytes, the output holds %lld", (long long)total, (long long)out_capacity);
    return codec_encode(ctx, x, ld, rows, d, precision, row_offsets, out, total);
}

static sat_status codec_decode(sat_ctx *ctx, const uint8_t *in, int64_t in_bytes, const int64_t *row_offsets, int64_t rows, int32_t d,
                               int32_t precision, float *x, int32_t ld)
{
    if (rows == 0) return SAT_OK;
    ProfScope prof(ctx, SATK_CODEC, 4.0 * (double)rows * d + 8.0 * (double)rows + (double)in_bytes, 0.0);
    sat_pdl(ctx->stream, k_codec_decode, (unsigned)cdiv64(rows * 32, 256), 256, 0)(in, in_bytes, row_offsets, rows, d, (float)codec_scale(precision), codec_scale(precision), x, ld,
                                                                             ctx->d_flag + 1);
    SAT_LAUNCHED(ctx);
    return SAT_OK;
}

extern "C" sat_status sat_codec_decode(sat_ctx *ctx, const uint8_t *in, int64_t in_bytes, const int64_t *row_offsets, int64_t rows, int32_t d,
                                       int32_t precision, float *x, int32_t ld)
{
    CHECK_CTX(ctx);
    SAT_TRY(codec_check(ctx, "sat_codec_decode", x, ld, rows, d, precision));
    if (!row_offsets || in_bytes < 0 || (rows > 0 && in_bytes > 0 && !in)) return sat_fail(ctx, SAT_EINVAL, "sat_codec_decode: null row_offsets / in, or negative in_bytes");
    return codec_decode(ctx, in, in_bytes, row_offsets, rows, d, precision, x, ld);
}

// encode + decode of one matrix in place through context scratch (what a compressed ring would hand back)
sat_status sat_codec_roundtrip(sat_ctx *ctx, float *x, int32_t ld, int64_t rows, int32_t d, int32_t precision, int64_t *bytes)
{
    SAT_TRY(sat_ensure(ctx, ctx->buf_codec_off, (size_t)(rows + 1) * sizeof(int64_t)));
    int64_t *offsets = (int64_t *)ctx->buf_codec_off.p;
    int64_t total = 0;
    SAT_TRY(codec_plan(ctx, x, ld, rows, d, precision, offsets, &total));
    SAT_TRY(sat_ensure(ctx, ctx->buf_codec_bytes, (size_t)(total > 0 ? total : 1)));
    uint8_t *data = (uint8_t *)ctx->buf_codec_bytes.p;
    SAT_TRY(codec_encode(ctx, x, ld, rows, d, precision, offsets, data, total));
    SAT_TRY(codec_decode(ctx, data, total, offsets, rows, d, precision, x, ld));
    if (bytes) *bytes = total;
    return SAT_OK;
}
