// Attention of one new token over a compressed key/value cache (Section 1: the
// cache is what long-context decoding loads; Section 3: keys are stored before
// the rotary embedding; Section 2.2: a cached vector is the sum of its codewords
// times its deviation).  The decoded keys and values never reach global memory:
//   1. scores   s[t][h][j] = sum_c q[h J + j][c] * rot(k^[t][h])[c]        (att_scores_kernel)
//   2. maxima   m[h][j] = max_t scale * s[t][h][j]                          (att_max_kernel)
//   3. weights  w[t][h][j] = exp(scale s - m) times the value's deviation, and the sums of the weights
//                                                                          (att_weights_kernel)
//   4. values   acc[h][j][c] = sum_t w[t][h][j] * (codewords of v^[t][h])[c] (att_values_kernel)
//   5. out[h J + j][c] = acc / weights                                      (att_finish_kernel)
// Steps 1 and 4 are the table decoder's gather: a CTA keeps the float32 channels of one slice of
// four codeword elements for all codes and stages in shared memory (16 bytes per code and stage,
// stage order rotated by lane so that a quarter warp's reads never collide), a warp takes one
// token (its 32 lanes are the 8 kv heads x 4 groups, so a thread keeps one (head, group) for the
// whole launch and with it its query values and its output accumulators in registers), and the
// eight slices of a token are eight CTAs whose partial scores meet in global memory through
// float reductions.
#include "prepared.cuh"

namespace rvq {

namespace {

constexpr int kAttThreads = 1024;
constexpr int kAttSlices = 8;            // four codeword elements per slice
constexpr int kAttMaxK = 1792;           // 128 bytes per code: 224 KB of shared memory

// Codeword element at place i of slice sl.  Keys with half-split rotary pairs on strided groups
// keep two elements and their partners 16 elements on (channels 64 apart) in one slice.
template <int LAYOUT, int ROPE>
__device__ __forceinline__ int att_element(int sl, int i)
{
    if (ROPE == 1 && LAYOUT == RVQ_GROUP_STRIDED) return 2 * sl + (i & 1) + 16 * (i >> 1);
    return 4 * sl + i;
}
template <int LAYOUT>
__device__ __forceinline__ int att_channel(int g, int e)
{
    return LAYOUT == RVQ_GROUP_STRIDED ? 4 * e + g : 32 * g + e;
}

// table[code][8 slots] = the four float32 channels of this slice: stage r in slot r, and with up to four stages (STEPS
// 4) once more in slot r + 4, so that eight lanes still read eight bank groups in half the steps; absent stages are zero
template <int LAYOUT, int ROPE, int STEPS>
__device__ __forceinline__ void att_fill_table(const Shape &s, const float *__restrict__ cb, int sl, float4 *table)
{
    for (int t = threadIdx.x; t < s.K * 8; t += kAttThreads) {
        const int r = t & (STEPS - 1), j = t >> 3;
        float4 e = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (r < s.R) {
            const float *src = cb + ((size_t)r * s.K + j) * 32;
            if (ROPE == 1 && LAYOUT == RVQ_GROUP_STRIDED) {
                const float2 a = __ldg(reinterpret_cast<const float2 *>(src + 2 * sl));
                const float2 b = __ldg(reinterpret_cast<const float2 *>(src + 2 * sl + 16));
                e = make_float4(a.x, a.y, b.x, b.y);
            } else {
                e = __ldg(reinterpret_cast<const float4 *>(src + 4 * sl));
            }
        }
        table[t] = e;
    }
}

// Where the codes of this lane's group are in a head vector's words, and how they are cut out.
struct AttCodes {
    int form;                     // 0: eight 16-bit codes; 1: fewer of them; 2: packed codes
    uint32_t first, shift;        // word and bit of the group's first code
};
__device__ __forceinline__ AttCodes att_codes(const Shape &s, int g)
{
    AttCodes a;
    a.form = s.bits == 16 ? (s.R == 8 ? 0 : 1) : 2;           // (codes of 1792 values: at most 88 bits, and 31 before them)
    a.first = (uint32_t)(g * s.R * s.bits) >> 5;
    a.shift = (uint32_t)(g * s.R * s.bits) & 31u;
    return a;
}
// The words of a group row with its codes, as they are stored, and the deviation of its head vector.
struct AttRow {
    uint32_t c0, c1, c2, c3;
    uint16_t sd;
};
// Position of a token: the caller's, or the token's index.
__device__ __forceinline__ int att_position(const int32_t *__restrict__ position, uint32_t token, uint32_t tokens)
{
    if (token >= tokens) return 0;
    return position ? __ldg(position + token) : (int)token;
}
__device__ __forceinline__ void att_fetch(const Shape &s, const AttCodes &ac, const void *__restrict__ codes,
                                          const uint16_t *__restrict__ std16, uint32_t token, uint32_t tokens, int lane,
                                          AttRow &a)
{
    a.c0 = a.c1 = a.c2 = a.c3 = 0u;
    a.sd = 0;
    if (token >= tokens) return;
    const uint32_t v = token * 8u + (uint32_t)(lane >> 2);    // (the launcher keeps tokens * 32 below 2^31)
    const int g = lane & 3;
    a.sd = __ldg(std16 + v);
    if (ac.form == 0) {
        const uint4 c = __ldg(reinterpret_cast<const uint4 *>(codes) + (v * 4u + (uint32_t)g));
        a.c0 = c.x; a.c1 = c.y; a.c2 = c.z; a.c3 = c.w;
        return;
    }
    const uint8_t *vec = reinterpret_cast<const uint8_t *>(codes) + (size_t)v * s.code_bytes;
    const uint32_t *words = reinterpret_cast<const uint32_t *>(vec) + ac.first;
    const uint32_t left = (uint32_t)s.code_bytes / 4u - ac.first;
    a.c0 = __ldg(words);
    if (left > 1) a.c1 = __ldg(words + 1);
    if (left > 2) a.c2 = __ldg(words + 2);
    if (left > 3) a.c3 = __ldg(words + 3);
}

// The codes of a row as four words, stage r in half r, absent stages 0.
__device__ __forceinline__ void att_cut(const Shape &s, const AttCodes &ac, AttRow &a)
{
    if (ac.form == 0) return;
    uint32_t w0 = __funnelshift_r(a.c0, a.c1, ac.shift), w1 = __funnelshift_r(a.c1, a.c2, ac.shift);
    uint32_t w2 = __funnelshift_r(a.c2, a.c3, ac.shift), w3 = a.c3 >> ac.shift;
    if (ac.form == 2) {
        // two codes from the low end at a time, then the window moves on by two codes
        const uint32_t mask = (1u << s.bits) - 1u, up = 16u - (uint32_t)s.bits, two = 2u * (uint32_t)s.bits;
        auto halves = [&](uint32_t w) { return (w & mask) | ((w << up) & (mask << 16)); };
        a.c0 = halves(w0);
        w0 = __funnelshift_r(w0, w1, two); w1 = __funnelshift_r(w1, w2, two); w2 = __funnelshift_r(w2, w3, two);
        a.c1 = halves(w0);
        w0 = __funnelshift_r(w0, w1, two); w1 = __funnelshift_r(w1, w2, two);
        a.c2 = halves(w0);
        w0 = __funnelshift_r(w0, w1, two);
        a.c3 = halves(w0);
    } else {
        a.c0 = w0; a.c1 = w1; a.c2 = w2; a.c3 = w3;
    }
    auto keep = [&](uint32_t &w, int r) { w = s.R > r + 1 ? w : s.R > r ? w & 0xFFFFu : 0u; };
    keep(a.c0, 0); keep(a.c1, 2); keep(a.c2, 4); keep(a.c3, 6);
}

// Sum over the stages of the four channels of this thread's row: STEPS 16-byte reads, stage
// rot ^ k (its last two bits with four steps) at step k.  (With stage rot + k, eight operations more, and two more per step for its address, the
// call over 131072 tokens takes 466 us instead of 438.)  PACKED: two additions per instruction -- us of the kernel, single / packed, scores 267 / 260, with four steps 114 / 107
// (60000 tokens); values 187 / 191 (register pairs cost moves), with four steps 72 / 67.  Codes past the codebook are read as code 0 and counted.
template <int STEPS, bool PACKED>
__device__ __forceinline__ void att_gather(const AttRow &a, uint32_t K, uint32_t rot, uint32_t smem_table,
                                           float (&acc)[4], uint32_t &bad)
{
    uint32_t c0 = a.c0, c1 = a.c1, c2 = a.c2, c3 = a.c3;
    {
        const uint32_t m = __vmaxu2(__vmaxu2(c0, c1), __vmaxu2(c2, c3));
        if (max(m & 0xFFFFu, m >> 16) >= K) {
            uint32_t *cc[4] = {&c0, &c1, &c2, &c3};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t lo = *cc[c] & 0xFFFFu, hi = *cc[c] >> 16;
                if (lo >= K) { lo = 0; ++bad; }
                if (hi >= K) { hi = 0; ++bad; }
                *cc[c] = lo | (hi << 16);
            }
        }
    }
    exchange_codes<STEPS>(rot, c0, c1, c2, c3);
    const uint32_t cw[4] = {c0, c1, c2, c3};
    uint64_t s01 = 0, s23 = 0;
    acc[0] = acc[1] = acc[2] = acc[3] = 0.0f;
#pragma unroll
    for (int k = 0; k < STEPS; ++k) {
        const uint32_t w = cw[k >> 1], code = (k & 1) ? w >> 16 : w & 0xFFFFu;
        const uint32_t slot = STEPS == 8 ? rot ^ k : ((rot ^ k) & 3u) | (rot & 4u);
        const uint32_t addr = code * 128u + (smem_table + slot * 16u);
        if (PACKED) {
            uint64_t f01, f23;
            asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(f01), "=l"(f23) : "r"(addr));
            s01 = k == 0 ? f01 : add_f32x2(s01, f01);
            s23 = k == 0 ? f23 : add_f32x2(s23, f23);
        } else {
            float f0, f1, f2, f3;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(f0), "=f"(f1), "=f"(f2), "=f"(f3) : "r"(addr));
            acc[0] += f0; acc[1] += f1; acc[2] += f2; acc[3] += f3;
        }
    }
    if (PACKED) {
        acc[0] = __uint_as_float((uint32_t)s01); acc[1] = __uint_as_float((uint32_t)(s01 >> 32));
        acc[2] = __uint_as_float((uint32_t)s23); acc[3] = __uint_as_float((uint32_t)(s23 >> 32));
    }
}

// (cos, sin) of the rotary pairs of this thread's four channels at position `pos`:
// c[i], s[i] belong to place i (half-split pairs on strided groups and adjacent pairs on
// contiguous groups have two pairs in the thread: places 0 and 1 of c, s).
template <int LAYOUT, int ROPE>
__device__ __forceinline__ void att_cos_sin(const float2 *__restrict__ cos_sin, int positions, int pos, int sl, int g,
                                            float (&c)[4], float (&sn)[4])
{
    c[0] = c[1] = c[2] = c[3] = 1.0f;
    sn[0] = sn[1] = sn[2] = sn[3] = 0.0f;
    if (ROPE == 0) return;
    const float2 *cs = cos_sin + (size_t)min(max(pos, 0), positions - 1) * 64;
    if (ROPE == 1 && LAYOUT == RVQ_GROUP_STRIDED) {
        // places (0, 2) and (1, 3): channels 4 (2 sl + i) + g and 64 further on; that channel is the pair
#pragma unroll
        for (int i = 0; i < 2; ++i) { const float2 t = __ldg(cs + 4 * (2 * sl + i) + g); c[i] = t.x; sn[i] = t.y; }
    } else if (ROPE == 2 && LAYOUT == RVQ_GROUP_CONTIGUOUS) {
        // channels 32 g + 4 sl + i: pairs 16 g + 2 sl + i / 2, both halves in the thread
        const float4 t = __ldg(reinterpret_cast<const float4 *>(cs + 16 * g + 2 * sl));
        c[0] = t.x; sn[0] = t.y; c[1] = t.z; sn[1] = t.w;
    } else if (ROPE == 1) {
        // contiguous groups: channel 32 g + 4 sl + i and its partner in group g ^ 2; pairs 32 (g & 1) + 4 sl + i
        const float4 *p = reinterpret_cast<const float4 *>(cs + 32 * (g & 1) + 4 * sl);
        const float4 a = __ldg(p), b = __ldg(p + 1);
        c[0] = a.x; sn[0] = a.y; c[1] = a.z; sn[1] = a.w; c[2] = b.x; sn[2] = b.y; c[3] = b.z; sn[3] = b.w;
    } else {
        // strided groups, pairs (2k, 2k + 1): channels 4 e + g and 4 e + (g ^ 1), e = 4 sl + i; pair 2 e + g / 2
#pragma unroll
        for (int i = 0; i < 4; ++i) { const float2 t = __ldg(cs + 2 * (4 * sl + i) + (g >> 1)); c[i] = t.x; sn[i] = t.y; }
    }
}

// Step 1.  ROPE 0: keys as stored; 1: pairs (k, k + 64); 2: pairs (2k, 2k + 1).
template <int LAYOUT, int ROPE, int J, int STEPS>
__global__ void __launch_bounds__(kAttThreads, 1)
att_scores_kernel(Shape s, const void *__restrict__ codes, const uint16_t *__restrict__ std16, int64_t tokens,
                  const float *__restrict__ cb, const float *__restrict__ q, const int32_t *__restrict__ position,
                  const float2 *__restrict__ cos_sin, int positions, float *__restrict__ scores, rvq_status *st)
{
    asm volatile("griddepcontrol.launch_dependents;");
    extern __shared__ __align__(128) uint8_t smem[];
    const int parts = gridDim.x / kAttSlices;
    if ((int)blockIdx.x >= parts * kAttSlices) return;
    const int sl = blockIdx.x % kAttSlices, part = blockIdx.x / kAttSlices;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, h = lane >> 2, g = lane & 3;
    att_fill_table<LAYOUT, ROPE, STEPS>(s, cb, sl, reinterpret_cast<float4 *>(smem));
    // the query values that meet this thread's four channels, for the J query heads of its kv head
    float qr[J][4];
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            qr[j][i] = __ldg(q + (size_t)(h * J + j) * 128 + att_channel<LAYOUT>(g, att_element<LAYOUT, ROPE>(sl, i)));
    __syncthreads();
    const uint32_t smem_table = (uint32_t)__cvta_generic_to_shared(smem);
    uint32_t bad = 0;
    // Loads run ahead of their use: the codes, the deviation and the (cos, sin) values of the next token
    // are asked for while this one is gathered, and the position of the token after that (the address
    // of the (cos, sin) values hangs on it).
    const uint32_t T = (uint32_t)tokens, step = (uint32_t)parts * 32u, t0 = (uint32_t)part * 32u + (uint32_t)warp;
    const AttCodes ac = att_codes(s, lane & 3);
    AttRow next;
    float cn[4], sn[4];
    att_fetch(s, ac, codes, std16, t0, T, lane, next);
    att_cos_sin<LAYOUT, ROPE>(cos_sin, positions, att_position(position, t0, T), sl, g, cn, sn);
    int pos_next = ROPE != 0 ? att_position(position, t0 + step, T) : 0;
    for (uint32_t t = t0; t < T; t += step) {
        AttRow cur = next;
        float cc[4], ss[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { cc[i] = cn[i]; ss[i] = sn[i]; }
        att_cos_sin<LAYOUT, ROPE>(cos_sin, positions, pos_next, sl, g, cn, sn);
        if (ROPE != 0) pos_next = att_position(position, t + 2 * step, T);
        att_fetch(s, ac, codes, std16, t + step, T, lane, next);
        float v[4];
        att_cut(s, ac, cur);
        att_gather<STEPS, true>(cur, (uint32_t)s.K, (uint32_t)lane & 7u, smem_table, v, bad);
        const float sd = __half2float(__ushort_as_half(cur.sd));
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] *= sd;
        if (ROPE != 0) {
            if (ROPE == 1 && LAYOUT == RVQ_GROUP_STRIDED) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float a = v[i], b = v[i + 2];
                    v[i] = a * cc[i] - b * ss[i];
                    v[i + 2] = b * cc[i] + a * ss[i];
                }
            } else if (ROPE == 2 && LAYOUT == RVQ_GROUP_CONTIGUOUS) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float a = v[2 * i], b = v[2 * i + 1];
                    v[2 * i] = a * cc[i] - b * ss[i];
                    v[2 * i + 1] = b * cc[i] + a * ss[i];
                }
            } else {
                // the partner is the same place of group g ^ 2 (half-split pairs) or g ^ 1 (adjacent pairs)
                const int other = ROPE == 1 ? 2 : 1;
                const bool first = (g & other) == 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float o = __shfl_xor_sync(0xFFFFFFFFu, v[i], other);
                    v[i] = first ? v[i] * cc[i] - o * ss[i] : v[i] * cc[i] + o * ss[i];
                }
            }
        }
        float part_s[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            float a = v[0] * qr[j][0];
            a = fmaf(v[1], qr[j][1], a);
            a = fmaf(v[2], qr[j][2], a);
            a = fmaf(v[3], qr[j][3], a);
            part_s[j] = a;
        }
        // the sums over the four groups are shared out: lane g ends with query head g (with two heads: g & 1), so that a
        // warp's reductions are consecutive floats
        float total;
        if (J == 4) {
            const float keep0 = (g & 1) ? part_s[1 % J] : part_s[0], keep1 = (g & 1) ? part_s[3 % J] : part_s[2 % J];
            const float send0 = (g & 1) ? part_s[0] : part_s[1 % J], send1 = (g & 1) ? part_s[2 % J] : part_s[3 % J];
            const float pair0 = keep0 + __shfl_xor_sync(0xFFFFFFFFu, send0, 1), pair1 = keep1 + __shfl_xor_sync(0xFFFFFFFFu, send1, 1);
            total = ((g & 2) ? pair1 : pair0) + __shfl_xor_sync(0xFFFFFFFFu, (g & 2) ? pair0 : pair1, 2);
        } else {
            total = J == 2 && (g & 1) ? part_s[J - 1] : part_s[0];
            total += __shfl_xor_sync(0xFFFFFFFFu, J == 2 && !(g & 1) ? part_s[J - 1] : part_s[0], 1);
            total += __shfl_xor_sync(0xFFFFFFFFu, total, 2);
        }
        if (g < J) atomicAdd(scores + (size_t)(t * 8u + (uint32_t)h) * J + g, total);
    }
    if (bad && st && sl == 0) atomicAdd(&st->bad_codes, bad);
}

// order-preserving map of a float onto unsigned integers (0 is below every float)
__device__ __forceinline__ uint32_t att_ordered(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float att_unordered(uint32_t u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

// Steps 2 and 3 take four columns per thread; the lanes and warps that have the same four meet here.  `columns` = 8 J: 8, 16 or 32.
template <typename F>
__device__ __forceinline__ void att_reduce_columns(float (&v)[4], int columns, float (*part)[32], F join)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, fours = columns / 4;
    for (int off = 16; off >= fours; off >>= 1)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = join(v[i], __shfl_xor_sync(0xFFFFFFFFu, v[i], off));
    if (lane < fours) *reinterpret_cast<float4 *>(&part[warp][4 * lane]) = make_float4(v[0], v[1], v[2], v[3]);
    __syncthreads();
}

// Step 2: m[column] = max over the tokens of scale * s[token][column].  (Four columns per thread and load, here and in step 3, one block per SM: the whole call over 131072 tokens 470 -> 466 us, 60000 235.4 -> 233.0;
// one column, two blocks per SM before; two blocks with four columns 466.6 and 234.2.)
__global__ void __launch_bounds__(kAttThreads)
att_max_kernel(const float *scores, int64_t tokens, int columns, float scale, uint32_t *m_ord)
{
    follow_previous();
    __shared__ __align__(16) float part[kAttThreads / 32][32];
    const int64_t all = tokens * (columns / 4), step = (int64_t)gridDim.x * kAttThreads;        // (a multiple of columns / 4)
    const float4 *s4 = reinterpret_cast<const float4 *>(scores);
    float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 4
    for (int64_t k = (int64_t)blockIdx.x * kAttThreads + threadIdx.x; k < all; k += step) {
        const float4 f = s4[k];
        m[0] = fmaxf(m[0], scale * f.x); m[1] = fmaxf(m[1], scale * f.y); m[2] = fmaxf(m[2], scale * f.z); m[3] = fmaxf(m[3], scale * f.w);
    }
    att_reduce_columns(m, columns, part, [](float a, float b) { return fmaxf(a, b); });
    if ((int)threadIdx.x < columns) {
        float top = part[0][threadIdx.x];
        for (int w = 1; w < kAttThreads / 32; ++w) top = fmaxf(top, part[w][threadIdx.x]);
        if (top > -INFINITY) atomicMax(m_ord + threadIdx.x, att_ordered(top));
    }
}

// Step 3: every score becomes its weight times its token's deviation, exp(scale s - m) = 2^(s * scale log2(e) -
// m log2(e)), and the weights are summed; once per token here instead of in each of the 32 rows and slices of step 4.
__global__ void __launch_bounds__(kAttThreads)
att_weights_kernel(float *scores, const uint16_t *__restrict__ std16, uint32_t tokens, int columns, int per_head_log,
                   float scale, const uint32_t *m_ord, float *weight_sum)
{
    follow_previous();
    __shared__ __align__(16) float part[kAttThreads / 32][32];
    constexpr float kLog2e = 1.4426950408889634f;
    const int fours = columns / 4, col = 4 * ((int)threadIdx.x % fours), fours_log = __ffs(fours) - 1;
    const float sl2 = scale * kLog2e;
    float mneg[4], sum[4] = {};
#pragma unroll
    for (int i = 0; i < 4; ++i) mneg[i] = -att_unordered(m_ord[col + i]) * kLog2e;
    const int64_t all = (int64_t)tokens * fours, step = (int64_t)gridDim.x * kAttThreads;
    float4 *s4 = reinterpret_cast<float4 *>(scores);
#pragma unroll 4
    for (int64_t k = (int64_t)blockIdx.x * kAttThreads + threadIdx.x; k < all; k += step) {
        const float4 f = s4[k];
        const uint16_t *sd = std16 + (size_t)(k >> fours_log) * 8;
        float w[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            w[i] = exp2f(fmaf(w[i], sl2, mneg[i]));
            sum[i] += w[i];
            w[i] *= __half2float(__ushort_as_half(__ldg(sd + ((col + i) >> per_head_log))));
        }
        s4[k] = make_float4(w[0], w[1], w[2], w[3]);
    }
    att_reduce_columns(sum, columns, part, [](float a, float b) { return a + b; });
    if ((int)threadIdx.x < columns) {
        float total = part[0][threadIdx.x];
        for (int w = 1; w < kAttThreads / 32; ++w) total += part[w][threadIdx.x];
        atomicAdd(weight_sum + threadIdx.x, total);
    }
}

// Step 4.
template <int LAYOUT, int J, int STEPS>
__global__ void __launch_bounds__(kAttThreads, 1)
att_values_kernel(Shape s, const void *__restrict__ codes, const uint16_t *__restrict__ std16, int64_t tokens,
                  const float *__restrict__ cb, const float *weights, float *out_acc, rvq_status *st)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const int parts = gridDim.x / kAttSlices;
    if ((int)blockIdx.x >= parts * kAttSlices) return;
    const int sl = blockIdx.x % kAttSlices, part = blockIdx.x / kAttSlices;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, h = lane >> 2;
    // (the table does not hang on the weights: it is filled while they are made)
    att_fill_table<LAYOUT, 0, STEPS>(s, cb, sl, reinterpret_cast<float4 *>(smem));
    follow_previous();
    __syncthreads();
    const uint32_t smem_table = (uint32_t)__cvta_generic_to_shared(smem);
    uint32_t bad = 0;
    float acc[J][4];
#pragma unroll
    for (int j = 0; j < J; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;
    const uint32_t T = (uint32_t)tokens, step = (uint32_t)parts * 32u;
    const AttCodes ac = att_codes(s, lane & 3);
    AttRow next;
    att_fetch(s, ac, codes, std16, (uint32_t)part * 32u + (uint32_t)warp, T, lane, next);
    for (uint32_t t = (uint32_t)part * 32u + (uint32_t)warp; t < T; t += step) {
        AttRow cur = next;
        // this token's weights, asked for before the gather
        float sc[J];
        {
            const float *src = weights + (size_t)(t * 8u + (uint32_t)h) * J;
            if (J == 4) { const float4 f = *reinterpret_cast<const float4 *>(src); sc[0] = f.x; sc[1] = f.y; sc[J - 2] = f.z; sc[J - 1] = f.w; }
            else if (J == 2) { const float2 f = *reinterpret_cast<const float2 *>(src); sc[0] = f.x; sc[J - 1] = f.y; }
            else sc[0] = *src;
        }
        att_fetch(s, ac, codes, std16, t + step, T, lane, next);
        float v[4];
        att_cut(s, ac, cur);
        att_gather<STEPS, STEPS == 4>(cur, (uint32_t)s.K, (uint32_t)lane & 7u, smem_table, v, bad);
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[j][i] = fmaf(sc[j], v[i], acc[j][i]);
    }
    // sums over the CTA's warps (a lane is the same (head, group) in all of them), then one
    // reduction per value into global memory; the table's memory is free now
    __syncthreads();
    float *red = reinterpret_cast<float *>(smem);            // [4 J][32 warps][32 lanes]
#pragma unroll
    for (int j = 0; j < J; ++j) {
#pragma unroll
        for (int i = 0; i < 4; ++i) red[((j * 4 + i) * 32 + warp) * 32 + lane] = acc[j][i];
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < 4 * J * 32; idx += kAttThreads) {
        const int ln = idx & 31, what = idx >> 5, j = what / 4, i = what % 4;
        float a = 0.0f;
        for (int w = 0; w < 32; ++w) a += red[(what * 32 + w) * 32 + ln];
        const int hh = ln >> 2, gg = ln & 3;
        atomicAdd(out_acc + (size_t)(hh * J + j) * 128 + att_channel<LAYOUT>(gg, 4 * sl + i), a);
    }
    if (bad && st && sl == 0) atomicAdd(&st->bad_codes, bad);
}

// Step 5.
__global__ void att_finish_kernel(const float *out_acc, const float *weight_sum, int heads,
                                  float *out)
{
    follow_previous();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < heads * 128) out[idx] = out_acc[idx] / weight_sum[idx >> 7];
}

// Short caches: one pass over the tokens, codewords straight from L2 (as in decode_direct.cu), the softmax carried
// along, instead of tables that take longer to fill than the few tokens to read (two tables, five launches:
// 35 us for 1000 tokens).  A CTA takes one kv head and a chunk of tokens, a warp one token at a time: lane =
// (group, four-element piece), the key's and the value's sixteen 16-byte loads in flight together; the J
// dot products are reduced so that lanes of row group `rho` end with query head j(rho), which keeps its running
// maximum and weight sum.  The warps' partial outputs meet in shared memory, the chunks' in att_combine_kernel.
// What bounds it: the chain codes -> codewords -> score -> weight of a warp's few tokens, then L2 (8 KB per token
// and kv head), which is why long caches keep the tables.
constexpr int kShortThreads = 256, kShortWarps = kShortThreads / 32;
constexpr int kShortMaxChunks = 37;      // two CTAs per SM, over the 8 kv heads

// Code number k of vector v as it is stored; nothing here waits for it.
__device__ __forceinline__ uint32_t att_raw_code(const Shape &s, const void *__restrict__ codes, uint32_t v, uint32_t k)
{
    const uint8_t *vec = reinterpret_cast<const uint8_t *>(codes) + (size_t)v * (uint32_t)s.code_bytes;
    if (s.bits == 16) return __ldg(reinterpret_cast<const uint16_t *>(vec) + k);
    const uint32_t o = k * (uint32_t)s.bits, sh = o & 31u;
    const uint32_t *p = reinterpret_cast<const uint32_t *>(vec) + (o >> 5);
    return __funnelshift_r(__ldg(p), sh + s.bits > 32u ? __ldg(p + 1) : 0u, sh) & ((1u << s.bits) - 1u);
}

// The codewords of four group rows: lane (row, stage = piece) has the row's code of that stage.
template <int DEPTH>
__device__ __forceinline__ void att_load_codewords(const Shape &s, const float *__restrict__ cb, uint32_t code, uint32_t lane,
                                                   uint64_t (&lo)[8], uint64_t (&hi)[8], uint32_t &bad)
{
    if (code >= (uint32_t)s.K) { code = 0; ++bad; }
    const uint32_t off = ((lane & 7u) * (uint32_t)s.K + code) * 128u;
    const uint8_t *piece = reinterpret_cast<const uint8_t *>(cb) + (lane & 7u) * 16u;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const uint32_t at = __shfl_sync(0xFFFFFFFFu, off, (lane & 24u) | r);
        if (DEPTH == 0) lo[r] = hi[r] = 0ull;
        if (DEPTH ? r < DEPTH : r < s.R) asm volatile("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(lo[r]), "=l"(hi[r]) : "l"(piece + at));
    }
}

template <int DEPTH>
__device__ __forceinline__ void att_sum_codewords(const uint64_t (&lo)[8], const uint64_t (&hi)[8], float sd, float (&o)[4])
{
    uint64_t a = lo[0], b = hi[0];
#pragma unroll
    for (int r = 1; r < (DEPTH ? DEPTH : 8); ++r) { a = add_f32x2(a, lo[r]); b = add_f32x2(b, hi[r]); }
    o[0] = __uint_as_float((uint32_t)a) * sd; o[1] = __uint_as_float((uint32_t)(a >> 32)) * sd;
    o[2] = __uint_as_float((uint32_t)b) * sd; o[3] = __uint_as_float((uint32_t)(b >> 32)) * sd;
}

template <int ROPE, int J, int DEPTH>                                 // DEPTH: of both, or 0 for any
__global__ void __launch_bounds__(kShortThreads, 2)
att_short_kernel(Shape sk, Shape sv, const float *__restrict__ q, const void *__restrict__ codes_k, const uint16_t *__restrict__ std_k,
                 const void *__restrict__ codes_v, const uint16_t *__restrict__ std_v, uint32_t tokens, const float *__restrict__ cb_k,
                 const float *__restrict__ cb_v, const int32_t *__restrict__ position, const float2 *__restrict__ cos_sin, int positions,
                 float scale_log2e, float *__restrict__ part, float2 *__restrict__ part_ml, rvq_status *st)
{
    __shared__ __align__(16) float acc_s[kShortWarps][J][128];         // [group * 32 + element]
    __shared__ float2 ml_s[kShortWarps][J];
    asm volatile("griddepcontrol.launch_dependents;");
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 3, piece = lane & 7;
    const uint32_t h = blockIdx.y, chunks = gridDim.x, chunk = blockIdx.x;
    const bool strided = sk.layout == RVQ_GROUP_STRIDED;
    const uint32_t per = (tokens + chunks - 1) / chunks, first = chunk * per, last = min(tokens, first + per);
    float qr[J][4];
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t e = 4 * piece + i;
            qr[j][i] = __ldg(q + (size_t)(h * J + j) * 128 + (strided ? 4 * e + g : 32 * g + e));
        }
    const uint32_t my_j = J == 4 ? g : J == 2 ? g >> 1 : 0;
    float m = -INFINITY, l = 0.0f, acc[J][4] = {};
    uint32_t bad = 0;
    uint32_t t = first + warp;
    uint32_t code_k = 0, code_v = 0;
    uint16_t sdk = 0, sdv = 0;
    int pos = 0;
    auto fetch = [&](uint32_t at) {
        const uint32_t v = at * 8u + h;
        if ((int)piece < (DEPTH ? DEPTH : sk.R)) code_k = att_raw_code(sk, codes_k, v, g * sk.R + piece);
        if ((int)piece < (DEPTH ? DEPTH : sv.R)) code_v = att_raw_code(sv, codes_v, v, g * sv.R + piece);
        sdk = __ldg(std_k + v);
        sdv = __ldg(std_v + v);
        if (ROPE != 0) pos = position ? __ldg(position + at) : (int)at;
    };
    if (t < last) fetch(t);
    for (; t < last; t += kShortWarps) {
        uint64_t klo[8], khi[8], vlo[8], vhi[8];
        att_load_codewords<DEPTH>(sk, cb_k, code_k, lane, klo, khi, bad);
        float2 cs[4];
        if (ROPE != 0) {
            const float2 *row = cos_sin + (size_t)min(max(pos, 0), positions - 1) * 64;
#pragma unroll
            for (uint32_t i = 0; i < 4; ++i) {
                const uint32_t e = 4 * piece + i, c = strided ? 4 * e + g : 32 * g + e;
                cs[i] = __ldg(row + (ROPE == 1 ? c & 63u : c >> 1));
            }
        }
        att_load_codewords<DEPTH>(sv, cb_v, code_v, lane, vlo, vhi, bad);
        const float fk = __half2float(__ushort_as_half(sdk)), fv = __half2float(__ushort_as_half(sdv));
        if (t + kShortWarps < last) fetch(t + kShortWarps);
        float o[4];
        att_sum_codewords<DEPTH>(klo, khi, fk, o);
        if (ROPE == 2 && !strided) {
#pragma unroll
            for (int i = 0; i < 4; i += 2) {
                const float a = o[i], b = o[i + 1];
                o[i] = a * cs[i].x - b * cs[i].y;
                o[i + 1] = b * cs[i].x + a * cs[i].y;
            }
        } else if (ROPE != 0) {
            // the other channel of the pair: group g ^ 2, group g ^ 1, or (half-split pairs, strided groups) 16 elements on
            const uint32_t other = ROPE == 2 ? 8 : strided ? 4 : 16;
            const bool low = (lane & other) == 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float p = __shfl_xor_sync(0xFFFFFFFFu, o[i], other);
                o[i] = low ? o[i] * cs[i].x - p * cs[i].y : o[i] * cs[i].x + p * cs[i].y;
            }
        }
        float p[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            p[j] = o[0] * qr[j][0];
#pragma unroll
            for (int i = 1; i < 4; ++i) p[j] = fmaf(o[i], qr[j][i], p[j]);
        }
        // sums over the warp, half of the query heads going to each half of the lanes, then to each quarter
        float sc;
        if (J == 4) {
            const bool up = (lane & 16) != 0, up2 = (lane & 8) != 0;
            float a = up ? p[J - 2] : p[0], b = up ? p[J - 1] : p[J > 1 ? 1 : 0];
            a += __shfl_xor_sync(0xFFFFFFFFu, up ? p[0] : p[J - 2], 16);
            b += __shfl_xor_sync(0xFFFFFFFFu, up ? p[J > 1 ? 1 : 0] : p[J - 1], 16);
            sc = up2 ? b : a;
            sc += __shfl_xor_sync(0xFFFFFFFFu, up2 ? a : b, 8);
        } else if (J == 2) {
            const bool up = (lane & 16) != 0;
            sc = up ? p[J - 1] : p[0];
            sc += __shfl_xor_sync(0xFFFFFFFFu, up ? p[0] : p[J - 1], 16);
            sc += __shfl_xor_sync(0xFFFFFFFFu, sc, 8);
        } else {
            sc = p[0] + __shfl_xor_sync(0xFFFFFFFFu, p[0], 16);
            sc += __shfl_xor_sync(0xFFFFFFFFu, sc, 8);
        }
#pragma unroll
        for (int x = 4; x > 0; x >>= 1) sc += __shfl_xor_sync(0xFFFFFFFFu, sc, x);
        sc *= scale_log2e;
        // (the first token: exp2(-inf) = 0; while no score is above -inf, so is every token's weight)
        const float m2 = fmaxf(m, sc), top = m2 == -INFINITY ? 0.0f : m2, corr = exp2f(m - top), w = exp2f(sc - top);
        const bool moved = m2 != m;
        l = fmaf(l, corr, w);
        m = m2;
        att_sum_codewords<DEPTH>(vlo, vhi, fv, o);
        if (__any_sync(0xFFFFFFFFu, moved)) {
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float c = __shfl_sync(0xFFFFFFFFu, corr, J == 4 ? 8 * j : J == 2 ? 16 * j : 0);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[j][i] *= c;
            }
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const float wj = __shfl_sync(0xFFFFFFFFu, w, J == 4 ? 8 * j : J == 2 ? 16 * j : 0);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[j][i] = fmaf(wj, o[i], acc[j][i]);
        }
    }
    // the warps' parts
#pragma unroll
    for (int j = 0; j < J; ++j)
        *reinterpret_cast<float4 *>(&acc_s[warp][j][4 * lane]) = make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
    if ((lane & (J == 4 ? 7u : J == 2 ? 15u : 31u)) == 0) ml_s[warp][my_j] = make_float2(m, l);
    __syncthreads();
    for (uint32_t idx = threadIdx.x; idx < J * 128; idx += kShortThreads) {
        const uint32_t j = idx >> 7, c = idx & 127;
        float top = -INFINITY, sum = 0.0f, a = 0.0f;
#pragma unroll
        for (int w = 0; w < kShortWarps; ++w) top = fmaxf(top, ml_s[w][j].x);
#pragma unroll
        for (int w = 0; w < kShortWarps; ++w) {
            const float f = ml_s[w][j].x == -INFINITY ? 0.0f : exp2f(ml_s[w][j].x - top);
            sum = fmaf(f, ml_s[w][j].y, sum);
            a = fmaf(f, acc_s[w][j][c], a);
        }
        part[((size_t)(h * J + j) * chunks + chunk) * 128 + c] = a;
        if (c == 0) part_ml[(size_t)(h * J + j) * chunks + chunk] = make_float2(top, sum);
    }
    if (bad && st) atomicAdd(&st->bad_codes, bad);
}

// One CTA per query head: the chunks' parts, weighted to their common maximum, over the sum of all weights.
__global__ void __launch_bounds__(128)
att_combine_kernel(const float *part, const float2 *part_ml, int chunks, int layout_v, float *out)
{
    __shared__ float2 ml_s[kShortMaxChunks];
    __shared__ float f_s[kShortMaxChunks];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int head = blockIdx.x, c = threadIdx.x;
    // (all parts asked for together, before the maxima that weigh them are known: after them 3000 tokens took 24.7 us a call instead of 22.9, 9000 50.2 instead of 49.7)
    float v[kShortMaxChunks];
#pragma unroll
    for (int k = 0; k < kShortMaxChunks; ++k) v[k] = k < chunks ? __ldcg(part + ((size_t)head * chunks + k) * 128 + c) : 0.0f;
    if (c < kShortMaxChunks) ml_s[c] = c < chunks ? part_ml[head * chunks + c] : make_float2(-INFINITY, 0.0f);
    __syncthreads();
    float top = -INFINITY, sum = 0.0f, a = 0.0f;
#pragma unroll
    for (int k = 0; k < kShortMaxChunks; ++k) top = fmaxf(top, ml_s[k].x);
    if (c < chunks) f_s[c] = ml_s[c].x == -INFINITY ? 0.0f : exp2f(ml_s[c].x - top);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kShortMaxChunks; ++k)
        if (k < chunks) {
            sum = fmaf(f_s[k], ml_s[k].y, sum);
            a = fmaf(f_s[k], v[k], a);
        }
    const int g = c >> 5, e = c & 31;
    out[head * 128 + (layout_v == RVQ_GROUP_STRIDED ? 4 * e + g : c)] = a / sum;
}

// Tokens up to which the one-pass kernel is the faster one.  Measured (us, tables / one pass, K = 1024, depth 8): 32 query
// heads 12000 tokens 75 / 62, 20000 103 / 94, 26000 123 / 119, 32768 146 / 146; 8 heads, packed 26000 126 / 125, 32768
// 149 / 156.  With up to four stages on both sides the tables take half the reads: 12000 tokens 63 / 63, 20000 90 / 95.
constexpr int64_t kShortTokens = 28672, kShortTokensShallow = 12288;
bool short_wanted(const Shape &sk, const Shape &sv, int64_t tokens)
{
    return tokens <= (sk.R <= 4 && sv.R <= 4 ? kShortTokensShallow : kShortTokens);
}

// Chunks of a short cache: no more than its tokens feed.
int short_chunks(int64_t tokens)
{
    const int64_t fed = (tokens + kShortWarps - 1) / kShortWarps;
    return (int)(fed < kShortMaxChunks ? fed : kShortMaxChunks);
}

size_t short_workspace(int64_t tokens, int q_heads)
{
    return (size_t)short_chunks(tokens) * q_heads * (128 * 4 + 8) + 256;
}

}  // namespace

// (token counts: the kernels index group rows, 32 per token, with 32-bit integers, and step past the end
// by up to two strides of at most 18 * 32 tokens)
constexpr int64_t kAttMaxTokens = (1LL << 26) - 4096;

bool attention_supported(const Shape &sk, const Shape &sv, int kv_heads, int q_heads, int64_t tokens)
{
    auto ok = [](const Shape &s) { return s.dim == 128 && s.gd == 32 && s.R <= 8 && s.K <= kAttMaxK; };
    const int J = kv_heads > 0 ? q_heads / kv_heads : 0;
    return ok(sk) && ok(sv) && kv_heads == 8 && q_heads == kv_heads * J && (J == 1 || J == 2 || J == 4) &&
           tokens <= kAttMaxTokens;
}

size_t attention_workspace_bytes(int64_t tokens, int q_heads)
{
    const size_t scores = ((size_t)tokens * q_heads * 4 + 255) / 256 * 256;
    const size_t tables = scores + 256 /* maxima */ + 256 /* weight sums */ + (size_t)q_heads * 128 * 4;
    const size_t shorter = tokens <= kShortTokens ? short_workspace(tokens, q_heads) : 0;
    return tables > shorter ? tables : shorter;
}

int launch_attention_decode(const Shape &sk, const Shape &sv, const float *q, int q_heads, const void *codes_k,
                            const uint16_t *std_k, const void *codes_v, const uint16_t *std_v, int64_t tokens,
                            const float *cb_k, const float *cb_v, const int32_t *position, const float *cos_sin,
                            int positions, int pairing, float scale, float *out, void *workspace, rvq_status *st,
                            cudaStream_t stream)
{
    const int J = q_heads / 8;
    const int sms = sm_count();
    if (sms <= 0) return RVQ_ERR_DEVICE;
    uint8_t *ws = reinterpret_cast<uint8_t *>(workspace);
    if (short_wanted(sk, sv, tokens)) {
        const int chunks = short_chunks(tokens), rope = cos_sin ? (pairing == RVQ_ROPE_HALVES ? 1 : 2) : 0;
        float *part = reinterpret_cast<float *>(ws);
        float2 *part_ml = reinterpret_cast<float2 *>(ws + (size_t)chunks * q_heads * 128 * 4);
        const float2 *cs = reinterpret_cast<const float2 *>(cos_sin);
        const float sl = scale * 1.4426950408889634f;
        auto launch = [&](auto kernel) {
            kernel<<<dim3((unsigned)chunks, 8), kShortThreads, 0, stream>>>(sk, sv, q, codes_k, std_k, codes_v, std_v, (uint32_t)tokens, cb_k,
                                                                           cb_v, position, cs, positions, sl, part, part_ml, st);
        };
        const int depth = sk.R != sv.R ? 0 : sk.R;
#define RVQ_SHORT_F(ROPE, JJ)                                                                                        \
        (depth == 8 ? launch(att_short_kernel<ROPE, JJ, 8>) : depth == 6 ? launch(att_short_kernel<ROPE, JJ, 6>)     \
         : depth == 4 ? launch(att_short_kernel<ROPE, JJ, 4>) : launch(att_short_kernel<ROPE, JJ, 0>))
#define RVQ_SHORT_J(ROPE) (J == 4 ? RVQ_SHORT_F(ROPE, 4) : J == 2 ? RVQ_SHORT_F(ROPE, 2) : RVQ_SHORT_F(ROPE, 1))
        if (rope == 0) RVQ_SHORT_J(0); else if (rope == 1) RVQ_SHORT_J(1); else RVQ_SHORT_J(2);
#undef RVQ_SHORT_J
#undef RVQ_SHORT_F
        int rc = check_launch();
        if (rc != RVQ_OK) return rc;
        // (its launch overlaps the first kernel; it waits for that one's results on the device)
        return launch_chained(true, att_combine_kernel, dim3((unsigned)q_heads), 128, 0, stream, part, part_ml, chunks, sv.layout, out);
    }
    const size_t score_bytes = ((size_t)tokens * q_heads * 4 + 255) / 256 * 256;
    float *scores = reinterpret_cast<float *>(ws);
    uint32_t *m_ord = reinterpret_cast<uint32_t *>(ws + score_bytes);
    float *weight_sum = reinterpret_cast<float *>(ws + score_bytes + 256);
    float *out_acc = reinterpret_cast<float *>(ws + score_bytes + 512);
    if (cudaMemsetAsync(ws, 0, score_bytes + 512 + (size_t)q_heads * 128 * 4, stream) != cudaSuccess) return RVQ_ERR_LAUNCH;

    int parts = sms / kAttSlices;
    const int64_t tiles = (tokens + 31) / 32;
    if (parts > tiles) parts = (int)tiles;
    if (parts < 1) parts = 1;
    const int rope = cos_sin ? (pairing == RVQ_ROPE_HALVES ? 1 : 2) : 0;
    int rc = RVQ_OK;
    auto scores_launch = [&](auto kernel) -> int {
        const size_t smem = (size_t)sk.K * 128;
        if (!allow_shared_memory(reinterpret_cast<const void *>(kernel), (int)smem))
            return RVQ_ERR_LAUNCH;
        kernel<<<parts * kAttSlices, kAttThreads, smem, stream>>>(sk, codes_k, std_k, tokens, cb_k, q, position,
                                                                   reinterpret_cast<const float2 *>(cos_sin), positions,
                                                                   scores, st);
        return check_launch();
    };
    auto values_launch = [&](auto kernel) -> int {
        size_t smem = (size_t)sv.K * 128;
        const size_t red = (size_t)4 * J * 32 * 32 * 4;
        if (smem < red) smem = red;
        if (!allow_shared_memory(reinterpret_cast<const void *>(kernel), (int)smem))
            return RVQ_ERR_LAUNCH;
        return launch_chained(true, kernel, dim3(parts * kAttSlices), kAttThreads, smem, stream, sv, codes_v, std_v, tokens, cb_v, scores, out_acc, st);
    };
#define RVQ_ATT_S4(LAY, ROPE, JJ) (sk.R <= 4 ? scores_launch(att_scores_kernel<LAY, ROPE, JJ, 4>) : scores_launch(att_scores_kernel<LAY, ROPE, JJ, 8>))
#define RVQ_ATT_S3(LAY, ROPE) (J == 4 ? RVQ_ATT_S4(LAY, ROPE, 4) : J == 2 ? RVQ_ATT_S4(LAY, ROPE, 2) : RVQ_ATT_S4(LAY, ROPE, 1))
#define RVQ_ATT_S2(LAY) (rope == 0 ? RVQ_ATT_S3(LAY, 0) : rope == 1 ? RVQ_ATT_S3(LAY, 1) : RVQ_ATT_S3(LAY, 2))
    rc = sk.layout == RVQ_GROUP_CONTIGUOUS ? RVQ_ATT_S2(RVQ_GROUP_CONTIGUOUS) : RVQ_ATT_S2(RVQ_GROUP_STRIDED);
#undef RVQ_ATT_S2
#undef RVQ_ATT_S3
#undef RVQ_ATT_S4
    if (rc != RVQ_OK) return rc;
    {
        int blocks = (int)((tokens * q_heads / 4 + kAttThreads - 1) / kAttThreads);
        if (blocks > sms) blocks = sms;
        if (blocks < 1) blocks = 1;
        rc = launch_chained(true, att_max_kernel, dim3(blocks), kAttThreads, 0, stream, scores, tokens, q_heads, scale, m_ord);
        if (rc != RVQ_OK) return rc;
        rc = launch_chained(true, att_weights_kernel, dim3(blocks), kAttThreads, 0, stream, scores, std_v, tokens, q_heads,
                            J == 4 ? 2 : J == 2 ? 1 : 0, scale, m_ord, weight_sum);
        if (rc != RVQ_OK) return rc;
    }
#define RVQ_ATT_V3(LAY, JJ) (sv.R <= 4 ? values_launch(att_values_kernel<LAY, JJ, 4>) : values_launch(att_values_kernel<LAY, JJ, 8>))
#define RVQ_ATT_V2(LAY) (J == 4 ? RVQ_ATT_V3(LAY, 4) : J == 2 ? RVQ_ATT_V3(LAY, 2) : RVQ_ATT_V3(LAY, 1))
    rc = sv.layout == RVQ_GROUP_CONTIGUOUS ? RVQ_ATT_V2(RVQ_GROUP_CONTIGUOUS) : RVQ_ATT_V2(RVQ_GROUP_STRIDED);
#undef RVQ_ATT_V2
#undef RVQ_ATT_V3
    if (rc != RVQ_OK) return rc;
    return launch_chained(true, att_finish_kernel, dim3((q_heads * 128 + 255) / 256), 256, 0, stream, out_acc, weight_sum, q_heads, out);
}

}  // namespace rvq
