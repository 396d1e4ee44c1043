// Decode of few head vectors (groups of 32, a power-of-two number of them from 4, depth <= 8), with or without the
// rotary embedding: codewords straight from the float32 codebooks in L2 (Section 2.2, last sentence; Section 3.2).
//
// The table decoders (decode_sliced.cu) fill up to 227 KB of shared memory per CTA before the first row: 5-9 us,
// 13-23 us for the rotary ones, however few the rows.  Here a warp takes four group rows of one head vector at a
// time, lane = (row, four-element piece): it fetches one code (stage = piece), the codes travel by shuffle,
// and each stage is one 16-byte load per lane, four whole 128-byte lines per instruction, all stages in flight
// together.  Float32 sums in stage order, multiplied by the deviation, rotated, rounded once.
// What bounds it: for few rows the chain codes -> codewords -> store (2.5 us); then L2, 4 KB per head vector of
// 128 channels, which is why the tables take over (decode_direct_wanted).
#include "prepared.cuh"

namespace rvq {

namespace {

constexpr int kDirectThreads = 128;

struct DirectRope {
    const int32_t *position;
    int per_position;
    const float2 *table;          // (cos, sin) [positions][dim / 2]
    int positions;
};

// ROPE 0: none; 1: pairs (k, k + dim/2); 2: pairs (2k, 2k + 1).
template <int ROPE>
__global__ void __launch_bounds__(kDirectThreads)
decode_direct_kernel(Shape s, const void *__restrict__ codes, const uint16_t *__restrict__ std16, int64_t n,
                     const float *__restrict__ cb, void *__restrict__ out, int64_t stride, rvq_status *st, DirectRope rope)
{
    const int lane = threadIdx.x & 31, rho = lane >> 3, q = lane & 7;
    const int G = s.G, R = s.R, lg = __ffs(G) - 1;
    const bool strided = s.layout == RVQ_GROUP_STRIDED;
    const int64_t sets = n << (lg - 2);                       // of four group rows
    const uint32_t K = (uint32_t)s.K;
    uint32_t bad = 0;
    for (int64_t set = (int64_t)blockIdx.x * (kDirectThreads / 32) + (threadIdx.x >> 5); set < sets;
         set += (int64_t)gridDim.x * (kDirectThreads / 32)) {
        const int64_t v = set >> (lg - 2);
        const int k = (int)(set & ((G >> 2) - 1));
        // rows of the set: groups 2k, 2k + 1 and the same G / 2 further on, so that the channels of a rotary pair
        // are in one warp whatever the pairing
        const int g = 2 * k + (rho & 1) + (rho >> 1) * (G >> 1);
        // lane: stage q of its row
        uint32_t code = 0;
        if (q < R) {
            code = read_code(reinterpret_cast<const uint8_t *>(codes) + v * s.code_bytes, g * R + q, s.bits, s.code_bytes);
            if (code >= K) { code = 0; ++bad; }
        }
        const float sd = __half2float(__ushort_as_half(__ldg(std16 + v)));
        float4 e[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint32_t j = __shfl_sync(0xFFFFFFFFu, code, (lane & 24) | r);
            e[r] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < R) e[r] = __ldg(reinterpret_cast<const float4 *>(cb + ((size_t)r * K + j) * 32) + q);
        }
        float2 cs[4];
        if (ROPE != 0) {
            const int pos = min(max(__ldg(rope.position + v / rope.per_position), 0), rope.positions - 1);
            const float2 *row = rope.table + (size_t)pos * (16 * G);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int el = 4 * q + i, c = strided ? (el << lg) + g : g * 32 + el;
                cs[i] = __ldg(row + (ROPE == 1 ? c & (16 * G - 1) : c >> 1));
            }
        }
        float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int r = 0; r < 8; ++r) { o[0] += e[r].x; o[1] += e[r].y; o[2] += e[r].z; o[3] += e[r].w; }
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] *= sd;
        if (ROPE == 2 && !strided) {
#pragma unroll
            for (int i = 0; i < 4; i += 2) {
                const float a = o[i], b = o[i + 1];
                o[i] = a * cs[i].x - b * cs[i].y;
                o[i + 1] = b * cs[i].x + a * cs[i].y;
            }
        } else if (ROPE != 0) {
            // the other channel of the pair: group g ^ G/2, group g ^ 1, or (half-split pairs, strided groups) 16 elements on
            const int other = ROPE == 2 ? 8 : strided ? 4 : 16;
            const bool first = (lane & other) == 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float p = __shfl_xor_sync(0xFFFFFFFFu, o[i], other);
                o[i] = first ? o[i] * cs[i].x - p * cs[i].y : o[i] * cs[i].x + p * cs[i].y;
            }
        }
        if (!strided) {
            const int64_t at = v * stride + g * 32 + 4 * q;
            if (s.dtype == RVQ_F32) {
                *reinterpret_cast<float4 *>(reinterpret_cast<float *>(out) + at) = make_float4(o[0], o[1], o[2], o[3]);
            } else {
                uint2 w;
                if (s.dtype == RVQ_BF16) {
                    const __nv_bfloat162 a = __floats2bfloat162_rn(o[0], o[1]), b = __floats2bfloat162_rn(o[2], o[3]);
                    w = make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
                } else {
                    const __half2 a = __floats2half2_rn(o[0], o[1]), b = __floats2half2_rn(o[2], o[3]);
                    w = make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
                }
                *reinterpret_cast<uint2 *>(reinterpret_cast<uint16_t *>(out) + at) = w;
            }
        } else {
            // lane rho of the four holds elements 4q .. 4q+3 of its group and wants element 4q + rho of all four
            float t[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                // round x: exchange with lane rho ^ x; both send the element that the other wants
                const float send = (rho ^ x) == 0 ? o[0] : (rho ^ x) == 1 ? o[1] : (rho ^ x) == 2 ? o[2] : o[3];
                const float got = x == 0 ? send : __shfl_xor_sync(0xFFFFFFFFu, send, 8 * x);
#pragma unroll
                for (int y = 0; y < 4; ++y) t[y] = (rho ^ x) == y ? got : t[y];
            }
            // t[y]: group of row y; rows 0, 1 and rows 2, 3 are neighbouring channels
            const int64_t at = v * stride + ((int64_t)(4 * q + rho) << lg) + 2 * k;
            if (s.dtype == RVQ_F32) {
                float *f = reinterpret_cast<float *>(out) + at;
                *reinterpret_cast<float2 *>(f) = make_float2(t[0], t[1]);
                *reinterpret_cast<float2 *>(f + (G >> 1)) = make_float2(t[2], t[3]);
            } else {
                uint32_t a, b;
                if (s.dtype == RVQ_BF16) {
                    const __nv_bfloat162 x = __floats2bfloat162_rn(t[0], t[1]), y = __floats2bfloat162_rn(t[2], t[3]);
                    a = *reinterpret_cast<const uint32_t *>(&x); b = *reinterpret_cast<const uint32_t *>(&y);
                } else {
                    const __half2 x = __floats2half2_rn(t[0], t[1]), y = __floats2half2_rn(t[2], t[3]);
                    a = *reinterpret_cast<const uint32_t *>(&x); b = *reinterpret_cast<const uint32_t *>(&y);
                }
                uint16_t *h = reinterpret_cast<uint16_t *>(out) + at;
                *reinterpret_cast<uint32_t *>(h) = a;
                *reinterpret_cast<uint32_t *>(h + (G >> 1)) = b;
            }
        }
    }
    if (bad && st) atomicAdd(&st->bad_codes, bad);
}

}  // namespace

#ifndef RVQ_DIRECT
#define RVQ_DIRECT 1
#endif
bool decode_direct_wanted(const Shape &s, int64_t n, bool rope)
{
    if (s.gd != 32 || s.G < 4 || (s.G & (s.G - 1)) != 0 || s.R > 8) return false;
    return n * (s.G / 4) <= (RVQ_DIRECT ? RVQ_DIRECT * 1024 : (rope ? 8192 : 4096));
}

int launch_decode_direct(const Shape &s, const void *codes, const uint16_t *std16, int64_t n, const float *cb, void *out,
                         int64_t stride, rvq_status *st, cudaStream_t stream, const int32_t *position, int per_position,
                         const float *table, int positions, int pairing)
{
    if (n == 0) return RVQ_OK;
    const int sms = sm_count();
    if (sms <= 0) return RVQ_ERR_DEVICE;
    const int64_t warps = n * (s.G / 4), want = (warps + kDirectThreads / 32 - 1) / (kDirectThreads / 32);
    const unsigned grid = (unsigned)(want < (int64_t)sms * 16 ? want : (int64_t)sms * 16);
    const DirectRope rope{position, per_position, reinterpret_cast<const float2 *>(table), positions};
    if (!position) decode_direct_kernel<0><<<grid, kDirectThreads, 0, stream>>>(s, codes, std16, n, cb, out, stride, st, rope);
    else if (pairing == RVQ_ROPE_HALVES) decode_direct_kernel<1><<<grid, kDirectThreads, 0, stream>>>(s, codes, std16, n, cb, out, stride, st, rope);
    else decode_direct_kernel<2><<<grid, kDirectThreads, 0, stream>>>(s, codes, std16, n, cb, out, stride, st, rope);
    return check_launch();
}

}  // namespace rvq
