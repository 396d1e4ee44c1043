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

constexpr int kDirectThreads = 128, kDirectBlocks = 6;        // (72-80 registers; eight blocks spill and are slower)

struct DirectRope {
    const int32_t *position;
    uint32_t per_position, heads;     // head vectors of a position; the same where they divide the call's, else 1
    const float2 *table;          // (cos, sin) [positions][dim / 2]
    int positions;
};

// ROPE 0: none; 1: pairs (k, k + dim/2); 2: pairs (2k, 2k + 1).  DEPTH: the depth, or 0 for any up to 8.
template <int ROPE, int DEPTH>
__global__ void __launch_bounds__(kDirectThreads, kDirectBlocks)
decode_direct_kernel(Shape s, const void *__restrict__ codes, const uint16_t *__restrict__ std16, uint32_t n,
                     const float *__restrict__ cb, void *__restrict__ out, int64_t stride, rvq_status *st, DirectRope rope)
{
    const uint32_t lane = threadIdx.x & 31, rho = lane >> 3, q = lane & 7;
    const uint32_t G = s.G, R = DEPTH ? DEPTH : s.R, lg = __ffs(G) - 1, lgk = lg - 2, K = s.K;
    const bool strided = s.layout == RVQ_GROUP_STRIDED;
    uint32_t bad = 0;
    // every warp takes a run of consecutive sets of four group rows; code and deviation of the next set are asked
    // for before the codewords of this one are added up.  Set number -> (head vector, part k of its groups): the
    // parts of a vector one after the other, or with rotary pairs the heads of a token first (they share the
    // part's cosines and sines).
    const uint32_t sets = n << lgk, warps = gridDim.x * (kDirectThreads / 32), warp = blockIdx.x * (kDirectThreads / 32) + (threadIdx.x >> 5);
    const uint32_t per = sets / warps, extra = sets - per * warps;
    uint32_t set = warp * per + min(warp, extra);
    const uint32_t end = set + per + (warp < extra ? 1u : 0u);
    // rows of set (v, k): groups 2k, 2k + 1 and the same G / 2 further on, so that the channels of a rotary pair
    // are in one warp whatever the pairing; lane: stage q of its row
    const uint32_t g0 = (rho & 1) + (rho >> 1) * (G >> 1);
    const uint32_t bits = s.bits, mask = (1u << bits) - 1u;
    const uint32_t stage_off = q * K * 128u;                  // bytes of the codebooks before stage q
    const bool has = q < R;
    const uint32_t parts = G >> 2, heads = ROPE != 0 ? rope.heads : 1u;
    struct Place { uint32_t v, k; };
    auto place = [&](uint32_t at) -> Place {
        if (ROPE == 0 || lgk == 0) return {at >> lgk, at & (parts - 1u)};
        const uint32_t unit = at / heads, head = at - unit * heads;          // (token, part), head
        return {(unit >> lgk) * heads + head, unit & (parts - 1u)};
    };
    auto fetch = [&](Place at, uint32_t &code, uint16_t &sd) {
        const uint32_t v = at.v, g = g0 + 2u * at.k;
        const uint8_t *vec = reinterpret_cast<const uint8_t *>(codes) + (size_t)v * (uint32_t)s.code_bytes;
        const uint32_t k = g * R + q;
        code = 0;
        if (has) {
            if (bits == 16) {
                code = __ldg(reinterpret_cast<const uint16_t *>(vec) + k);
            } else {
                const uint32_t o = k * bits, w = o >> 5, sh = o & 31u;
                const uint32_t *p = reinterpret_cast<const uint32_t *>(vec) + w;
                code = __funnelshift_r(__ldg(p), sh + bits > 32u ? __ldg(p + 1) : 0u, sh) & mask;
            }
        }
        sd = __ldg(std16 + v);
    };
    uint32_t next_code = 0, pairs_of = 0xFFFFFFFFu;
    Place next = place(min(set, sets - 1u));
    uint16_t next_sd = 0;
    float2 cs[4];
    const uint8_t *piece = reinterpret_cast<const uint8_t *>(cb) + q * 16u;
    if (set < end) fetch(next, next_code, next_sd);
    for (; set < end; ++set) {
        const uint32_t v = next.v, k = next.k, g = g0 + 2u * k;
        const float sd = __half2float(__ushort_as_half(next_sd));
        if (next_code >= K) { next_code = 0; ++bad; }
        const uint32_t off = stage_off + next_code * 128u;    // of this lane's codeword (8 * 65536 * 128 bytes fit 32 bits)
        uint64_t lo[8], hi[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint32_t at = __shfl_sync(0xFFFFFFFFu, off, (lane & 24) | r);
            lo[r] = hi[r] = 0ull;
            if (r < (DEPTH ? DEPTH : (int)R))
                asm("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(lo[r]), "=l"(hi[r]) : "l"(piece + at));
        }
        if (set + 1 < end) { next = place(set + 1); fetch(next, next_code, next_sd); }
        if (ROPE != 0) {
            const uint32_t t = v / rope.per_position;
            if (t * parts + k != pairs_of) {                  // (warp-uniform)
                pairs_of = t * parts + k;
                const int pos = min(max(__ldg(rope.position + t), 0), rope.positions - 1);
                const float2 *row = rope.table + (size_t)pos * (16 * G);
#pragma unroll
                for (uint32_t i = 0; i < 4; ++i) {
                    const uint32_t el = 4 * q + i, c = strided ? (el << lg) + g : g * 32 + el;
                    cs[i] = __ldg(row + (ROPE == 1 ? c & (16 * G - 1) : c >> 1));
                }
            }
        }
        uint64_t s0 = lo[0], s1 = hi[0];
#pragma unroll
        for (int r = 1; r < (DEPTH ? DEPTH : 8); ++r) { s0 = add_f32x2(s0, lo[r]); s1 = add_f32x2(s1, hi[r]); }
        float o[4] = {__uint_as_float((uint32_t)s0), __uint_as_float((uint32_t)(s0 >> 32)),
                      __uint_as_float((uint32_t)s1), __uint_as_float((uint32_t)(s1 >> 32))};
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
            const uint32_t other = ROPE == 2 ? 8 : strided ? 4 : 16;
            const bool first = (lane & other) == 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float p = __shfl_xor_sync(0xFFFFFFFFu, o[i], other);
                o[i] = first ? o[i] * cs[i].x - p * cs[i].y : o[i] * cs[i].x + p * cs[i].y;
            }
        }
        if (!strided) {
            const size_t at = (size_t)v * stride + g * 32 + 4 * q;
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
            for (uint32_t x = 0; x < 4; ++x) {
                // round x: exchange with lane rho ^ x; both send the element that the other wants
                const float send = (rho ^ x) == 0 ? o[0] : (rho ^ x) == 1 ? o[1] : (rho ^ x) == 2 ? o[2] : o[3];
                const float got = x == 0 ? send : __shfl_xor_sync(0xFFFFFFFFu, send, 8 * x);
#pragma unroll
                for (uint32_t y = 0; y < 4; ++y) t[y] = (rho ^ x) == y ? got : t[y];
            }
            // t[y]: group of row y; rows 0, 1 and rows 2, 3 are neighbouring channels
            const size_t at = (size_t)v * stride + ((4 * q + rho) << lg) + 2 * k;
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

// Where the table decoders are the faster ones: 16-bit outputs at depth 8 with up to 1536 codes (8-channel level
// tables, or 4-channel float32 ones for large deviations), from a number of group rows on that pays for filling
// them.  Which tables a batch takes, and so where it crosses, hangs on its deviations, which the host does not know: the lines
// stand where values cross, and for rotated vectors where keys do.  Measured (us, tables / direct, K = 1024, dim 128):
//   values (level tables)     16384 vectors 8.3 / 8.2, 28672 10.4 / 10.3, 32768 10.4 / 10.4, 65536 14.4 / 18.6, 131072 22.6 / 33.1;
//   keys (float32 tables)     28672 16.5 / 11.8, 65536 22.7 / 20.6, 98304 29.4 / 28.8, 131072 37.0 / 39.2, 262144 62 / 78: from 28673 to
//                             about 100000 keys that are read back unrotated lose up to 5 us;
//   keys, rotated             65536 30.9 / 25.6, 98304 39.1 / 37.1, 131072 47.3 / 49.7, 196608 66 / 74;
//   moderate deviations, rotated   32768 14.4 / 13.3, 65536 18.6 / 22.6, 131072 32.9 / 43.1: these lose up to 10 us before the line.
// dim 256: 65536 27 / 33.  Direct wins at every size for 2048 codes (262144 vectors 74 / 61; keys 117 / 75, rotary
// 232 / 93), float32 outputs (110 / 68) and smaller depths (depth 4: 57 / 41, float32 103 / 46).
bool decode_direct_wanted(const Shape &s, int64_t n, bool rope, bool prepared)
{
    const int64_t sets = n * (s.G / 4);
    if (s.gd != 32 || s.G < 4 || (s.G & (s.G - 1)) != 0 || s.R > 8 || sets > 0x7FFFFFFF) return false;
    const bool tables = prepared && s.dtype != RVQ_F32 && s.K <= kDecodeWideK && s.R == 8 && s.bits >= 10 && s.G <= 32;
    if (!tables || (rope && s.G != 4)) return true;
    return sets <= (rope ? 131072 : s.G == 4 ? 28672 : 65536);
}

int launch_decode_direct(const Shape &s, const void *codes, const uint16_t *std16, int64_t n, const float *cb, void *out,
                         int64_t stride, rvq_status *st, cudaStream_t stream, const int32_t *position, int per_position,
                         const float *table, int positions, int pairing)
{
    if (n == 0) return RVQ_OK;
    const int sms = sm_count();
    if (sms <= 0) return RVQ_ERR_DEVICE;
    const int64_t warps = n * (s.G / 4), want = (warps + kDirectThreads / 32 - 1) / (kDirectThreads / 32);
    const unsigned grid = (unsigned)(want < (int64_t)sms * kDirectBlocks ? want : (int64_t)sms * kDirectBlocks);
    const DirectRope rope{position, (uint32_t)per_position, n % per_position == 0 ? (uint32_t)per_position : 1u, reinterpret_cast<const float2 *>(table), positions};
    const int kind = !position ? 0 : pairing == RVQ_ROPE_HALVES ? 1 : 2;
#define RVQ_DIRECT_KINDS(D) (kind == 0 ? decode_direct_kernel<0, D> : kind == 1 ? decode_direct_kernel<1, D> : decode_direct_kernel<2, D>)
    auto kernel = s.R == 8 ? RVQ_DIRECT_KINDS(8) : s.R == 6 ? RVQ_DIRECT_KINDS(6) : s.R == 4 ? RVQ_DIRECT_KINDS(4) : RVQ_DIRECT_KINDS(0);
#undef RVQ_DIRECT_KINDS
    kernel<<<grid, kDirectThreads, 0, stream>>>(s, codes, std16, (uint32_t)n, cb, out, stride, st, rope);
    return check_launch();
}

}  // namespace rvq
