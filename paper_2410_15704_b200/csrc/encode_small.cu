// Encode of a few head vectors (a decode step's new tokens): latency, not throughput.
//
// On a tile of 128 rows or less the tensor-core kernel spends its time in chains that wait for one
// another, stage after stage, chunk after chunk of the codebook: 95 us for one token's 8 vectors at 2048
// codes.  Here a cluster of up to eight CTAs splits the codebook: every CTA streams its codewords of
// every stage (float32 blocks of the prepared section) into shared memory, a thread takes one codeword
// into registers and computes its exact distances to the cluster's rows (direct form, the scalar
// kernel's operation order, so the codes are the same).  The minima of all warps meet in every CTA's
// shared memory (st.async, counted by an mbarrier), every CTA picks the winner for itself and reads its
// codeword from the CTA that holds it.
// What bounds it: the chain of the stages.  Measured for 4 rows at 1024 codes: distances and
// minima 1050 cycles of a stage, the exchange 260, winner and residual 500, the barrier and the next
// stage's table 300.
#include "encode_mma.cuh"

namespace rvq {

namespace {

constexpr int kSmallAtOnce = 2;                   // rows that a thread takes at a time
constexpr int kSmallThreads = 512;
constexpr int kSmallRows = 32;                    // group rows per cluster at most
constexpr int kSmallMaxCluster = 8;
constexpr int kSmallTableBytes = 10 * kFloatBlockBytes;   // eight stages of one block, or five of two

struct SmallParams {
    Shape s;
    const void *x;
    int64_t n, stride;
    const uint8_t *blocks;      // float32 blocks, [R][block of 128 codewords]
    void *codes;
    uint16_t *std16;
    rvq_status *st;
    float *energy;
    int vectors;        // head vectors per cluster
    int rows;           // their group rows
    int blocks_per_stage;
};

struct SmallWork {
    // (distance bits, code) of the best of every warp's 32 codewords, from every CTA of the cluster
    unsigned long long keys[2][kSmallRows][kSmallMaxCluster * 8];
    float z[kSmallRows + kSmallAtOnce][32];
    float xs[kSmallRows * 32];
    float dev[kSmallRows];
    uint16_t codes[kSmallRows][kFloatMaxStages];
    uint64_t full[kFloatMaxStages], arrived[2];
    volatile uint32_t abort_flag;
};
constexpr int kSmallSharedBytes = kSmallTableBytes + (int)sizeof(SmallWork);

// blockDim.x = PER * 128 threads for every kSmallAtOnce rows of the cluster, up to kSmallThreads.
template <int PER>                                                // blocks of 128 codewords per CTA and stage
__global__ void __launch_bounds__(kSmallThreads, 1)
encode_small_kernel(const SmallParams p)
{
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t *table = smem;                                        // [buffers][PER blocks]
    SmallWork &w = *reinterpret_cast<SmallWork *>(smem + kSmallTableBytes);
    constexpr int kBuffers = PER == 1 ? kFloatMaxStages : 5;
    constexpr uint32_t kStageBytes = PER * kFloatBlockBytes;
    const Shape &s = p.s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x;
    const int G = s.G, R = s.R, dim = s.dim;
    const int rank = (int)cluster_rank(), ctas = (int)gridDim.y;  // CTA of the cluster, CTAs of a cluster
    const int64_t v0 = (int64_t)blockIdx.x * p.vectors;           // first head vector of this cluster
    const int mine = min(PER, p.blocks_per_stage - rank * PER);   // (the last CTA of an odd number of blocks: one of two)
    const uint8_t *src = p.blocks + (size_t)rank * kStageBytes;
    const size_t src_stage = (size_t)p.blocks_per_stage * kFloatBlockBytes;
    auto copy_stage = [&](int r, int buffer) {
        const uint32_t bar = smem_u32(&w.full[buffer]);
        mbar_expect_tx(bar, (uint32_t)mine * kFloatBlockBytes);
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(table) + (uint32_t)buffer * kStageBytes), "l"(src + r * src_stage),
                       "r"((uint32_t)mine * kFloatBlockBytes), "r"(bar) : "memory");
    };
    // the head vectors, widened, while the last warp sets up the barriers and starts the copies
    const int live = (int)min((int64_t)p.vectors, p.n - v0);
    if (warp == threads / 32 - 1) {
        if (lane < kBuffers) mbar_init(smem_u32(&w.full[lane]), 1);
        if (lane < 2) mbar_init(smem_u32(&w.arrived[lane]), 1);
        if (lane == 0) w.abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        __syncwarp();
        if (lane < kBuffers && lane < R) copy_stage(lane, lane);
    }
    if (ctas > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    for (int t = tid; t < p.rows * 32; t += threads) {
        const int v = t / dim;
        w.xs[t] = v < live ? load_as_float(p.x, (v0 + v) * p.stride + (t - v * dim), s.dtype) : 0.0f;
    }
    __syncthreads();
    if (warp == 0) {
        // deviations (the scalar kernel's order of additions): one lane per row
        const int vl = lane / G, g = lane - vl * G, base = lane - g;
        const bool row = lane < p.rows;
        const float *xr = w.xs + (row ? vl * dim + (s.layout == RVQ_GROUP_STRIDED ? g : g * 32) : 0);
        const int step = s.layout == RVQ_GROUP_STRIDED ? G : 1;
        float c[32], a = 0.0f, mu = 0.0f, sum = 0.0f;
#pragma unroll
        for (int i = 0; i < 32; ++i) c[i] = xr[i * step];
#pragma unroll
        for (int i = 0; i < 32; ++i) a += c[i];
        for (int k = 0; k < G; ++k) mu += __shfl_sync(0xFFFFFFFFu, a, (base + k) & 31);
        mu /= (float)dim;
        a = 0.0f;
#pragma unroll
        for (int i = 0; i < 32; ++i) a += (c[i] - mu) * (c[i] - mu);
        for (int k = 0; k < G; ++k) sum += __shfl_sync(0xFFFFFFFFu, a, (base + k) & 31);
        const float dev = sqrtf(sum / (float)(dim - s.ddof));
        const bool deg = vl >= live || deviation_is_degenerate(dev);
        if (row) w.dev[lane] = deg ? 0.0f : dev;                  // (0: codes 0, residual 0)
        if (row && rank == 0 && vl < live && g == 0) {
            const uint16_t hb = deg ? (uint16_t)0 : __half_as_ushort(__float2half_rn(dev));
            p.std16[v0 + vl] = hb;
            if (p.st) {
                if (deg) atomicAdd(&p.st->degenerate_vectors, 1u);
                else if ((hb & 0x7FFFu) == 0 || (hb & 0x7FFFu) >= 0x7C00u) atomicAdd(&p.st->std_out_of_half, 1u);
            }
        }
    }
    __syncthreads();
    for (int t = tid; t < p.rows * 32; t += threads) {
        const int row = t >> 5, v = row / G;
        const float dev = w.dev[row];
        w.z[row][t & 31] = dev == 0.0f ? 0.0f : w.xs[v * dim + channel_of(s.layout, G, 32, row - v * G, t & 31)] / dev;
    }
    if (ctas > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // every CTA's barriers are set up
    __syncthreads();

    // thread: codeword c of this CTA, kSmallAtOnce rows from `first` on, then those `next` further on
    const int c = tid & (PER * 128 - 1), first = kSmallAtOnce * (tid / (PER * 128)), next = kSmallAtOnce * (threads / (PER * 128));
    const int slots = ctas * PER * 4;                             // warps of a cluster that have codewords of one row
    const int slot = rank * PER * 4 + (c >> 5);
    const bool real = (c >> 7) < mine;
    const uint32_t arrived0 = smem_u32(&w.arrived[0]);
    const uint32_t to_keys = map_to(smem_u32(&w.keys[0][0][slot]), (uint32_t)min(lane, ctas - 1));    // in CTA `lane`
    const uint32_t to_arrived = map_to(arrived0, (uint32_t)min(lane, ctas - 1));
    constexpr uint32_t kRowKeys = kSmallMaxCluster * 8 * 8, kAllKeys = kSmallRows * kRowKeys;      // bytes
    bool ok = true;
    int buffer = 0, next_buffer = 0;
    uint32_t full_par = 0;                                        // of next_buffer
    int r = 0;
    // this thread's codeword of the next stage
    float4 e[8];
    auto take_codeword = [&] {
        const bool there = mbar_wait(smem_u32(&w.full[next_buffer]), full_par, &w.abort_flag);
        const float4 *mine4 = reinterpret_cast<const float4 *>(table + (size_t)next_buffer * kStageBytes) + (c >> 7) * 1024 + (c & 127);
#pragma unroll
        for (int q = 0; q < 8; ++q) e[q] = mine4[q * 128];
        if (++next_buffer == kBuffers) { next_buffer = 0; full_par ^= 1u; }
        return there;
    };
    ok = take_codeword();
#pragma unroll 1
    for (; r < R; ++r) {
        const uint32_t par = (uint32_t)r & 1u;
        if (tid == 0) mbar_expect_tx(arrived0 + 8u * par, (uint32_t)(p.rows * slots * 8));
        const uint8_t *stage = table + (size_t)buffer * kStageBytes;
#pragma unroll 1
        for (int row = first; row < p.rows; row += next) {
            float d[kSmallAtOnce] = {};
#pragma unroll
            for (int q = 0; q < 8; ++q) {
#pragma unroll
                for (int k = 0; k < kSmallAtOnce; ++k) {
                    const float4 u = *reinterpret_cast<const float4 *>(&w.z[row + k][4 * q]);
                    float t;
                    t = u.x - e[q].x; d[k] = fmaf(t, t, d[k]); t = u.y - e[q].y; d[k] = fmaf(t, t, d[k]);
                    t = u.z - e[q].z; d[k] = fmaf(t, t, d[k]); t = u.w - e[q].w; d[k] = fmaf(t, t, d[k]);
                }
            }
            // non-negative floats order like their bit patterns; a distance that is infinite or NaN never wins
            uint32_t bits[kSmallAtOnce], m[kSmallAtOnce], who[kSmallAtOnce];
#pragma unroll
            for (int k = 0; k < kSmallAtOnce; ++k) bits[k] = real ? __float_as_uint(d[k]) : 0xFFFFFFFFu;
#pragma unroll
            for (int k = 0; k < kSmallAtOnce; ++k) m[k] = __reduce_min_sync(0xFFFFFFFFu, bits[k]);
#pragma unroll
            for (int k = 0; k < kSmallAtOnce; ++k) who[k] = __ballot_sync(0xFFFFFFFFu, bits[k] == m[k]);
            // this warp's best of these rows, to every CTA of the cluster: lane l to CTA l
#pragma unroll
            for (int k = 0; k < kSmallAtOnce; ++k) {
                const unsigned long long key = ((unsigned long long)m[k] << 32) | (uint32_t)(rank * PER * 128 + (c & ~31) + __ffs(who[k]) - 1);
                if (lane < ctas && row + k < p.rows)
                    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
                                 ::"r"(to_keys + par * kAllKeys + (uint32_t)(row + k) * kRowKeys), "l"(key), "r"(to_arrived + 8u * par) : "memory");
            }
        }
        // (while the minima travel: read at the stage's start, 16 warps' codewords were 512 cycles of its distances)
        if (r + 1 < R) ok = take_codeword() && ok;
        ok = mbar_wait(arrived0 + 8u * par, (uint32_t)(r >> 1) & 1u, &w.abort_flag) && ok;
        const bool subtract = r + 1 < R || p.energy != nullptr;
        float e2 = 0.0f;
#pragma unroll 1
        for (int row = warp; row < p.rows; row += threads / 32) {
            unsigned long long k = lane < slots ? w.keys[par][row][lane] : ~0ull;
            if (PER == 2 && lane + 32 < slots) k = min(k, w.keys[par][row][lane + 32]);
            const uint32_t hi = (uint32_t)(k >> 32), best = __reduce_min_sync(0xFFFFFFFFu, hi);
            uint32_t j = __reduce_min_sync(0xFFFFFFFFu, hi == best ? (uint32_t)k : 0xFFFFFFFFu);
            const float dev = w.dev[row];
            if (best >= 0x7F800000u || dev == 0.0f) j = 0;
            if (lane == 0) w.codes[row][r] = (uint16_t)j;
            if (subtract) {
                const uint32_t at = smem_u32(stage) + ((j >> 7) & (PER - 1)) * kFloatBlockBytes + (uint32_t)(lane >> 2) * 2048u +
                                    (j & 127u) * 16u + (uint32_t)(lane & 3) * 4u;
                float ev;
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(ev) : "r"(map_to(at, (j >> 7) / PER)) : "memory");
                const float nz = dev == 0.0f ? 0.0f : w.z[row][lane] - ev;
                w.z[row][lane] = nz;
                e2 = fmaf(nz, nz, e2);
            }
        }
        if (p.energy && rank == 0) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) e2 += __shfl_xor_sync(0xFFFFFFFFu, e2, off);
            if (lane == 0 && e2 != 0.0f) atomicAdd(p.energy + r, e2);
        }
        if (!ok) w.abort_flag = 1u;
        __syncthreads();
        if (w.abort_flag) { ok = false; break; }
        // Every CTA has read this CTA's codewords of stage r - 1 (it could not have sent its minima of stage r
        // before): their place is free.
        if (PER == 2 && tid == 0 && r >= 1 && r - 1 + kBuffers < R) copy_stage(r - 1 + kBuffers, r - 1);
        if (++buffer == kBuffers) buffer = 0;
    }
    if (!ok && tid == 0) {
        // (the stages from here on are still coming in)
        for (int k = r; k < R && k < kBuffers + max(r - 1, 0); ++k)
            mbar_drain(smem_u32(&w.full[k % kBuffers]), (uint32_t)(k / kBuffers) & 1u);
        if (p.st) atomicAdd(&p.st->wait_timeouts, 1u);
    }
    if (ctas > 1 && (p.energy || !ok))                            // (codewords of other CTAs were read last)
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    if (rank != 0) return;

    // codes out (Section 3.2 storage)
    if (s.bits == 16) {
        uint16_t *o = reinterpret_cast<uint16_t *>(p.codes) + v0 * G * R;
        for (int t = tid; t < live * G * R; t += threads) { const int row = t / R; o[t] = w.codes[row][t - row * R]; }
    } else {
        const int words = s.code_bytes / 4;
        for (int t = tid; t < live * words; t += threads) {
            const int v = t / words, wd = t - v * words;
            uint32_t word = 0;
            const int k_lo = (32 * wd) / s.bits, k_hi = min(s.per_vector - 1, (32 * wd + 31) / s.bits);
            for (int k = k_lo; k <= k_hi; ++k) {
                const uint32_t val = w.codes[v * G + k / R][k % R];
                const int sh = k * s.bits - 32 * wd;
                word |= sh >= 0 ? (val << sh) : (val >> (-sh));
            }
            reinterpret_cast<uint32_t *>(p.codes)[(v0 + v) * words + wd] = word;
        }
    }
}

struct SmallPlan {
    const void *kernel;
    int per_cta, ctas, at_once;
};

// How a shape is split, and how many clusters of that split the current device runs at a time (0: none).
SmallPlan small_plan(const Shape &s)
{
    const int blocks = slots_per_stage(s.K), per = blocks <= kSmallMaxCluster ? 1 : 2;
    SmallPlan plan{per == 1 ? reinterpret_cast<const void *>(encode_small_kernel<1>) : reinterpret_cast<const void *>(encode_small_kernel<2>),
                   per, (blocks + per - 1) / per, 0};
    plan.at_once = resident_clusters(plan.kernel, plan.ctas, kSmallThreads, kSmallSharedBytes);
    return plan;
}

}  // namespace

// Group rows per cluster up to which this encoder is faster than tiles of 128 rows: a row costs about 1.6 us at two blocks per CTA and
// 1 us at one, a tile's stages about the same for one row as for 128.  us, this encoder / tiles: 2048 codes 16 rows 32.6 / 32.9, 20 39.1 / 33.3; 1024 codes 20 rows
// 27.5 / 28.1, 24 29.8 / 28.1; 512 codes 20 rows 25.6 / 26.1, 24 27.7 / 26.1; at depth 4, 1024 codes, 24 rows 16.6 / 17.7.  Up to three chunks, where
// a tile is one CTA's (encode_tensor.cu): 256 codes 16 rows 20.4 / 22.0, 20 25.0 / 22.0.
bool encode_small_wanted(const Shape &s, int64_t n)
{
    if (!float_blocks_prepared(s) || s.raw || s.G > kSmallRows || n < 1 || n > 4096) return false;
    const SmallPlan plan = small_plan(s);
    const int64_t vectors = plan.at_once > 0 ? (n + plan.at_once - 1) / plan.at_once : 0;
    const int most = plan.per_cta == 2 || slots_per_stage(s.K) <= 3 ? 16 : s.R <= 4 ? 24 : 20;
    return vectors == 1 || (vectors > 0 && vectors * s.G <= most);
}

int launch_encode_small(const Shape &s, const void *x, int64_t n, int64_t stride, const void *prepared, void *codes,
                        uint16_t *std16, rvq_status *st, cudaStream_t stream, float *energy)
{
    const SmallPlan plan = small_plan(s);
    if (plan.at_once <= 0 || !allow_shared_memory(plan.kernel, kSmallSharedBytes)) return RVQ_ERR_LAUNCH;
    const int vectors = (int)((n + plan.at_once - 1) / plan.at_once);
    SmallParams p{s, x, n, stride, reinterpret_cast<const uint8_t *>(prepared) + float_blocks_offset(s), codes, std16, st, energy,
                  vectors, vectors * s.G, slots_per_stage(s.K)};
    int threads = plan.per_cta * 128 * ((p.rows + kSmallAtOnce - 1) / kSmallAtOnce);
    if (threads > kSmallThreads) threads = kSmallThreads;
    void *args[] = {&p};
    return launch_clusters(plan.kernel, (int)((n + vectors - 1) / vectors), plan.ctas, threads, kSmallSharedBytes, stream, args);
}

}  // namespace rvq
