// Encode of a few head vectors (a decode step's new tokens): latency, not throughput.
//
// On a tile of 128 rows or less the tensor-core kernel spends its time in chains that wait for one
// another, stage after stage, chunk after chunk of the codebook: 95 us for one token's 8 vectors at 2048
// codes.  Here a cluster of up to eight CTAs splits the codebook: every CTA streams its codewords of
// every stage (float32 blocks of the prepared section) into shared memory, a thread takes one codeword
// into registers and computes its exact distances to the cluster's rows (direct form, the scalar
// kernel's operation order, so the codes are the same).  The minima of all warps meet in every CTA's
// shared memory (st.async, counted by an mbarrier), every CTA picks the winner for itself and reads its
// codeword from the CTA that holds it.  For a token or two a cluster takes one or two groups of a vector (small_share_plan).
// What bounds it: the chain of the stages.  Measured for 4 rows at 1024 codes, when a stage began with reading the
// codewords and not while the minima of the one before travel: distances and
// minima 1050 cycles of a stage, the exchange 260, winner and residual 500, the barrier and the next
// stage's table 300.
#include "encode_mma.cuh"

namespace rvq {

namespace {

constexpr int kSmallThreads = 512;
constexpr int kSmallRows = 32;                    // group rows per cluster at most
constexpr int kSmallMaxCluster = 8;
// stages in shared memory at a time, by the blocks of 128 codewords that a CTA has of each
template <int PER> constexpr int kSmallBuffers = PER == 1 ? kFloatMaxStages : PER == 2 ? 5 : 3;

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
    int rows;           // group rows per cluster: theirs, or a share of the only one's
    int shares;         // clusters per head vector, each with `rows` of its groups (1: whole vectors)
    int blocks_per_stage;
};

// ROWS: group rows of a cluster at most.
template <int ROWS>
struct SmallWork {
    // (distance bits, code) of the best of every warp's 32 codewords, from every CTA of the cluster
    unsigned long long keys[2][ROWS][kSmallMaxCluster * 8];
    float z[ROWS + 1][32];
    float xs[kSmallRows * 32];
    float dev[kSmallRows];
    uint16_t codes[ROWS][kFloatMaxStages];
    uint64_t full[kFloatMaxStages], arrived[2];
    volatile uint32_t abort_flag;
};
template <int PER> constexpr int kSmallMostRows = PER == 4 ? 2 : kSmallRows;
template <int PER> constexpr int kSmallSharedBytes = kSmallBuffers<PER> * PER * kFloatBlockBytes + (int)sizeof(SmallWork<kSmallMostRows<PER>>);

// PER: blocks of 128 codewords per CTA and stage.  AT_ONCE: rows that a thread takes at a time.
// blockDim.x = PER * 128 threads for every AT_ONCE rows of the cluster, up to kSmallThreads.
template <int PER, int AT_ONCE>
__global__ void __launch_bounds__(kSmallThreads, 1)
encode_small_kernel(const SmallParams p)
{
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t *table = smem;                                        // [buffers][PER blocks]
    constexpr int kBuffers = kSmallBuffers<PER>, kRows = kSmallMostRows<PER>;
    constexpr uint32_t kStageBytes = PER * kFloatBlockBytes;
    SmallWork<kRows> &w = *reinterpret_cast<SmallWork<kRows> *>(smem + kBuffers * kStageBytes);
    const Shape &s = p.s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x;
    const int G = s.G, R = s.R, dim = s.dim;
    const int rank = (int)cluster_rank(), ctas = (int)gridDim.y;  // CTA of the cluster, CTAs of a cluster
    // first head vector of this cluster, and the first of its groups
    const int64_t v0 = p.shares > 1 ? (int64_t)blockIdx.x / p.shares : (int64_t)blockIdx.x * p.vectors;
    const int g0 = p.shares > 1 ? (int)blockIdx.x % p.shares * p.rows : 0;
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
    for (int t = tid; t < p.vectors * dim; t += threads) {
        const int v = t / dim;
        w.xs[t] = v < live ? load_as_float(p.x, (v0 + v) * p.stride + (t - v * dim), s.dtype) : 0.0f;
    }
    __syncthreads();
    if (warp == 0) {
        // deviations (the scalar kernel's order of additions): one lane per row
        const int vl = lane / G, g = lane - vl * G, base = lane - g;
        const bool row = lane < p.vectors * G;
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
        if (row && rank == 0 && vl < live && g == 0 && g0 == 0) {
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
        const int row = (t >> 5) + g0, v = row / G;
        const float dev = w.dev[row];
        w.z[t >> 5][t & 31] = dev == 0.0f ? 0.0f : w.xs[v * dim + channel_of(s.layout, G, 32, row - v * G, t & 31)] / dev;
    }
    if (ctas > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // every CTA's barriers are set up
    __syncthreads();

    // thread: codeword c of this CTA, AT_ONCE rows from `first` on, then those `next` further on
    const int c = tid & (PER * 128 - 1), first = AT_ONCE * (tid / (PER * 128)), next = AT_ONCE * (threads / (PER * 128));
    const int slots = ctas * PER * 4;                             // warps of a cluster that have codewords of one row
    const int slot = rank * PER * 4 + (c >> 5);
    const bool real = (c >> 7) < mine;
    const uint32_t arrived0 = smem_u32(&w.arrived[0]);
    const uint32_t to_keys = map_to(smem_u32(&w.keys[0][0][slot]), (uint32_t)min(lane, ctas - 1));    // in CTA `lane`
    const uint32_t to_arrived = map_to(arrived0, (uint32_t)min(lane, ctas - 1));
    constexpr uint32_t kRowKeys = kSmallMaxCluster * 8 * 8, kAllKeys = kRows * kRowKeys;      // bytes
    bool ok = true;
    int buffer = 0, next_buffer = 0;
    uint32_t full_par = 0;                                        // of next_buffer
    int r = 0, copies = min(R, kBuffers);                         // stages asked for (thread 0)
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
            float d[AT_ONCE] = {};
#pragma unroll
            for (int q = 0; q < 8; ++q) {
#pragma unroll
                for (int k = 0; k < AT_ONCE; ++k) {
                    const float4 u = *reinterpret_cast<const float4 *>(&w.z[row + k][4 * q]);
                    float t;
                    t = u.x - e[q].x; d[k] = fmaf(t, t, d[k]); t = u.y - e[q].y; d[k] = fmaf(t, t, d[k]);
                    t = u.z - e[q].z; d[k] = fmaf(t, t, d[k]); t = u.w - e[q].w; d[k] = fmaf(t, t, d[k]);
                }
            }
            // non-negative floats order like their bit patterns; a distance that is infinite or NaN never wins
            uint32_t bits[AT_ONCE], m[AT_ONCE], who[AT_ONCE];
#pragma unroll
            for (int k = 0; k < AT_ONCE; ++k) bits[k] = real ? __float_as_uint(d[k]) : 0xFFFFFFFFu;
#pragma unroll
            for (int k = 0; k < AT_ONCE; ++k) m[k] = __reduce_min_sync(0xFFFFFFFFu, bits[k]);
#pragma unroll
            for (int k = 0; k < AT_ONCE; ++k) who[k] = __ballot_sync(0xFFFFFFFFu, bits[k] == m[k]);
            // this warp's best of these rows, to every CTA of the cluster: lane l to CTA l
#pragma unroll
            for (int k = 0; k < AT_ONCE; ++k) {
                const unsigned long long key = ((unsigned long long)m[k] << 32) | (uint32_t)(rank * PER * 128 + (c & ~31) + __ffs(who[k]) - 1);
                if (lane < ctas && row + k < p.rows)
                    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
                                 ::"r"(to_keys + par * kAllKeys + (uint32_t)(row + k) * kRowKeys), "l"(key), "r"(to_arrived + 8u * par) : "memory");
            }
        }
        // (while the minima travel: read at the stage's start, 16 warps' codewords were 512 cycles of its distances)
        if (r + 1 < R) ok = take_codeword() && ok;
        ok = mbar_wait(arrived0 + 8u * par, (uint32_t)(r >> 1) & 1u, &w.abort_flag) && ok;
        // Every CTA has read this CTA's codewords of stage r - 1 (it could not have sent its minima of stage r
        // before): their place is free.
        if (PER > 1 && tid == 0 && ok && r >= 1 && copies < R) {
            copy_stage(copies, copies % kBuffers);
            ++copies;
        }
        const bool subtract = r + 1 < R || p.energy != nullptr;
        float e2 = 0.0f;
#pragma unroll 1
        for (int row = warp; row < p.rows; row += threads / 32) {
            unsigned long long k = lane < slots ? w.keys[par][row][lane] : ~0ull;
            if (PER > 1 && lane + 32 < slots) k = min(k, w.keys[par][row][lane + 32]);
            const uint32_t hi = (uint32_t)(k >> 32), best = __reduce_min_sync(0xFFFFFFFFu, hi);
            uint32_t j = __reduce_min_sync(0xFFFFFFFFu, hi == best ? (uint32_t)k : 0xFFFFFFFFu);
            const float dev = w.dev[g0 + row];
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
        if (++buffer == kBuffers) buffer = 0;
    }
    if (!ok && tid == 0) {
        // (the stages from here on are still coming in)
        for (int k = r; k < copies; ++k)
            mbar_drain(smem_u32(&w.full[k % kBuffers]), (uint32_t)(k / kBuffers) & 1u);
        if (p.st) atomicAdd(&p.st->wait_timeouts, 1u);
    }
    if (ctas > 1 && (p.energy || !ok))                            // (codewords of other CTAs were read last)
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    if (rank != 0) return;

    // codes out (Section 3.2 storage)
    if (p.shares > 1) {
        // (a row's codes are whole bytes, and those of a vector whole words: small_plan)
        const int row_bytes = R * s.bits / 8;
        uint8_t *o = reinterpret_cast<uint8_t *>(p.codes) + v0 * s.code_bytes + g0 * row_bytes;
        for (int t = tid; t < p.rows * row_bytes; t += threads) {
            const int row = t / row_bytes, bit = 8 * (t - row * row_bytes);
            uint32_t byte = 0;
            for (int k = bit / s.bits, at = k * s.bits - bit; at < 8 && k < R; ++k, at += s.bits)
                byte |= at >= 0 ? (uint32_t)w.codes[row][k] << at : (uint32_t)w.codes[row][k] >> -at;
            o[t] = (uint8_t)byte;
        }
    } else if (s.bits == 16) {
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
    const void *kernel;                        // null: not for this encoder
    int ctas, vectors, rows, shares, threads, smem;
    int64_t clusters;
};

template <int PER, int AT_ONCE>
void small_kernel(SmallPlan &plan)
{
    plan.kernel = reinterpret_cast<const void *>(encode_small_kernel<PER, AT_ONCE>);
    plan.smem = kSmallSharedBytes<PER>;
    const int threads = PER * 128 * ((plan.rows + AT_ONCE - 1) / AT_ONCE);
    plan.threads = threads < kSmallThreads ? threads : kSmallThreads;
}

// A vector of whose groups several clusters of up to four CTAs take one or two each, where all of these run at a time: a
// token's or two.  (Clusters of eight CTAs with all rows of a vector leave half of the SMs idle, and have twice the
// distances each: 8 vectors, 2048 codes 16.4 -> 14.35 us, 1024 codes 12.3 -> 12.3, 16 vectors 20.5 -> 16.4 and 16.4 ->
// 14.35.  Calls back to back come in steps of 2.05 us.)
SmallPlan small_share_plan(const Shape &s, int64_t n)
{
    SmallPlan plan{};
    const int blocks = slots_per_stage(s.K), per = blocks <= 4 ? 1 : blocks <= 8 ? 2 : 4;
    // (codes are written by bytes)
    if (s.G < 2 || s.R * s.bits % 8 != 0 || s.per_vector * s.bits % 32 != 0) return plan;
    for (int rows = 1; rows <= 2 && rows < s.G; ++rows) {
        SmallPlan t{};
        t.ctas = (blocks + per - 1) / per; t.vectors = 1; t.rows = rows; t.shares = s.G / rows; t.clusters = n * t.shares;
        if (rows == 1) {
            if (per == 1) small_kernel<1, 1>(t); else if (per == 2) small_kernel<2, 1>(t); else small_kernel<4, 1>(t);
        } else {
            if (per == 1) small_kernel<1, 2>(t); else if (per == 2) small_kernel<2, 2>(t); else small_kernel<4, 2>(t);
        }
        if (t.clusters <= resident_clusters(t.kernel, t.ctas, kSmallThreads, t.smem)) return t;
    }
    return plan;
}

// Group rows per cluster up to which this encoder is faster than tiles of 128 rows: a row costs about 1.5 us at two blocks per CTA and
// 1 us at one, a tile's stages about the same for one row as for 128.  us, this encoder / tiles: 2048 codes 16 rows 32.1 / 34.8, 20 38.9 / 34.8;
// 1536 codes 20 rows 30.7 / 32.8, 24 36.9 / 34.8; 1024 codes 20 rows 26.7 / 30.8, 24 28.7 / 28.7, 28 32.8 / 29.4; 512 codes 24 rows 26.7 / 28.7, 28 30.7 / 28.7; at
// depth 4, 1024 codes, 24 rows 16.9 / 18.4.  Up to three chunks, where a tile is one CTA's (encode_tensor.cu): 384 codes 20 rows 24.6 / 26.6, 24 26.7 / 26.6;
// 256 codes 16 rows 20.5 / 24.6, 20 24.6 / 24.6, 24 26.7 / 24.4.
SmallPlan small_plan(const Shape &s, int64_t n)
{
    SmallPlan plan{};
    if (!float_blocks_prepared(s) || s.raw || s.G > kSmallRows || n < 1 || n > 4096) return plan;
    plan = small_share_plan(s, n);
    if (plan.kernel) return plan;
    const int blocks = slots_per_stage(s.K), per = blocks <= kSmallMaxCluster ? 1 : 2;
    plan.ctas = (blocks + per - 1) / per;
    const int at_once = resident_clusters(per == 1 ? reinterpret_cast<const void *>(encode_small_kernel<1, 2>) : reinterpret_cast<const void *>(encode_small_kernel<2, 2>),
                                          plan.ctas, kSmallThreads, per == 1 ? kSmallSharedBytes<1> : kSmallSharedBytes<2>);
    const int64_t vectors = at_once > 0 ? (n + at_once - 1) / at_once : 0;
    const int most = blocks > 12 ? 16 : blocks > 8 || blocks <= 3 ? 20 : 24;
    if (vectors == 0 || (vectors > 1 && vectors * s.G > most)) return plan;
    plan.vectors = (int)vectors; plan.rows = (int)vectors * s.G; plan.shares = 1; plan.clusters = (n + vectors - 1) / vectors;
    if (per == 1) small_kernel<1, 2>(plan); else small_kernel<2, 2>(plan);
    return plan;
}

}  // namespace

bool encode_small_wanted(const Shape &s, int64_t n) { return small_plan(s, n).kernel != nullptr; }

int launch_encode_small(const Shape &s, const void *x, int64_t n, int64_t stride, const void *prepared, void *codes,
                        uint16_t *std16, rvq_status *st, cudaStream_t stream, float *energy)
{
    const SmallPlan plan = small_plan(s, n);
    if (!plan.kernel || !allow_shared_memory(plan.kernel, plan.smem)) return RVQ_ERR_LAUNCH;
    SmallParams p{s, x, n, stride, reinterpret_cast<const uint8_t *>(prepared) + float_blocks_offset(s), codes, std16, st, energy,
                  plan.vectors, plan.rows, plan.shares, slots_per_stage(s.K)};
    void *args[] = {&p};
    return launch_clusters(plan.kernel, (int)plan.clusters, plan.ctas, plan.threads, plan.smem, stream, args);
}

}  // namespace rvq
