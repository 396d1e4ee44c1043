// Tensor-core encode of few row tiles (up to one per SM): one tile's codebook sweep split.
//
// The throughput kernel (encode_tensor.cu) gives an SM three tiles of 128 rows and lets them share the
// operand stream; with fewer tiles than three per SM most of the chip is idle and the tiles that run
// wait, chunk after chunk, for one accumulator each (154 tiles: 145 us at 2048 codes, as long as one).
// Here a tile belongs to a cluster of C CTAs (1 .. 8: split_ctas), each of
// which sweeps its share of the stage's chunks with up to three accumulators in flight over one A operand.
// An epilogue group of four warps per accumulator folds its chunks into running minima of the tile's
// 128 rows (encode_mma.cuh), as the throughput kernel does for all chunks.  At the stage end the owner group of
// a CTA joins the groups' parts -- the two best chunks, the sets of columns inside the error window -- and sends the
// CTA's part of every row to all CTAs of the cluster (st.async, counted by an mbarrier); each owner group merges the
// parts of its rows -- one part with one column inside the window: the choice is certified; otherwise the listed
// columns are compared exactly in float32 -- and takes the residual to the next stage.  All CTAs of a
// cluster make the same choice from the same parts.
// What bounds it: the chain of the stages.  One of 5200 cycles at 20 tiles and 2048 codes (6 CTAs of two or three chunks):
// operand 400, first accumulator 900 later, the third and its fold 1900 after that, the joined part 300, the exchange
// 500-800, merge and window 550, the codeword, asked for as soon as a candidate is known, 900.  us with parts sent by
// every group, one issuer that waited before each chain and the codeword fetched at the end, and now: 616 values at
// 2048 codes 45.7 / 39.0, 2400 keys at 1024 54.5 / 46.6, 4720 at 2048 (one CTA per tile) 82.6 / 66.1, 4720 at 512
// 45.2 / 39.0.  (The cycles were read with approximate roots in the window; the rounded ones add some 250.)
#include "encode_mma.cuh"

namespace rvq {

namespace {

constexpr int kGroups = 3;                                // accumulators, and epilogue groups of 128 threads
constexpr int kSplitThreads = 512;                        // 12 epilogue warps, three issuers, loader
constexpr int kSplitRing = 6;
constexpr int kEarly = 4;                                 // pieces that a thread has on their way at the start
constexpr int kMaxParts = 8;                              // CTAs of a cluster
// TMEM column of the A operand (32 columns), and of the constant one (8)
constexpr int kATmem = kGroups * 128, kOnesTmem = kATmem + 32;

struct Part {                                             // what a group, or a CTA, knows of a row at the stage end
    float m1, m2;                                         // its two lowest chunk minima
    uint32_t sets;                                  // columns inside its window (Listed::word); bit 24: a third chunk
    uint32_t chunks;                                      // chunk of m1, chunk of m2 << 16
};

constexpr int kSOffB = 0;
constexpr int kSOffZ = kSOffB + kSplitRing * kSlotBytes;  // residuals, float [32][kZPitch]
constexpr int kZPitch = 129;                              // (odd: neither rows nor elements of a row share banks)
constexpr int kSOffParts = kSOffZ + 32 * kZPitch * 4;     // Part [2][kMaxParts][128]
// Part [kGroups - 1][128], of the groups but the owners
constexpr int kSOffLocal = kSOffParts + 2 * kMaxParts * 128 * 16;
constexpr int kSOffCodes = kSOffLocal + (kGroups - 1) * 128 * 16;
constexpr int kSOffNorm = kSOffCodes + 128 * 16 * 2;      // squared norms of the scaled residuals
constexpr int kSOffBars = kSOffNorm + 128 * 4;
constexpr int kSOffStages = kSOffBars + 256;              // StageConst[16]
constexpr int kSplitSmem = kSOffStages + 16 * (int)sizeof(StageConst);

constexpr int kSFull = 0, kSEmpty = kSplitRing, kSReady = 2 * kSplitRing, kSAccFull = kSReady + 1,
              kSAccFree = kSAccFull + kGroups, kSArrived = kSAccFree + kGroups, kSLocal = kSArrived + 2,
              kSDrain = kSLocal + 1, kSBars = kSDrain + kGroups;

struct SplitParams {
    Shape s;
    const void *x;
    int64_t n, stride;
    const float *cb;
    const uint8_t *prepared;
    void *codes;
    uint16_t *std16;
    rvq_status *st;
    float *energy;
    int groups;         // accumulators in use: min(kGroups, chunks of a CTA)
};

// One stage's chunks grp, grp + P .. of a CTA's, folded from accumulator `grp` into w; false when a wait gave up.
__device__ __forceinline__ bool sweep_chunks(Sweep &w, int grp, int P, int base, int cnt, uint32_t acc,
                                             uint32_t bar_full, uint32_t bar_free, uint32_t &acc_par, uint32_t bar_empty,
                                             uint32_t first_use, int lane, volatile uint32_t *abort_flag)
{
    w.clear();
    const bool releases = (threadIdx.x & 127) < 32;
    uint32_t slot = (first_use + (uint32_t)grp) % (uint32_t)kSplitRing;
#pragma unroll 1
    for (int c = grp; c < cnt; c += P) {
        bool ok = mbar_wait(bar_full, acc_par, abort_flag);
        ok = __all_sync(0xFFFFFFFFu, ok);
        acc_par ^= 1u;
        if (!ok) return false;
        // (the chain has read its operand slot: the loader may fill it again)
        if (releases && lane == 0) mbar_arrive(bar_empty + 8u * slot);
        if ((slot += (uint32_t)P) >= (uint32_t)kSplitRing) slot -= (uint32_t)kSplitRing;
        tc_fence_after();
        uint32_t ua[32], ub[32], uc[32], ud[32];
        tmem_ld32_issue(acc, ua);
        tmem_ld32_issue(acc + 32, ub);
        tmem_ld32_issue(acc + 64, uc);
        tmem_ld32_issue(acc + 96, ud);
        tmem_ld_wait4(ua, ub, uc, ud);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_free);
        float lowest;
        fold_block(w, ua, 0, lowest);
        fold_block(w, ub, 1, lowest);
        fold_block(w, uc, 2, lowest);
        fold_block(w, ud, 3, lowest);
        rank_chunk(w, lowest, base + c);
    }
    return true;
}

__global__ void __launch_bounds__(kSplitThreads, 1)
encode_split_kernel(const SplitParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kSOffBars);
    uint32_t *tmem_word = reinterpret_cast<uint32_t *>(smem + kSOffBars + kSBars * 8);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + kSOffBars + kSBars * 8 + 4);
    const Shape &s = p.s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int S = slots_per_stage(s.K), R = s.R, P = p.groups;
    const int rank = (int)cluster_rank(), ctas = (int)gridDim.y;
    // this CTA's chunks of every stage
    const int per = S / ctas, rem = S - per * ctas;
    const int base = rank * per + min(rank, rem), cnt = per + (rank < rem ? 1 : 0);
    const uint32_t bar0 = smem_u32(bars);
    auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };

    // the tile's head vectors by all groups: the first pieces on their way while the CTA sets itself up
    const int lg = __ffs(s.G) - 1, lp = lg + (s.elem_bytes == 4 ? 3 : 2);      // log2 of a vector's groups and pieces
    const int64_t v_tile = ((int64_t)blockIdx.x * 128) >> lg;
    const int pieces = 128 << (lp - lg);
    uint4 raw[kEarly];
#pragma unroll
    for (int u = 0; u < kEarly; ++u) {
        const int k = tid + 128 * P * u;
        raw[u] = make_uint4(0u, 0u, 0u, 0u);
        if (tid < 128 * P && k < pieces)
            raw[u] = load_piece(s, p.x, p.n, p.stride, v_tile + (k >> lp), k & ((1 << lp) - 1));
    }
    if (tid == 0) {
        for (int i = 0; i < kSplitRing; ++i) { mbar_init(BAR(kSFull + i), 1); mbar_init(BAR(kSEmpty + i), 1); }
        mbar_init(BAR(kSReady), 4);
        for (int g = 0; g < kGroups; ++g) {
            mbar_init(BAR(kSAccFull + g), 1); mbar_init(BAR(kSAccFree + g), 4); mbar_init(BAR(kSDrain + g), 1);
        }
        mbar_init(BAR(kSArrived), 1);
        mbar_init(BAR(kSArrived + 1), 1);
        mbar_init(BAR(kSLocal), 4 * max(P - 1, 1));
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 12) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_word)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    StageConst *sc = reinterpret_cast<StageConst *>(smem + kSOffStages);
    load_stage_consts(p.prepared, R, tid, sc);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (ctas > 1) asm volatile("barrier.cluster.arrive.relaxed;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    const uint32_t tmem = *tmem_word;
    // the constant A operand (the issuer hears of it with the first A operand, from the same warps)
    if (warp < 4) tmem_ones(tmem + ((uint32_t)(warp * 32) << 16) + kOnesTmem);

    // (the role warps' registers go to the epilogue warps, as in the throughput kernel: 4 x 40 + 12 x 152 of 16 x
    // 128)
    if (warp >= 12) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == 13) {
            // ------------------------------------------------------------ operand loader
            if (lane == 0) {
                const uint8_t *image = p.prepared + kPreparedImageOffset + (size_t)base * kSlotStride;
                uint32_t slot = 0, par = 1, issued = 0;
                bool ok = true;
                for (int r = 0; r < R && ok; ++r)
                    for (int c = 0; c < cnt; ++c) {
                        if (issued >= (uint32_t)kSplitRing) ok = mbar_wait(BAR(kSEmpty + slot), par, abort_flag);
                        if (!ok) break;
                        mbar_expect_tx(BAR(kSFull + slot), kSlotBytes);
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                     ::"r"(smem_u32(smem + kSOffB) + slot * (uint32_t)kSlotBytes),
                                       "l"(image + ((size_t)r * S + c) * kSlotStride),
                                       "r"((uint32_t)kSlotBytes), "r"(BAR(kSFull + slot)) : "memory");
                        ++issued;
                        if (++slot == (uint32_t)kSplitRing) { slot = 0; par ^= 1u; }
                    }
                for (uint32_t k = issued > (uint32_t)kSplitRing ? issued - kSplitRing : 0u; k < issued; ++k)
                    mbar_drain(BAR(kSFull + (int)(k % kSplitRing)), (k / kSplitRing) & 1u);
            }
        } else {
            // ------------------------------------------------------------ MMA issuers, one per accumulator
            // A wait costs 150-200 cycles also when there is nothing to wait for, a commit as much.  So the first
            // chunks of a stage, one per accumulator, are waited for before the operand is, and their chains go out
            // together, from the first issuer (their accumulators are free: the owners make an operand only after all
            // groups' parts); the chunks after them come from a warp per accumulator, whose waits overlap.
            // No wait may be more than one phase ahead of its barrier, or it would take an old phase for its own.
            // Accumulators: every issuer waits for each fold in turn.  Slots: the use before, six chunks back, is the
            // issuer's own or of an earlier stage; of that the first issuer, where it has not waited for all of a
            // stage's slots itself, knows by the other groups' parts, the others by the fold of this stage's first
            // chunk.
            const int mine = warp == 12 ? 0 : warp - 13;
            const uint64_t bdesc0 = make_smem_desc(smem_u32(smem + kSOffB), kSlotCodewords * 16, 128);
            const int first = min(cnt, P);
            const bool more = cnt > mine + P;
            uint32_t folds = 0;                                               // of this accumulator, waited for
            bool ok = mine < first && (mine == 0 || more);
            for (int r = 0; r < R && ok; ++r) {
                const uint32_t use0 = (uint32_t)(r * cnt);         // the CTA's chunks are numbered through all stages
                if (mine == 0) {
                    if (r > 0 && cnt > P) ok = mbar_wait(BAR(kSLocal), (uint32_t)(r - 1) & 1u, abort_flag);
                    for (int c = 0; c < first && ok; ++c)
                        ok = mbar_wait(BAR(kSFull + (use0 + c) % kSplitRing), ((use0 + c) / kSplitRing) & 1u, abort_flag);
                    if (ok) ok = mbar_wait(BAR(kSReady), (uint32_t)r & 1u, abort_flag);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < kGroups; ++k)
                            if (k < first) {
                                issue_chain(tmem + 128u * (uint32_t)k, tmem + kATmem,
                                            bdesc0 + (uint64_t)((use0 + k) % kSplitRing * (uint32_t)(kSlotBytes >> 4)),
                                            tmem + kOnesTmem);
                                mma_commit(BAR(kSAccFull + k));
                            }
                    }
                    __syncwarp();
                }
                if (!more) continue;
                for (int c = mine + P; c < cnt && ok; c += P) {
                    const uint32_t use = use0 + (uint32_t)c;
                    ok = mbar_wait(BAR(kSAccFree + mine), folds & 1u, abort_flag);
                    ++folds;
                    if (ok) ok = mbar_wait(BAR(kSFull + use % kSplitRing), (use / kSplitRing) & 1u, abort_flag);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        issue_chain(tmem + 128u * (uint32_t)mine, tmem + kATmem,
                                    bdesc0 + (uint64_t)(use % kSplitRing * (uint32_t)(kSlotBytes >> 4)), tmem + kOnesTmem);
                        mma_commit(BAR(kSAccFull + mine));
                    }
                    __syncwarp();
                }
                if (ok) ok = mbar_wait(BAR(kSAccFree + mine), folds & 1u, abort_flag);
                ++folds;
            }
            // (nothing of this warp's is in flight at a regular end)
            if (mine < first) {
                __syncwarp();
                if (elect_one()) mma_commit(BAR(kSDrain + mine));
                mbar_drain(BAR(kSDrain + mine), 0u);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue groups
        asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
        const int grp = warp >> 2, q4 = warp & 3;
        const int row = q4 * 32 + lane;
        const uint32_t lanes = (uint32_t)(q4 * 32) << 16;
        float *z_park = reinterpret_cast<float *>(smem + kSOffZ) + row;                 // [i][row]
        float *norm = reinterpret_cast<float *>(smem + kSOffNorm);
        uint16_t *codes_s = reinterpret_cast<uint16_t *>(smem + kSOffCodes);            // [row][16]
        const Part *parts = reinterpret_cast<const Part *>(smem + kSOffParts);          // [2][kMaxParts][128]
        const uint32_t mine = smem_u32(smem + kSOffParts) + (uint32_t)(rank * 128 + row) * 16u;
        Part *local = reinterpret_cast<Part *>(smem + kSOffLocal) + row;
        const int G = s.G;
        uint32_t acc_par = 0;
        uint32_t n_rescored = 0, n_exhaustive = 0, n_degenerate = 0, n_stdrange = 0;
        if (grp < P) {                                                       // (groups without an accumulator sit by)
            const int64_t v_first = v_tile + q4 * 32 / G;
            const int64_t v = v_first + lane / G;
            const bool valid = v < p.n;
            // the tile's head vectors, widened: element i of row at [i][row]
            float *zs = reinterpret_cast<float *>(smem + kSOffZ);
#pragma unroll
            for (int u = 0; u < kEarly; ++u) {
                const int k = tid + 128 * P * u;
                if (k < pieces) scatter_piece<kZPitch>(s, raw[u], k & ((1 << lp) - 1), zs + ((k >> lp) << lg));
            }
            for (int k = tid + 128 * P * kEarly; k < pieces; k += 128 * P)
                scatter_piece<kZPitch>(s, load_piece(s, p.x, p.n, p.stride, v_tile + (k >> lp), k & ((1 << lp) - 1)),
                                       k & ((1 << lp) - 1), zs + ((k >> lp) << lg));
            asm volatile("bar.sync 1, %0;" ::"r"(128 * P) : "memory");
            const uint32_t acc = tmem + lanes + 128u * (uint32_t)grp;
            if (grp != 0) {
                // ---- the other groups: their part of every row, to the owners
#pragma unroll 1
                for (int r = 0; r < R; ++r) {
                    const StageConst prm = sc[r];
                    if (grp >= cnt) {
                        // a group without chunks, which no chain holds back: not before the owners, who have read its
                        // last part by then
                        const bool ok = mbar_wait(BAR(kSReady), (uint32_t)r & 1u, abort_flag);
                        if (!__all_sync(0xFFFFFFFFu, ok)) break;
                    }
                    Sweep w;
                    if (!sweep_chunks(w, grp, P, base, cnt, acc, BAR(kSAccFull + grp), BAR(kSAccFree + grp), acc_par,
                                      BAR(kSEmpty), (uint32_t)(r * cnt), lane, abort_flag)) break;
                    w.zz = grp < cnt ? norm[row] : 0.0f;     // (a group without chunks has nothing inside any window)
                    w.win = 2.125f * (prm.a * sqrtf(w.zz) * 1.0001f + prm.b);
                    const float lim = threshold(w, w.m1, prm);
                    local[(grp - 1) * 128] = Part{w.m1, w.m2, listed(w, lim).word() | (w.m3 <= lim ? 1u << 24 : 0u),
                                                  (uint32_t)w.c1 | ((uint32_t)w.c2 << 16)};
                    __syncwarp();
                    if (lane == 0) mbar_arrive(BAR(kSLocal));
                }
            } else {
                // (the owners hold the residual from the stage end to the next operand and park it during the sweep)
                float z[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) z[i] = z_park[i * kZPitch];
                const float dev = group_deviation(s, z, lane);
                const bool deg = deviation_is_degenerate(dev) || !valid;
                divide_row(z, dev, deg);
                if (valid && (lane & (G - 1)) == 0 && rank == 0) {
                    const uint16_t hb = deviation_is_degenerate(dev) ? (uint16_t)0
                                                                     : __half_as_ushort(__float2half_rn(dev));
                    p.std16[v] = hb;
                    if (deviation_is_degenerate(dev)) ++n_degenerate;
                    else if ((hb & 0x7FFFu) == 0 || (hb & 0x7FFFu) >= 0x7C00u) ++n_stdrange;
                }
                bool ok = true;
#pragma unroll 1
                for (int r = 0; r < R; ++r) {
                    const StageConst prm = sc[r];
                    const float *cbr = p.cb + (size_t)r * s.K * 32;
                    const uint32_t par = (uint32_t)r & 1u;
                    Sweep w;
                    uint32_t ab[32];
                    w.zz = split_operand(z, prm.scale, ab);
                    norm[row] = w.zz;
                    tmem_st32(tmem + lanes + kATmem, ab);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(BAR(kSReady));
                    if (warp == 0 && lane == 0 && ctas > 1)
                        mbar_expect_tx(BAR(kSArrived + par), (uint32_t)ctas * 128u * 16u);
#pragma unroll
                    for (int i = 0; i < 32; ++i) z_park[i * kZPitch] = z[i];
                    w.win = 2.125f * (prm.a * sqrtf(w.zz) * 1.0001f + prm.b);
                    ok = sweep_chunks(w, 0, P, base, cnt, acc, BAR(kSAccFull), BAR(kSAccFree), acc_par, BAR(kSEmpty),
                                      (uint32_t)(r * cnt), lane, abort_flag);
                    if (!ok) break;
                    uint32_t sets;
                    {
                        const float lim = threshold(w, w.m1, prm);
                        sets = listed(w, lim).word() | (w.m3 <= lim ? 1u << 24 : 0u);
                    }
                    // ---- the owners: the CTA's part, to every CTA of the cluster.  A group's sets were taken
                    // against its own minimum, a limit at least as high as the CTA's: they hold every column that
                    // counts.
                    if (P > 1) {
                        ok = mbar_wait(BAR(kSLocal), par, abort_flag);
                        ok = __all_sync(0xFFFFFFFFu, ok);
                        if (!ok) break;
                        const float own = w.m1;
                        Part q[kGroups - 1];
#pragma unroll
                        for (int k = 0; k < kGroups - 1; ++k) {
                            q[k] = k < P - 1 ? local[k * 128] : Part{INFINITY, INFINITY, 0u, 0u};
                            rank_chunk(w, q[k].m1, (int)(q[k].chunks & 0xFFFFu));
                            rank_chunk(w, q[k].m2, (int)(q[k].chunks >> 16));
                        }
                        const float lim = threshold(w, w.m1, prm);
                        sets = own <= lim ? sets : 0u;
#pragma unroll
                        for (int k = 0; k < kGroups - 1; ++k) sets |= q[k].m1 <= lim ? q[k].sets : 0u;
                        sets |= w.m3 <= lim ? 1u << 24 : 0u;
                    }
                    Part best{w.m1, w.m2, sets, (uint32_t)w.c1 | ((uint32_t)w.c2 << 16)};
                    float next = INFINITY;                                   // the second lowest minimum of the parts
                    const Part *mp = parts + par * (kMaxParts * 128) + row;
                    if (ctas > 1) {
#pragma unroll
                        for (int to = 0; to < kMaxParts; ++to)
                            if (to < ctas)
                                asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                                             ::"r"(map_to(mine + par * (uint32_t)(kMaxParts * 128 * 16), (uint32_t)to)),
                                               "r"(__float_as_uint(best.m1)), "r"(__float_as_uint(best.m2)),
                                               "r"(best.sets), "r"(best.chunks),
                                               "r"(map_to(BAR(kSArrived + par), (uint32_t)to)) : "memory");
                        ok = mbar_wait(BAR(kSArrived + par), (uint32_t)(r >> 1) & 1u, abort_flag);
                        ok = __all_sync(0xFFFFFFFFu, ok);
                        if (!ok) break;
                        // merge the parts
                        Part q[kMaxParts];
#pragma unroll
                        for (int k = 0; k < kMaxParts; ++k)
                            q[k] = k < ctas ? mp[k * 128] : Part{INFINITY, INFINITY, 0u, 0u};
                        best = q[0];
#pragma unroll
                        for (int k = 1; k < kMaxParts; ++k) {
                            const bool lower = q[k].m1 < best.m1;
                            next = fminf(next, fmaxf(best.m1, q[k].m1));
                            best.m2 = lower ? q[k].m2 : best.m2;
                            best.sets = lower ? q[k].sets : best.sets;
                            best.chunks = lower ? q[k].chunks : best.chunks;
                            best.m1 = fminf(best.m1, q[k].m1);
                        }
                    }
                    // The column of the lowest score is the choice of nearly every row: its codeword is asked for
                    // before it is known to be.
                    const float m1 = best.m1;
                    const Listed in = listed_of(best.sets);
                    const int j1 = (int)(best.chunks & 0xFFFFu) * 128 + in.column(), jm = min(max(j1, 0), s.K - 1);
                    float ev[32];
                    load_codeword(cbr + (size_t)jm * 32, ev);
                    const float lim = threshold(w, m1, prm);
                    // (a padded column scores 60000: if nothing real scored less, scan everything)
                    const bool scan_all = !(w.zz < 3.6e9f) || !(w.win < INFINITY) || !(m1 < 59000.0f);
                    const bool unique = next > lim && best.m2 > lim && ((best.sets >> 24) & 1u) == 0u &&
                                        in.single() && (uint32_t)j1 < (uint32_t)s.K;
                    int bj = (uint32_t)j1 < (uint32_t)s.K ? j1 : 0;
                    uint32_t todo = __ballot_sync(0xFFFFFFFFu, !deg && (scan_all || !unique));
                    while (todo) {
                        // rows with more than one candidate: the warp compares the listed columns of one row at a
                        // time exactly (lane = column of a block), lowest index on ties
                        const int src = __ffs(todo) - 1;
                        todo &= todo - 1;
                        float zs[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) zs[i] = z_park[i * kZPitch + (src - lane)];
                        const float lim_s = __shfl_sync(0xFFFFFFFFu, lim, src);
                        bool all_s = __shfl_sync(0xFFFFFFFFu, (int)scan_all, src) != 0;
                        // lane k looks at part k of that row
                        Part q{INFINITY, INFINITY, 0u, 0u};
                        if (ctas == 1) {
                            q = Part{__shfl_sync(0xFFFFFFFFu, best.m1, src), __shfl_sync(0xFFFFFFFFu, best.m2, src),
                                     __shfl_sync(0xFFFFFFFFu, best.sets, src), __shfl_sync(0xFFFFFFFFu, best.chunks, src)};
                        } else if (lane < ctas) {
                            q = mp[lane * 128 + (src - lane)];
                        }
                        uint32_t inside = __ballot_sync(0xFFFFFFFFu, lane < ctas && q.m1 <= lim_s);
                        // a third chunk somewhere
                        all_s = all_s || __any_sync(0xFFFFFFFFu, ((inside >> lane) & 1u) && ((q.sets >> 24) & 1u));
                        float bv = INFINITY;
                        int bi = 0x7FFFFFFF;
                        if (all_s) {
                            compare_all(zs, cbr, s.K, lane, bv, bi);
                        } else {
                            const int second = q.m2 <= lim_s ? (int)(q.chunks >> 16) : -1;
                            for (; inside; inside &= inside - 1u) {
                                const int k = __ffs(inside) - 1;
                                compare_listed(zs, cbr, s.K, lane, 32, __shfl_sync(0xFFFFFFFFu, q.sets, k),
                                               (int)(__shfl_sync(0xFFFFFFFFu, q.chunks, k) & 0xFFFFu),
                                               __shfl_sync(0xFFFFFFFFu, second, k),
                                               __shfl_sync(0xFFFFFFFFu, second >= 0 ? 2 : 1, k), bv, bi);
                            }
                        }
                        best_of(32, bv, bi);
                        if (lane == src) {
                            bj = bi < s.K ? bi : 0;
                            if (rank == 0) { if (all_s) ++n_exhaustive; else ++n_rescored; }
                        }
                    }
                    if (deg) bj = 0;
                    if (bj != jm) load_codeword(cbr + (size_t)bj * 32, ev);
                    float e2 = 0.0f;
#pragma unroll
                    for (int i = 0; i < 32; ++i) z[i] = z_park[i * kZPitch];
                    if (!deg) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            z[i] -= ev[i];
                            e2 = fmaf(z[i], z[i], e2);
                        }
                    }
                    __syncwarp();                                    // (the comparison above reads other lanes' rows)
                    if (p.energy && rank == 0) {
                        if (!valid) e2 = 0.0f;
#pragma unroll
                        for (int off = 16; off > 0; off >>= 1) e2 += __shfl_xor_sync(0xFFFFFFFFu, e2, off);
                        if (lane == 0) atomicAdd(p.energy + r, e2);
                    }
                    codes_s[row * 16 + r] = (uint16_t)bj;
                }
                if (ok) {
                    __syncwarp();
                    if (rank == 0) emit_codes(s, codes_s + q4 * 32 * 16, v_first, p.n, lane, p.codes);
                }
            }
        }
        if (p.st) {
            if (n_rescored) atomicAdd(&p.st->rescored_rows, n_rescored);
            if (n_exhaustive) atomicAdd(&p.st->exhaustive_rows, n_exhaustive);
            if (n_degenerate) atomicAdd(&p.st->degenerate_vectors, n_degenerate);
            if (n_stdrange) atomicAdd(&p.st->std_out_of_half, n_stdrange);
        }
    }

    tc_fence_before();
    __syncthreads();
    // (no CTA ends while another may still send to it)
    if (ctas > 1) asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    if (warp == 12) {
        tc_fence_after();
        if (lane == 0 && *abort_flag && p.st) atomicAdd(&p.st->wait_timeouts, 1u);
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

// CTAs per tile; 0: this kernel is not the one to take.  A stage of a tile costs its CTAs about 450 cycles per
// chunk (the chains follow one another), 350 per fold of a group, and 60 per CTA that parts go to, beside 3000
// that do not depend on the split; all tiles have to be on the chip at once.  With more tiles than SMs, two tiles one
// after the other lose to the throughput kernel (2048 codes: 130 us against 101), and so does this kernel with up to
// three chunks (there).
int split_ctas(const Shape &s, int64_t tiles, int sms)
{
    const int S = slots_per_stage(s.K);
    if (S <= kGroups || tiles > sms) return 0;
    int best = 1, least = 1 << 30;
    for (int c = 1; c <= kMaxParts && c <= S; ++c) {
        const int cnt = (S + c - 1) / c, groups = cnt < kGroups ? cnt : kGroups;
        const int cost = 450 * cnt + 350 * ((cnt + groups - 1) / groups) + 60 * c;
        if (cost >= least || tiles * c > sms) continue;
        if (c > 1 && tiles > resident_clusters(reinterpret_cast<const void *>(encode_split_kernel), c, kSplitThreads,
                                               kSplitSmem)) continue;
        best = c;
        least = cost;
    }
    return best;
}

}  // namespace

bool encode_split_wanted(const Shape &s, int64_t n)
{
    if (!encode_tensor_supported(s) || n < 1 || n > (1 << 24)) return false;
    const int sms = sm_count();
    return sms > 0 && split_ctas(s, (n * s.G + 127) / 128, sms) > 0;
}

int launch_encode_split(const Shape &s, const void *x, int64_t n, int64_t stride, const float *cb,
                        const void *prepared, void *codes, uint16_t *std16, rvq_status *st,
                        cudaStream_t stream, float *energy)
{
    const int sms = sm_count();
    const int tiles = (int)((n * s.G + 127) / 128), ctas = split_ctas(s, tiles, sms);
    const void *kernel = reinterpret_cast<const void *>(encode_split_kernel);
    if (ctas <= 0 || !allow_shared_memory(kernel, kSplitSmem)) return RVQ_ERR_LAUNCH;
    const int per = (slots_per_stage(s.K) + ctas - 1) / ctas;
    SplitParams p{s, x, n, stride, cb, reinterpret_cast<const uint8_t *>(prepared), codes, std16, st, energy,
                  per < kGroups ? per : kGroups};
    void *args[] = {&p};
    return launch_clusters(kernel, tiles, ctas, kSplitThreads, kSplitSmem, stream, args);
}

}  // namespace rvq
