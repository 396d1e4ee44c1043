// Tensor-core encode for group_dim 32 (Section 2.2, Algorithm 1).
//
// One persistent CTA per SM takes a contiguous run of 128-row tiles and works
// through it in rounds of up to three tiles (one row per thread, 12 epilogue
// warps; rounds are sized evenly, e.g. 7 tiles = 3 + 2 + 2) plus four role
// warps: one MMA issuer per tile (the warp runs its loop as one, a single lane
// issues) and the operand loader.  The role warps give registers up
// (setmaxnreg 40) and the epilogue warps take them (152).
//   - Scores ||e||^2 - 2 z.e of a 128-row tile against 128 codewords are one
//     tcgen05.mma chain (M=128, N=128, seven K=16 steps over the split
//     half-precision operands described in prepare.cu), accumulated in float32
//     in TMEM.
//     EIGHT: the two small products of the split (remainder x head) in e4m3, as two K=32 steps beside
//     three K=16 ones: 327 cycles per chain instead of 455, at an error of up to 2^-13 |z||e| in the score that the
//     window allows for (window8).  For contiguous groups, eight or more chunks and even codebooks (eight_from
//     says why).
//     PACKED: these chains with scores that are read and folded as 16-bit whole numbers, two to a register (PackedSweep):
//     84 minimum operations per chunk and row instead of 140, at an error of 1.5 units of 2^-15 of the range that a
//     row's scores can have.  262144 values, 2048 codes: 2090 -> 1965 us in a burst.
//   - The B operand (128 codewords per slot) streams from the prepared block
//     through a ring of shared-memory slots filled by cp.async.bulk; every
//     slot serves all three tiles.
//   - Epilogue threads read their row's 128 scores with four tcgen05.ld of 32
//     columns issued together, hand the accumulator back to the issuer as soon
//     as they have landed, and fold them afterwards while the next chain runs.
//     The fold keeps running minima over three partitions of the stage's
//     columns: by 128-column chunk (the two lowest chunks and the value of the third), by 16-column block of a
//     chunk, and by place within a block (16 places): 35 minimum
//     operations per 32 scores.  At the stage end the sets of chunks, blocks
//     and places whose minimum lies inside the window bound where the
//     exact argmin can be: when each set has one member the column is known,
//     and its codeword already on the way; otherwise the columns in the product of
//     the sets are compared exactly in float32 against the float32 codebook (direct
//     form, lowest index on ties), up to four rows of a warp at a time with eight lanes or more to each; with
//     a third chunk inside the window, in the listed blocks and places of all chunks.  A full exact scan
//     covers rows whose scores say nothing.  The emitted code is the exact-L2 choice.
//   - The A operand (the residual split into half-precision head and remainder)
//     lives in TMEM next to its tile's scores, so the tensor core fetches only B
//     from shared memory; the constant (1 1 1 0 ...) rows that pick up the
//     squared norms are eight more columns, used by every MMA chain.
//   - The float32 residual lives in registers between stages and is parked in
//     shared memory during a stage's sweep; x is read once and only codes and
//     the half-precision deviation are written.
//   - With the EMA statistics asked for (Section 3), every stage's rows join the bins of their codes:
//     the stage's output, parked for the next sweep, is added by the tile's MMA issuer warp between
//     two chains of that sweep (count x codeword is added back by the caller's finishing kernel); the
//     last stage's input is added by the epilogue warps.
// TMEM columns of tile t: scores [160 t, 160 t + 128), A operand
// [160 t + 128, 160 t + 160) (16 columns of head, 16 of remainder); the constant operand [480, 488) (PACKED: of tile t, [480 + 8 t, 488 + 8 t)).
// Every wait is bounded; a wait that gives up sets status->wait_timeouts, and
// the kernel waits (bounded as well) for its copies and chains in flight and returns.
#include "encode_mma.cuh"

#include <type_traits>

namespace rvq {

namespace {

constexpr int kTiles = 3;
constexpr int kRowsPerPass = 128 * kTiles;
constexpr int kEpiThreads = kRowsPerPass;
constexpr int kThreads = kEpiThreads + 32 * (kTiles + 1);  // + one MMA issuer warp per tile + loader warp
constexpr int kRing = 9;                                  // operand slots in flight
constexpr int kOnesCol = 480;                             // TMEM column of the constant operand (8 columns)
constexpr int kTileCols = 160;                            // TMEM columns per tile: 128 scores + 32 of A operand

constexpr int kOffB = 0;
constexpr int kOffZ = kOffB + kRing * kSlotBytes;                     // parked residuals, float [32][kPitch]
constexpr int kPitch = kRowsPerPass + 1;                              // (odd: scatter_piece)
constexpr int kOffCodes = kOffZ + 32 * kPitch * 4;
constexpr int kOffBars = kOffCodes + kRowsPerPass * 16 * 2;
constexpr int kOffFlags = kOffBars + 256;                   // per row of the round: 1 for a vector's, 0 past the last
constexpr int kOffStages = kOffFlags + kRowsPerPass;                  // StageConst[16]
constexpr int kSmemBytes = kOffStages + 16 * (int)sizeof(StageConst);
constexpr int kDeferMinSlots = 6;                       // chunks a stage needs for its issuers to take the statistics

// Chunks a stage needs for the chain with 8-bit corrections, which is for contiguous groups: it is a tenth faster on
// values (262144 vectors, 2048 codes: 2545 -> 2315 us in a burst, 2928 -> 2625 under the power cap; 524288, 1024
// codes: 2850 -> 2660, 3271 -> 3005; 512 codes: 1950 -> 2020).
// It also needs rounds of three tiles, whose chains queue up at the tensor core: with fewer tiles per SM a chain's
// length is not what a stage waits for, and the added work at the stage end is (values, us, half precision / 8 bits,
// tiles per SM at most: 1024 codes 64 / 75 at two, 122 / 137 at four, 145 / 138 at five; 2048 codes 147 / 156 at
// three, 207 / 191 at four).  With packed scores earlier: 1024 codes 73 / 73 at two, 93 / 90 at three, 129 / 129 at four,
// 145 / 140 at five, 495 / 465 at twenty; 2048 codes 72 / 78 at one, 112 / 107 at two, 143 / 135 at three, 233 / 209 at
// five; 768 codes 110 / 113 at four, 408 / 406 at twenty; 512 codes 51 / 57 at two, 327 / 346 at twenty.
// And it needs rows whose window stays narrow.  With outlier channels 2.2-2.9 % of the rows and stages have more than
// one candidate instead of 0.5 %, and the more the farther the outliers stand out.  The data are not known on the
// host; the codebooks, which follow them, are looked at when they are prepared (PreparedHeader::even: outliers, and
// codewords far smaller than the largest, kMostInverse), and the kernel reads there which chain to take.  131072 vectors, us in a burst, by the kurtosis of the codewords' entries (1024
// codes; 2048 codes; measured with candidates compared row by row): 3: 721 -> 722, 1265 -> 1165; 4.1: 721 -> 744,
// 1261 -> 1204; 4.4: 720 -> 726, 1264 -> 1197; 7.8: 721 -> 762, 1261 -> 1230; 9.3: 718 -> 769, 1259 -> 1273; 13: 720
// -> 768, 1270 -> 1314; 24: 720 -> 807, 1280 -> 1343; 44: 722 -> 904, 1274 -> 1590.  (Under the power cap the shorter
// chain gains another 6-7 % on both.)
// However long the call is: with candidates compared four rows at a time, long calls on heavy-tailed keys gain a
// little while the outlier channels stay moderate, on either kind of groups, but no size bounds what they lose (2048
// codes, 194176 vectors = 41 tiles per SM on contiguous groups, us in a burst, rows compared, by the factor on eight
// outlier channels of 128: 5: 1885 -> 1729, 1.7 %; 20: 1890 -> 1913, 2.8 %; 60: 1881 -> 2244, 4.7 %; 200: 1867 ->
// 3427, 9.9 %; 1000 on four channels: 1872 -> 64295, 45 %; strided groups 20: 1892 -> 1826, 60: 1881 -> 2105, 1000:
// 1885 -> 44969; 1024 codes with statistics, 100 tiles per SM, 1000: 2768 -> 51737 and 2753 -> 27474).
constexpr int kEightMinSlots = 8;
// The smallest PreparedHeader::even with which a call takes them (2: packed scores); 3: none.
inline uint32_t eight_from(const Shape &s, int64_t tiles, int sms)
{
    const int slots = slots_per_stage(s.K);
    if (slots < kEightMinSlots || s.layout != RVQ_GROUP_CONTIGUOUS || s.raw) return 3u;
    return tiles > (int64_t)sms * (slots >= 16 ? 3 : 4) ? 1u : tiles > (int64_t)sms * (slots >= 16 ? 1 : 2) ? 2u : 3u;
}

// Seven steps in half precision; five, with the small products in 8 bits; five, and scores as 16-bit whole numbers.
enum Chain { kHalf, kEight, kPacked };

// barrier slots
constexpr int kBarFull = 0, kBarEmpty = kRing, kBarAReady = 2 * kRing, kBarAccFull = 2 * kRing + kTiles,
              kBarAccFree = 2 * kRing + 2 * kTiles, kNumBars = 2 * kRing + 3 * kTiles;

struct Params {
    Shape s;
    const void *x;
    int64_t n, stride;
    const float *cb;
    const uint8_t *prepared;
    void *codes;
    uint16_t *std16;
    rvq_status *st;
    int tiles;          // 128-row tiles in the whole problem
    uint32_t *stat_cnt; // optional EMA statistics of this batch: counts [R][K] ...
    float *stat_sum;    // ... and sums of the stage inputs [R][K][32]; both null when not wanted
    float *energy;      // optional [R]: sum over the rows of the squared norm of what each stage leaves
    uint32_t wait_limit;   // polls after which a wait gives up (kWaitLimit; smaller only in the timeout self-test)
    int drop_last_chain;   // timeout self-test: 1 = tile 0's issuer leaves out the CTA's very last chain; else 0
    uint32_t eight_from;   // encode_tensor_either_kernel: eight_from
    int defer_stats;       // 1 = the statistics of every stage but the last are added by the MMA issuer warps (below)
};

// The tiles of one CTA: a contiguous run, done in `rounds` rounds of nearly equal size (<= kTiles).
struct Work {
    int first, count, rounds;
    __device__ __forceinline__ int round_size(int k) const { return count / rounds + (k < count % rounds ? 1 : 0); }
    __device__ __forceinline__ int round_first(int k) const
    {
        return first + k * (count / rounds) + min(k, count % rounds);
    }
};

// 16 warps, launched with 128 registers per thread; the four role warps then keep 40 each and the
// twelve epilogue warps take 152 (4 x 40 + 12 x 152 = 1984 of the 2048 per lane).
// EIGHT: the small products in 8 bits (issue_chain8).
// LONE: one tile per CTA, of up to three chunks a stage, without statistics.  The other tiles' accumulators take the
// tile's second and third chunk, whose chains go out behind the first's at once instead of after its fold; all warps
// take part in the way in.
// (4096 float32 vectors at 256 codes 27.8 -> 24.9 us, at 384 34.1 -> 30.5.  The split encoder with a CTA per tile
// takes 30.8 and 35.7: with up to three chunks the parts' join costs more than the folds that it puts side by side.)
template <int CHAIN, bool LONE>
__device__ __forceinline__ void encode_tensor_body(const Params &p)
{
    constexpr bool EIGHT = CHAIN != kHalf, PACKED = CHAIN == kPacked;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kOffBars);
    uint32_t *tmem_word = reinterpret_cast<uint32_t *>(smem + kOffBars + kNumBars * 8);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + kOffBars + kNumBars * 8 + 4);

    const Shape &s = p.s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int S = slots_per_stage(s.K);
    Work work;
    {
        const int per = p.tiles / (int)gridDim.x, rem = p.tiles % (int)gridDim.x, b = (int)blockIdx.x;
        work.count = per + (b < rem ? 1 : 0);
        work.first = b * per + min(b, rem);
        work.rounds = (work.count + kTiles - 1) / kTiles;
    }
    const int my_passes = work.rounds;
    StageConst *sc = reinterpret_cast<StageConst *>(smem + kOffStages);
    const uint8_t *image = p.prepared + kPreparedImageOffset + (EIGHT ? kSlotTail : 0);
    uint4 raw[3];
    const int lg = __ffs(s.G) - 1, lp = lg + (s.elem_bytes == 4 ? 3 : 2);      // log2 of a vector's groups and pieces
    const int pieces = 128 << (lp - lg);
    if (LONE) {
        const int64_t v_tile = ((int64_t)blockIdx.x * 128) >> lg;
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            const int k = tid + kEpiThreads * u;
            if (tid < kEpiThreads && k < pieces)
                raw[u] = load_piece(s, p.x, p.n, p.stride, v_tile + (k >> lp), k & ((1 << lp) - 1));
        }
    }
    const uint32_t bar0 = smem_u32(bars);
    auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };

    if (tid == 0) {
        for (int i = 0; i < kRing; ++i) {
            mbar_init(BAR(kBarFull + i), 1); mbar_init(BAR(kBarEmpty + i), LONE ? 1 : kTiles);
        }
        for (int t = 0; t < kTiles; ++t) {
            mbar_init(BAR(kBarAReady + t), 4); mbar_init(BAR(kBarAccFull + t), 1); mbar_init(BAR(kBarAccFree + t), 4);
        }
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kEpiThreads / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_word)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    load_stage_consts(p.prepared, s.R, tid, sc);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_word;
    // the constant A operand, shared by all tiles (the issuers hear of it with their first A operand)
    // (PACKED: a tile's own, written again in every stage)
    if (warp < (PACKED ? 4 * kTiles : 4)) tmem_ones(tmem + ((uint32_t)((warp & 3) * 32) << 16) + kOnesCol + 8 * (warp >> 2));
    if (LONE) {
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            const int k = tid + kEpiThreads * u;
            if (tid < kEpiThreads && k < pieces)
                scatter_piece<kPitch>(s, raw[u], k & ((1 << lp) - 1),
                                      reinterpret_cast<float *>(smem + kOffZ) + ((k >> lp) << lg));
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    // The four role warps need few registers; their share goes to the
    // epilogue warps, which hold the four 32-column blocks of a chunk's scores at a time
    // (12 warps x 32 x 152 + 4 warps x 32 x 40 = 63488 of the 65536 the block was launched with).
    if (warp >= kEpiThreads / 32) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == kEpiThreads / 32 + kTiles) {
            // ------------------------------------------------------------ operand loader
            // One thread streams the B slots of every (pass, stage) through the ring; a slot is
            // free again once the MMA chains of all tiles that read it have completed.
            if (lane == 0 && my_passes > 0) {
                const uint32_t total = (uint32_t)my_passes * (uint32_t)s.R * (uint32_t)S;
                const uint32_t per_pass = (uint32_t)s.R * (uint32_t)S;
                uint32_t slot = 0, rs = 0, empty_par = 1;          // parity of the previous completion of empty[slot]
                uint32_t nl = 0;
                int pass = 0;
                for (; nl < total; ++nl) {
                    if (rs == (uint32_t)S && pass + 1 < my_passes) {
                        // the next round's head vectors into L2, while this round's stages run
                        const int64_t v0 = (int64_t)work.round_first(pass + 1) * 128 / s.G;
                        int64_t left = (int64_t)work.round_size(pass + 1) * 128 / s.G;
                        left = v0 + left <= p.n ? left : p.n - v0;
                        const bool dense = p.stride == s.dim;
                        const uint32_t bytes = (uint32_t)(s.dim * s.elem_bytes) * (dense ? (uint32_t)left : 1u);
                        const uint8_t *from = reinterpret_cast<const uint8_t *>(p.x) + v0 * p.stride * s.elem_bytes;
                        for (int64_t k = 0; k < (dense ? 1 : left); ++k, from += p.stride * s.elem_bytes)
                            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(from), "r"(bytes) : "memory");
                    }
                    if (nl >= (uint32_t)kRing && !mbar_wait(BAR(kBarEmpty + slot), empty_par, abort_flag)) break;
                    mbar_expect_tx(BAR(kBarFull + slot), kSlotBytes);
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(smem_u32(smem + kOffB) + slot * (uint32_t)kSlotBytes),
                                   "l"(image + (size_t)rs * kSlotStride), "r"((uint32_t)kSlotBytes),
                                   "r"(BAR(kBarFull + slot)) : "memory");
                    if (++rs == per_pass) { rs = 0; ++pass; }
                    if (++slot == (uint32_t)kRing) { slot = 0; empty_par ^= 1u; }
                }
                for (uint32_t k = nl > (uint32_t)kRing ? nl - kRing : 0u; k < nl; ++k)
                    mbar_drain(BAR(kBarFull + (int)(k % kRing)), (k / kRing) & 1u);
            }
        } else {
            // ------------------------------------------------------------ MMA issuer of tile t
            // A warp per tile, so that the tiles' waits overlap.
            // Whatever it does between two tcgen05.mma chains delays its tile, so descriptors
            // are built once and all counters advance by increments.
            // (The whole warp runs the loop with warp-uniform values and one lane issues: operands that the
            // compiler knows to be uniform can stay in uniform registers, which tcgen05.mma reads directly.)
            if (LONE) {
                if (warp == kEpiThreads / 32) {
                    const uint64_t bdesc0 = make_smem_desc(smem_u32(smem + kOffB), kSlotCodewords * 16, 128);
                    int sent = 0;                                             // chains
                    bool ok = true;
                    for (int r = 0; r < s.R && ok; ++r) {
                        const uint32_t use0 = (uint32_t)(r * S);
                        for (int c = 0; c < S && ok; ++c)
                            ok = mbar_wait(BAR(kBarFull + (int)((use0 + c) % kRing)), ((use0 + c) / kRing) & 1u, abort_flag);
                        if (ok) ok = mbar_wait(BAR(kBarAReady), (uint32_t)r & 1u, abort_flag);
                        ok = __all_sync(0xFFFFFFFFu, ok);
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll 1
                        for (int k = 0; k < S; ++k, ++sent) {
                            if (p.drop_last_chain && r == s.R - 1 && k == S - 1) break;
                            if (elect_one()) {
                                issue_chain(tmem + (uint32_t)(k * kTileCols), tmem + 128,
                                            bdesc0 + (uint64_t)((use0 + k) % kRing * (uint32_t)(kSlotBytes >> 4)),
                                            tmem + kOnesCol);
                                mma_commit(BAR(kBarAccFull + k));
                            }
                            __syncwarp();
                        }
                    }
                    for (int k = max(sent - S, 0); k < sent; ++k)
                        mbar_drain(BAR(kBarAccFull + k % S), (uint32_t)(k / S) & 1u);
                }
            } else if (my_passes > 0) {
                const int t = __shfl_sync(0xFFFFFFFFu, warp, 0) - kEpiThreads / 32;
                const uint32_t total = (uint32_t)my_passes * (uint32_t)s.R * (uint32_t)S;
                const uint64_t bdesc0 = make_smem_desc(smem_u32(smem + kOffB), kSlotCodewords * 16, 128);
                const uint32_t acc = tmem + t * kTileCols, a0 = acc + 128;
                const uint32_t bar_ready = BAR(kBarAReady + t), bar_free = BAR(kBarAccFree + t),
                               bar_acc = BAR(kBarAccFull + t);
                const uint32_t per_round = (uint32_t)s.R * (uint32_t)S;
                uint32_t slot = 0, full_par = 0, s_in = 0, ready_par = 0, free_par = 1, in_round = 0, stage = 0;
                int round = 0;
                // Deferred statistics (Section 3's EMA sums): while stage r+1 is swept, its input z_{r+1} -- what
                // stage r left -- sits parked in shared memory, and this warp, idle between two chains, adds it to
                // the bins of the stage-r codes, one group of 32 rows after each of the chains 1..4 of the stage.
                // The sum of a bin's stage-r INPUTS is that plus count * codeword (z_r = z_{r+1} + C_r[j]), which the
                // caller adds afterwards.  Ordering: the epilogue parks z_{r+1} and has written the stage-r codes
                // before it hands chunk 0's accumulator back, which this warp has waited for before chain 1; and it
                // cannot finish the stage, and park anew, before the chains that this warp issues after the
                // additions.
                const float *zp = reinterpret_cast<const float *>(smem + kOffZ);
                const uint16_t *codes_s = reinterpret_cast<const uint16_t *>(smem + kOffCodes);
                const uint8_t *flags_s = smem + kOffFlags;
                bool ok = true, first = true, active = t < work.round_size(0);
                uint32_t last_par = 1;                                   // parity of this tile's last chain
                for (uint32_t q = 0; q < total && ok; ++q) {
                    ok = mbar_wait(BAR(kBarFull + slot), full_par, abort_flag);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!active) {
                        // this tile sits the round out, but the slot still waits for its release
                        if (ok && lane == 0) mbar_arrive(BAR(kBarEmpty + slot));
                        if (++slot == (uint32_t)kRing) { slot = 0; full_par ^= 1u; }
                        if (++in_round == per_round) {
                            in_round = 0; ++round; active = round < work.rounds && t < work.round_size(round);
                        }
                        continue;                  // (an idle round keeps `stage` at 0: it is only read while active)
                    }
                    if (ok && s_in == 0) ok = mbar_wait(bar_ready, ready_par, abort_flag);
                    if (ok && !first) ok = mbar_wait(bar_free, free_par, abort_flag);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                    first = false;
                    tc_fence_after();
                    const uint64_t bd = bdesc0 + (uint64_t)(slot * (uint32_t)(kSlotBytes >> 4));
                    // (self-test of the give-up path: the chain that nothing comes after is left out, so that the
                    // epilogue's wait for it runs out with no copy or MMA of this CTA still in flight)
                    if (p.drop_last_chain && t == 0 && q == total - 1) break;
                    if (elect_one()) {
                        if (EIGHT) issue_chain8(acc, a0, bd, tmem + kOnesCol + (PACKED ? 8 * t : 0));
                        else issue_chain(acc, a0, bd, tmem + kOnesCol);
                        mma_commit(bar_acc);
                        mma_commit(BAR(kBarEmpty + slot));
                    }
                    __syncwarp();
                    last_par ^= 1u;
                    if (p.defer_stats && stage >= 1u && s_in >= 1u && s_in <= 4u) {
                        const int rl = t * 128 + (int)(s_in - 1u) * 32 + lane;
                        if (flags_s[rl]) {
                            const size_t bin = (size_t)(stage - 1u) * s.K + codes_s[rl * 16 + (int)(stage - 1u)];
                            atomicAdd(p.stat_cnt + bin, 1u);
                            float4 *m = reinterpret_cast<float4 *>(p.stat_sum + bin * 32);
#pragma unroll
                            for (int q4 = 0; q4 < 8; ++q4)
                                atomicAdd(m + q4, make_float4(zp[(4 * q4) * kPitch + rl], zp[(4 * q4 + 1) * kPitch + rl],
                                                              zp[(4 * q4 + 2) * kPitch + rl], zp[(4 * q4 + 3) * kPitch + rl]));
                        }
                        __syncwarp();
                    }
                    free_par ^= 1u;
                    if (++slot == (uint32_t)kRing) { slot = 0; full_par ^= 1u; }
                    if (++s_in == (uint32_t)S) { s_in = 0; ready_par ^= 1u; ++stage; }
                    if (++in_round == per_round) {
                        in_round = 0; stage = 0; ++round; active = round < work.rounds && t < work.round_size(round);
                    }
                }
                mbar_drain(bar_acc, last_par);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue warps
        asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
        const int tile = warp >> 2, q4 = warp & 3;
        const int rloc = tile * 128 + q4 * 32 + lane;
        const uint32_t taddr = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(tile * kTileCols);
        float *z_park = reinterpret_cast<float *>(smem + kOffZ) + rloc;                    // [i][row]
        uint16_t *codes_s = reinterpret_cast<uint16_t *>(smem + kOffCodes);                // [row][R]
        const int G = s.G;
        uint32_t chunk_use = 0;
        int slot = 0;
        uint32_t n_rescored = 0, n_exhaustive = 0, n_degenerate = 0, n_stdrange = 0;
        bool ok = true;

        for (int pass = 0; pass < my_passes && ok; ++pass) {
            if (tile >= work.round_size(pass)) continue;            // this tile sits the round out
            const int64_t row0 = (int64_t)(work.round_first(pass) + tile) * 128;   // first row of this tile
            const int64_t grow = row0 + q4 * 32 + lane;
            const int64_t v = grow / G;
            const int g = (int)(grow - v * G);
            const bool valid = v < p.n;

            // (through the warp's share of the parking area)
            float z[32];
            if (LONE) {
#pragma unroll
                for (int i = 0; i < 32; ++i) z[i] = z_park[i * kPitch];
            } else {
                load_group_rows<kPitch>(s, p.x, p.n, p.stride, (row0 + q4 * 32) / G, lane, z_park - lane, z);
            }
            const float dev = group_deviation(s, z, lane);
            // (raw rows are stage inputs already: taken as they are, no deviation stored)
            const bool deg = s.raw ? !valid : (deviation_is_degenerate(dev) || !valid);
            if (p.defer_stats) smem[kOffFlags + rloc] = valid ? 1 : 0;
            if (!s.raw) {
                divide_row(z, dev, deg);
            } else if (deg) {
#pragma unroll
                for (int i = 0; i < 32; ++i) z[i] = 0.0f;
            }
            if (valid && g == 0 && !s.raw) {
                const uint16_t hb = deviation_is_degenerate(dev) ? (uint16_t)0 : __half_as_ushort(__float2half_rn(dev));
                p.std16[v] = hb;
                if (deviation_is_degenerate(dev)) ++n_degenerate;
                else if ((hb & 0x7FFFu) == 0 || (hb & 0x7FFFu) >= 0x7C00u) ++n_stdrange;
            }

#pragma unroll 1
            for (int r = 0; r < s.R && ok; ++r) {
                const StageConst prm = sc[r];
                const float *cbr = p.cb + (size_t)r * s.K * 32;
                // scaled half-precision copy of the residual -> A operand row; error window of this row
                uint32_t ab[32];
                std::conditional_t<PACKED, PackedSweep, Sweep> w;
                if constexpr (PACKED) {
                    w.start(z, prm);
                    w.ll = split_operand8(z, prm.scale * w.c, ab);
                    tmem_st4(tmem + ((uint32_t)(q4 * 32) << 16) + kOnesCol + 8 * tile, w.row_constants());
                } else if (EIGHT) {
                    w.zz = squared_norm(z) * prm.scale * prm.scale;
                    w.ll = split_operand8(z, prm.scale, ab);
                } else {
                    w.zz = split_operand(z, prm.scale, ab);
                }
                tmem_st32(taddr + 128, ab);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(BAR(kBarAReady + tile));
                // park the float32 residual in shared memory for the sweep
#pragma unroll
                for (int i = 0; i < 32; ++i) z_park[i * kPitch] = z[i];
                // 2 * bound, with slack for this arithmetic
                if constexpr (!EIGHT) w.win = 2.125f * (prm.a * sqrtf(w.zz) * 1.0001f + prm.b);
                w.clear();
                // (no entry reaches 60000 in half precision; none is above 2^14, where 64 times its remainder leaves
                // the 8-bit range)
                bool force_scan;
                if constexpr (EIGHT) force_scan = !(w.zz < 2.68e8f) || !(prm.a < INFINITY);
                else force_scan = !(w.zz < 3.6e9f) || !(w.win < INFINITY);

#pragma unroll 1
                for (int c = 0; c < S && ok; ++c) {
                    ok = LONE ? mbar_wait(BAR(kBarAccFull + c), (uint32_t)r & 1u, abort_flag, p.wait_limit)
                              : mbar_wait(BAR(kBarAccFull + tile), chunk_use & 1u, abort_flag, p.wait_limit);
                    ok = __all_sync(0xFFFFFFFFu, ok);          // tcgen05.ld below needs the whole warp
                    ++chunk_use;
                    if (!ok) break;
                    if (LONE) {
                        if (tid == 0) mbar_arrive(BAR(kBarEmpty + slot));       // the chain has read its slot
                        slot = slot + 1 < kRing ? slot + 1 : 0;
                    }
                    tc_fence_after();
                    // All four 32-column blocks are asked for at once and the accumulator goes back to
                    // the MMA issuer as soon as they have landed: the reduction below runs while the
                    // next chain computes.
                    const uint32_t acc = LONE ? taddr + (uint32_t)(c * kTileCols) : taddr;
                    if constexpr (PACKED) {
                        uint32_t ua[32], ub[32];
                        tmem_ld64_packed_issue(acc, ua);
                        tmem_ld64_packed_issue(acc + 64, ub);
                        tmem_ld_wait2(ua, ub);
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(BAR(kBarAccFree + tile));      // the accumulator may be overwritten
                        uint32_t lowest = 0xFFFFFFFFu;
                        fold_packed(w, ua, 0, lowest);
                        fold_packed(w, ub, 1, lowest);
                        w.rank(lowest, c);
                    } else {
                        uint32_t ua[32], ub[32], uc[32], ud[32];
                        tmem_ld32_issue(acc, ua);
                        tmem_ld32_issue(acc + 32, ub);
                        tmem_ld32_issue(acc + 64, uc);
                        tmem_ld32_issue(acc + 96, ud);
                        tmem_ld_wait4(ua, ub, uc, ud);
                        tc_fence_before();
                        __syncwarp();
                        if (!LONE && lane == 0) mbar_arrive(BAR(kBarAccFree + tile));
                        float lowest;
                        fold_block(w, ua, 0, lowest);
                        fold_block(w, ub, 1, lowest);
                        fold_block(w, uc, 2, lowest);
                        fold_block(w, ud, 3, lowest);
                        rank_chunk(w, lowest, c);
                    }
                }
                if (!ok) break;
                // The column of the lowest score is the choice of nearly every row: its codeword is asked for before
                // it is known to be (the trip to L2 takes as long as the rest of the stage end: asked for after it,
                // 225 -> 217 us on 32768 keys, 30.7 -> 28.2 on 4096 float32 vectors with 256 codes; a prefetch of the
                // running winner into L1 before the last chunk, on top of this, costs 1.2 %).
                const auto m1 = w.lowest();
                const int c1 = w.chunk1(), c2 = w.chunk2();
                const int jm = min(max(c1 * 128 + listed(w, m1).column(), 0), s.K - 1);
                float ev[32];
                load_codeword(cbr + (size_t)jm * 32, ev);

                // ---- stage end: the columns that can still be the exact argmin are those of a listed
                // chunk, in a listed block of the chunk, at a listed place.  When each of
                // the three lists has one entry (almost always) that column is the choice: every other
                // column is farther than the approximation and float32 evaluation errors can bridge.
                const auto lim = [&] {
                    if constexpr (EIGHT) return threshold8(w, m1, sc[r]);
                    else return threshold(w, m1, sc[r]);
                }();
                const Listed in = listed(w, lim);
                const int j1 = c1 * 128 + in.column();
                // (if nothing real scored less than a padded column, scan everything)
                const bool scan_all = force_scan || !(m1 < w.kPadded);
                // with columns inside the window (three or more: taken as all)
                const int chunks = w.third() <= lim ? S : w.second() <= lim ? 2 : 1;
                const bool unique = chunks == 1 && in.single() && (uint32_t)j1 < (uint32_t)s.K;
                const bool flagged = !deg && (scan_all || !unique);
                int bj = (uint32_t)j1 < (uint32_t)s.K ? j1 : 0;
                // Rows with more than one candidate: their candidate columns are compared
                // exactly in float32, direct form: smallest distance, lowest index on ties.  Four rows at a time,
                // eight lanes to a row, or fewer with more; rows whose scores say nothing one by one, all columns, by the whole warp.
                // (One row at a time, and all columns also where a third chunk came inside the window: 32768 keys 219
                // -> 215 us, 262144 values 2515 -> 2495.  All lanes for a single row, half for two, and no integer
                // divisions: 65536 values with one group of four 10 times smaller 609 -> 570, in a burst.)
                uint32_t scans = __ballot_sync(0xFFFFFFFFu, flagged && scan_all);
                uint32_t todo = __ballot_sync(0xFFFFFFFFu, flagged) & ~scans;
                while (todo | scans) {
                    float zs[32], bv = INFINITY;
                    int bi = 0x7FFFFFFF;
                    if (scans) {
                        const int src = __ffs(scans) - 1;
                        scans &= scans - 1u;
#pragma unroll
                        for (int i = 0; i < 32; ++i) zs[i] = z_park[i * kPitch + (src - lane)];
                        compare_all(zs, cbr, s.K, lane, bv, bi);
                        best_of(32, bv, bi);
                        if (lane == src) { bj = bi < s.K ? bi : 0; ++n_exhaustive; }
                        continue;
                    }
                    // a warp's lanes for one row, half of them each for two, a quarter each for more: this lane's row
                    const int share = (todo & (todo - 1u)) == 0u ? 5 : __popc(todo) == 2 ? 4 : 3;
                    int src = __ffs(todo) - 1;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (k <= (lane >> share) && todo) src = __ffs(todo) - 1;
                        todo &= todo - 1u;
                    }
#pragma unroll
                    for (int i = 0; i < 32; ++i) zs[i] = z_park[i * kPitch + (src - lane)];
                    compare_listed(zs, cbr, s.K, lane & ((1 << share) - 1), 1 << share, __shfl_sync(0xFFFFFFFFu, in.word(), src),
                                   __shfl_sync(0xFFFFFFFFu, c1, src), __shfl_sync(0xFFFFFFFFu, c2, src),
                                   __shfl_sync(0xFFFFFFFFu, chunks, src), bv, bi);
                    best_of(1 << share, bv, bi);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int row = __shfl_sync(0xFFFFFFFFu, src, 8 * k), best = __shfl_sync(0xFFFFFFFFu, bi, 8 * k);
                        if (lane == row) bj = best < s.K ? best : 0;
                    }
                }
                if (flagged && !scan_all) ++n_rescored;
                if (deg) bj = 0;
                if (bj != jm) load_codeword(cbr + (size_t)bj * 32, ev);
                // take the residual back
#pragma unroll
                for (int i = 0; i < 32; ++i) z[i] = z_park[i * kPitch];
                if (p.stat_sum && valid && !(p.defer_stats && r < s.R - 1)) {
                    // EMA statistics (Section 3): this row's stage input joins the bin of its code
                    // (all stages but the last are the issuer warps' when deferred)
                    const size_t bin = (size_t)r * s.K + bj;
                    atomicAdd(p.stat_cnt + bin, 1u);
                    float4 *m = reinterpret_cast<float4 *>(p.stat_sum + bin * 32);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        atomicAdd(m + q, make_float4(z[4 * q], z[4 * q + 1], z[4 * q + 2], z[4 * q + 3]));
                }
                // (a degenerate row's codes are 0 whatever its residual, which starts from zero and matters to the
                // statistics only)
                if (!deg || (p.stat_sum && valid)) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) z[i] -= ev[i];
                }
                if (p.energy) {
                    // squared norm of the residual leaving this stage (scaled units), summed over the
                    // warp's rows: one atomic per warp and stage
                    float e2 = 0.0f;
#pragma unroll
                    for (int i = 0; i < 32; ++i) e2 = fmaf(z[i], z[i], e2);
                    if (deg) e2 = 0.0f;
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) e2 += __shfl_xor_sync(0xFFFFFFFFu, e2, off);
                    if (lane == 0) atomicAdd(p.energy + r, e2);
                }
                codes_s[rloc * 16 + r] = (uint16_t)bj;
            }
            if (!ok) break;

            // ---- emit the codes of this pass (Section 3.2 storage)
            __syncwarp();
            emit_codes(s, codes_s + (rloc - lane) * 16, (row0 + q4 * 32) / G, p.n, lane, p.codes);
            __syncwarp();
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
    if (warp == kEpiThreads / 32) {
        tc_fence_after();
        if (lane == 0 && *abort_flag && p.st) atomicAdd(&p.st->wait_timeouts, 1u);
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

__global__ void __launch_bounds__(kThreads, 1) encode_tensor_kernel(const __grid_constant__ Params p)
{
    encode_tensor_body<kHalf, false>(p);
}
__global__ void __launch_bounds__(kThreads, 1) encode_tensor_lone_kernel(const __grid_constant__ Params p)
{
    encode_tensor_body<kHalf, true>(p);
}

// Where the 8-bit corrections are possible: by the codebooks.
__global__ void __launch_bounds__(kThreads, 1) encode_tensor_either_kernel(const __grid_constant__ Params p)
{
    const uint32_t even = reinterpret_cast<const PreparedHeader *>(p.prepared)->even;
    if (even < p.eight_from) encode_tensor_body<kHalf, false>(p);
    else if (even == 1u) encode_tensor_body<kEight, false>(p);
    else encode_tensor_body<kPacked, false>(p);
}

}  // namespace

bool encode_tensor_supported(const Shape &s)
{
    return s.gd == 32 && s.G <= 32 && (s.G & (s.G - 1)) == 0 && slots_per_stage(s.K) * 4 <= 65535;
}

// Stages 0 .. this - 1 of the fused statistics hold the sums of what those stages LEFT (their bins' inputs
// minus count * codeword): the caller adds count * codeword (launch_stats_finish).
int encode_tensor_deferred_stages(const Shape &s)
{
    return encode_tensor_supported(s) && slots_per_stage(s.K) >= kDeferMinSlots && s.R > 1 ? s.R - 1 : 0;
}

int launch_encode_tensor(const Shape &s, const void *x, int64_t n, int64_t stride, const float *cb,
                         const void *prepared, void *codes, uint16_t *std16, rvq_status *st,
                         cudaStream_t stream, uint32_t *stat_cnt, float *stat_sum, float *energy,
                         uint32_t wait_limit, int drop_last_chain)
{
    if (n == 0) return RVQ_OK;
    const int64_t rows = n * s.G;
    const int64_t tiles = (rows + 127) / 128;
    if (tiles > 0x7FFFFFFF) return RVQ_ERR_UNSUPPORTED;
    const int sms = sm_count();
    if (sms <= 0) return RVQ_ERR_DEVICE;
    const bool lone = tiles <= sms && slots_per_stage(s.K) <= kTiles && !s.raw && !stat_sum;
    const uint32_t from = eight_from(s, tiles, sms);
    auto kernel = lone ? encode_tensor_lone_kernel
                : from < 3u ? encode_tensor_either_kernel : encode_tensor_kernel;
    if (!allow_shared_memory(reinterpret_cast<const void *>(kernel), kSmemBytes)) return RVQ_ERR_LAUNCH;
    Params p{s, x, n, stride, cb, reinterpret_cast<const uint8_t *>(prepared), codes, std16, st, (int)tiles,
             stat_cnt, stat_sum, energy, wait_limit ? wait_limit : kWaitLimit, drop_last_chain, from,
             stat_sum != nullptr && encode_tensor_deferred_stages(s) > 0 ? 1 : 0};
    // (fewer tiles than three per SM: one or two in each, not three in some)
    const int grid = (int)(tiles < sms ? tiles : sms);
    kernel<<<grid, kThreads, kSmemBytes, stream>>>(p);
    return check_launch();
}

}  // namespace rvq
