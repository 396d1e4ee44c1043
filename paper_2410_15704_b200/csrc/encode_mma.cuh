// What the tensor-core encoders share: mbarriers and bounded waits, tcgen05 operands, chains and
// TMEM reads, the fold of the scores into running minima, the error window, exact distances, and the
// ends of the path (rows in, deviation, operand, codes out).
#pragma once

#include "prepared.cuh"

namespace rvq {

constexpr uint32_t kWaitLimit = 4u * 1000u * 1000u;
// f16 x f16 or e4m3 x e4m3 -> f32, M = N = 128
constexpr uint32_t kChainDesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// The address, in CTA `rank` of the cluster, of what is at `addr` in this one.
__device__ __forceinline__ uint32_t map_to(uint32_t addr, uint32_t rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Bounded wait; returns false (and raises the CTA's abort flag) when it gives up.  A phase that has
// completed already is recognised by the non-blocking test (a plain shared-memory read); only a
// phase still pending goes through the suspending form.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag,
                                          uint32_t limit = kWaitLimit)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
#pragma unroll 1
    for (uint32_t it = 0; it < limit; ++it) {
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
        if ((it & 1023u) == 1023u && *abort_flag) return false;
    }
    *abort_flag = 1u;
    return false;
}

// Wait, when a role ends, for what it has left in flight (a phase of `bar` that a copy or a chain of MMAs will
// complete): shared memory and TMEM stay the CTA's until then, also when its other waits have given up.  With nothing
// in flight, as always at a regular end, this is one test of the barrier.
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity)
{
    uint32_t ok = 0u;
#pragma unroll 1
    for (uint32_t it = 0; it < 100000u && !ok; ++it)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
}

__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    // K-major, no swizzle: 8x16-byte core matrices; LBO steps along the
    // contraction, SBO along rows; descriptor version 1.
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

__device__ __forceinline__ void mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_e4m3_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// One lane of a converged warp, chosen by the hardware.  The compiler knows of this predicate that a
// single lane passes it, and lets the MMA instructions behind it read uniform registers as they are;
// behind `lane == 0` it wraps each of them in a loop over lanes (77 against 39-67 cycles per
// instruction, measured).
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r != 0u;
}

__device__ __forceinline__ float min3(float a, float b, float c)
{
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

#define RVQ_OUT32(u) "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), \
    "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15]), \
    "=r"(u[16]), "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]), "=r"(u[22]), "=r"(u[23]), \
    "=r"(u[24]), "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]), "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
#define RVQ_INOUT32(u) "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]), "+r"(u[7]), \
    "+r"(u[8]), "+r"(u[9]), "+r"(u[10]), "+r"(u[11]), "+r"(u[12]), "+r"(u[13]), "+r"(u[14]), "+r"(u[15]), \
    "+r"(u[16]), "+r"(u[17]), "+r"(u[18]), "+r"(u[19]), "+r"(u[20]), "+r"(u[21]), "+r"(u[22]), "+r"(u[23]), \
    "+r"(u[24]), "+r"(u[25]), "+r"(u[26]), "+r"(u[27]), "+r"(u[28]), "+r"(u[29]), "+r"(u[30]), "+r"(u[31])
#define RVQ_IN32(u) "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(u[5]), "r"(u[6]), "r"(u[7]), \
    "r"(u[8]), "r"(u[9]), "r"(u[10]), "r"(u[11]), "r"(u[12]), "r"(u[13]), "r"(u[14]), "r"(u[15]), \
    "r"(u[16]), "r"(u[17]), "r"(u[18]), "r"(u[19]), "r"(u[20]), "r"(u[21]), "r"(u[22]), "r"(u[23]), \
    "r"(u[24]), "r"(u[25]), "r"(u[26]), "r"(u[27]), "r"(u[28]), "r"(u[29]), "r"(u[30]), "r"(u[31])

// Start loading 32 consecutive TMEM columns of this thread's lane.  The
// registers are not valid until a wait has been given the same array.
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&u)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : RVQ_OUT32(u) : "r"(taddr));
}
// Waits for every tcgen05.ld of this thread; the arrays pass through so that no
// use of them can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_ld_wait4(uint32_t (&u)[32], uint32_t (&v)[32], uint32_t (&w)[32], uint32_t (&x)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" : RVQ_INOUT32(u) : : "memory");
    asm volatile("" : RVQ_INOUT32(v) : : "memory");
    asm volatile("" : RVQ_INOUT32(w) : : "memory");
    asm volatile("" : RVQ_INOUT32(x) : : "memory");
}
__device__ __forceinline__ void tmem_ld_wait2(uint32_t (&u)[32], uint32_t (&v)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" : RVQ_INOUT32(u) : : "memory");
    asm volatile("" : RVQ_INOUT32(v) : : "memory");
}
// The low halves of 64 consecutive columns, two to a register.
__device__ __forceinline__ void tmem_ld64_packed_issue(uint32_t taddr, uint32_t (&u)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.pack::16b.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : RVQ_OUT32(u) : "r"(taddr));
}
// (the wait for it is tmem_st32's)
__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint4 u)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                 : : "r"(taddr), "r"(u.x), "r"(u.y), "r"(u.z), "r"(u.w) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&u)[32])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
                 "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
                 "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
                 : : "r"(taddr), RVQ_IN32(u) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// The constant A operand of the norm's step, (1 1 1 0 ... 0) in every row: eight TMEM columns, written once by the
// four warps that reach the 128 lanes.  (From shared memory the tensor core read 4 KB for it in every chain.)
__device__ __forceinline__ void tmem_ones(uint32_t taddr)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %3, %3, %3, %3, %3};"
                 : : "r"(taddr), "r"(0x3C003C00u), "r"(0x00003C00u), "r"(0u) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Per-row state of one stage's sweep over the scores.
struct Sweep {
    float win;               // error window
    float zz, ll;  // squared norms of the scaled residual (m1 + zz is the best squared distance) and of its remainder
    float m1, m2, m3;        // the three lowest chunk minima ...
    int c1, c2;              // ... and the chunks of the first two
    static constexpr float kPadded = 59000.0f;      // (a padded column scores 60000)
    __device__ __forceinline__ float lowest() const { return m1; }
    __device__ __forceinline__ float second() const { return m2; }
    __device__ __forceinline__ float third() const { return m3; }
    __device__ __forceinline__ int chunk1() const { return c1; }
    __device__ __forceinline__ int chunk2() const { return c2; }
    float hb[8];             // minimum per block of 16 columns inside its 128-column chunk
    float d[16];             // minimum per column position inside its block

    __device__ __forceinline__ void clear()
    {
        m1 = m2 = m3 = INFINITY;
        c1 = c2 = 0;
#pragma unroll
        for (int q = 0; q < 16; ++q) d[q] = INFINITY;
#pragma unroll
        for (int q = 0; q < 8; ++q) hb[q] = INFINITY;
    }
};

// 32 columns of scores (blocks 2 b and 2 b + 1 of their chunk) folded into the running minima of two
// partitions of a chunk's columns: the 16 places inside a block (one three-input minimum takes in the two
// columns of a place) and the eight blocks; `chunk`, the chunk's own minimum, takes them in as well.  Together
// with the chunk list a column that could be the argmin is pinned to (listed chunk) x (block of the
// chunk) x (place): when every one of the three lists has a single entry, to one column.
// 35 minimum operations per 32 scores: they run on the narrow integer/compare pipe, which this sweep
// keeps about as busy as the tensor pipe, so their number per score is what the sweep's speed
// hangs on (36.5 with blocks of 32 columns and their halves as two partitions).
__device__ __forceinline__ void fold_block(Sweep &w, const uint32_t (&u)[32], int b, float &chunk)
{
#pragma unroll
    for (int c = 0; c < 16; ++c) w.d[c] = min3(w.d[c], __uint_as_float(u[c]), __uint_as_float(u[c + 16]));
    float hm[2];
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
        const uint32_t *v = u + 16 * hf;
        const float a0 = min3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
        const float a1 = min3(__uint_as_float(v[3]), __uint_as_float(v[4]), __uint_as_float(v[5]));
        const float a2 = min3(__uint_as_float(v[6]), __uint_as_float(v[7]), __uint_as_float(v[8]));
        const float a3 = min3(__uint_as_float(v[9]), __uint_as_float(v[10]), __uint_as_float(v[11]));
        const float a4 = min3(__uint_as_float(v[12]), __uint_as_float(v[13]), __uint_as_float(v[14]));
        hm[hf] = fminf(min3(a0, a1, a2), min3(a3, a4, __uint_as_float(v[15])));
        w.hb[2 * b + hf] = fminf(w.hb[2 * b + hf], hm[hf]);
    }
    chunk = b == 0 ? fminf(hm[0], hm[1]) : min3(chunk, hm[0], hm[1]);
}

// What a stage's rows need to know of its codebook (prepare.cu), copied to shared memory at the start: asked for in
// the prepared block when it was needed, every stage end waited for it.
struct StageConst {
    float scale, a, b;                      // operand scale; |score error| <= a ||Z|| + b
    float emax, eerr, elo;       // norms, the stage's largest: codeword, what its two halves miss, its remainder half
};
__device__ __forceinline__ void load_stage_consts(const uint8_t *prepared, int R, int tid, StageConst *out)
{
    if (tid < R) {
        const StageParams q = reinterpret_cast<const StageParams *>(prepared + kPreparedParamsOffset)[tid];
        // StageMaxima
        const uint4 m = __ldg(reinterpret_cast<const uint4 *>(prepared + kPreparedMaximaOffset) + tid);
        out[tid] = StageConst{q.scale, q.a, q.b, __uint_as_float(m.x), __uint_as_float(m.y), __uint_as_float(m.w)};
    }
}

// A column can only be the exact-L2 choice (in real arithmetic, and in the float32 direct-form
// arithmetic of the all-float32 kernel, whose relative error on a distance is below 34 * 2^-24) if its
// approximate score is at most threshold(m1): the window covers the approximation error of both
// scores, the last term the float32 evaluation error of both distances (2 * 34 * 2^-24 < 2^-17.5).
// Both columns concerned, the approximate and the exact winner, lie within rho of the row, rho^2 being the
// approximate winner's squared distance, at most m1 + zz + win; so their norms are at most E = ||Z|| + rho,
// and the error bound of prepare.cu, which allows every codeword the largest norm of the stage, is taken
// with E where that is smaller.
// (Roots are the rounded ones: approximate ones save 0.8-2 % on small calls, 300 tokens' keys 46.3 -> 45.4 us, 512
// float32 tokens at 256 codes 26.05 -> 25.8, and 0.3 % on 4096 tokens' keys, 191.3 -> 190.7; they are less exact.)
__device__ __forceinline__ float threshold(const Sweep &w, float m1, const StageConst &sb)
{
    const float nz = sqrtf(w.zz) * 1.0001f, d2 = fmaxf(m1 + w.zz, 0.0f);
    const float e = fminf(sb.emax, (nz + sqrtf(d2 + w.win)) * 1.0001f);
    const float elo = fminf(sb.elo, 4.8828125e-4f * e + 1.7e-7f),
                eerr = fminf(sb.eerr, 2.384185791015625e-7f * e + 1.7e-7f);
    const float a = 2.0f * (4.8828125e-4f * elo + 2.384185791015625e-7f * e + eerr) + 3.814697265625e-6f * e;
    const float b = e * (1.9073486328125e-6f * e + 4.76837158203125e-7f);
    const float win = fminf(w.win, 2.125f * (a * nz + b));
    return m1 + win + 5.4e-6f * (d2 + win);
}

// The same for the chain with 8-bit corrections.  With e4m3's rounding error of at most c = 0.0595 of a value (its
// half unit in the last place, and the rounding of the remainder to a half before it) or 2^-10 near zero, and E as
// above, the dot product is off by at most
//   |z_lo.e - [64 z_lo][e/64]|        <= ||z_lo|| (cE + (1 + c)(cE + 64 sqrt(32) 2^-10)) + sqrt(32) 2^-16 (1 + c) E
//   |z_hi.e_lo - [z_hi/64][64 e_lo]|  <= (cN + 0.354) L + ((1 + c) N + 0.354)(cL + sqrt(32) 2^-16)
// with N = ||z||, L = ||e_lo||, z the row's operand; twice that for the score, plus the accumulation as before (prepare.cu; five
// instructions of two kinds add up no worse than seven of one).  That comes to some 2^-13 |z||e|; the worst of 6.3
// million chains was 3.1e-5 |z||e| on normal data and 1.13e-4 (2^-13.1) with x20 outlier channels.  (c_norm: what multiplies the norm).
__device__ __forceinline__ float window8(float nz, float nl, float e, float c_norm, const StageConst &sb)
{
    constexpr float c = 0.0595f;
    const float elo = fminf(sb.elo + sb.eerr, 4.8828125e-4f * e + 1.7e-7f);
    const float t1 = nl * (c * e + (1.0f + c) * (c * e + 0.354f)) + 8.7e-5f * 1.06f * e;
    const float t2 = (c * nz + 0.354f) * elo + ((1.0f + c) * nz + 0.354f) * (c * elo + 8.7e-5f);
    return 2.125f * (2.0f * (t1 + t2) + 1.9073486328125e-6f * e * (c_norm * e + 2.0f * nz) + 4.76837158203125e-7f * e);
}
__device__ __forceinline__ float threshold8(const Sweep &w, float m1, const StageConst &sb)
{
    const float nz = sqrtf(w.zz) * 1.0001f, nl = sqrtf(w.ll) * 1.0001f, d2 = fmaxf(m1 + w.zz, 0.0f);
    const float full = window8(nz, nl, sb.emax, 1.0f, sb);
    const float win = fminf(full, window8(nz, nl, fminf(sb.emax, (nz + sqrtf(d2 + full)) * 1.0001f), 1.0f, sb));
    return m1 + win + 5.4e-6f * (d2 + win);
}

// Members of the two partitions whose minimum is at most `limit` (bit k: member k).  The comparisons are
// subtractions, on the floating-point pipe; one funnel shift each collects their signs.
struct Listed {
    uint32_t places, blocks;
    __device__ __forceinline__ bool single() const { return ((places & (places - 1u)) | (blocks & (blocks - 1u))) == 0u; }
    // the two in one word: places, blocks << 16
    __device__ __forceinline__ uint32_t word() const { return places | (blocks << 16); }
    // column inside the chunk of the lowest members
    __device__ __forceinline__ int column() const { return (__ffs(blocks) - 1) * 16 + __ffs(places) - 1; }
};
__device__ __forceinline__ Listed listed_of(uint32_t word) { return {word & 0xFFFFu, (word >> 16) & 0xFFu}; }
__device__ __forceinline__ Listed listed(const Sweep &w, float limit)
{
    uint32_t q = 0u, b = 0u;
#pragma unroll
    for (int i = 15; i >= 0; --i) q = __funnelshift_l(__float_as_uint(limit - w.d[i]), q, 1);
#pragma unroll
    for (int i = 7; i >= 0; --i) b = __funnelshift_l(__float_as_uint(limit - w.hb[i]), b, 1);
    return {~q & 0xFFFFu, ~b & 0xFFu};
}

// The minimum `v` of chunk c joins the three lowest chunk minima (a tie stays behind the earlier chunk,
// and so among those that the exact re-scoring compares).
__device__ __forceinline__ void rank_chunk(Sweep &w, float v, int c)
{
    const bool first = v < w.m1, second = v < w.m2;
    w.m3 = fminf(w.m3, fmaxf(w.m2, v));
    w.c2 = second ? (first ? w.c1 : c) : w.c2;
    w.m2 = fminf(w.m2, fmaxf(w.m1, v));
    w.c1 = first ? c : w.c1;
    w.m1 = fminf(w.m1, v);
}

// ---- Scores as 16-bit whole numbers, for the chain with 8-bit corrections.
// The chain's last step, the norm's, also adds 1.5 * 2^22, so that the accumulator's unit is 1/2 and the low sixteen bits
// of its word are the score in that unit: tcgen05.ld packs them in pairs (columns 2k and 2k + 1 in a register), and
// one three-input minimum of pairs folds in four scores.  For that the scores of a row have to lie within [0, 2^15): the
// row's operand and the constants that multiply the norm are scaled by c, and `off` lifts the lowest score
// that the row can have, -c ||Z||^2, to 20 (a score is within c (-||Z||^2 ... emax^2 + 2 ||Z|| emax) of a codeword).
constexpr float kPackedRange = 32000.0f;
// What the last step loses: it cuts its addends to 1/4 and the sum to 1/2, towards zero.  With four addends that are no multiples of
// it the errors of two scores differ by at most 1.5; measured on B200 against float64 sums of the very operands, 9.4
// million chains with 8-bit corrections and without, they lay within -0.81 ... 0.25.
constexpr float kPackedCut = 1.5f;

__device__ __forceinline__ float squared_norm(const float (&z)[32])
{
    float q[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < 32; ++i) q[i & 3] = fmaf(z[i], z[i], q[i & 3]);
    return (q[0] + q[1]) + (q[2] + q[3]);
}

struct PackedSweep {
    static constexpr uint32_t kPadded = 64800u;      // (a padded column scores 65504, no other one above 64100)
    float zz, ll;            // squared norms of the scaled residual, and of the remainder of its operand
    float c, off;            // row scale (a half) and lift (a half)
    uint32_t v1, v2, v3;     // the three lowest chunk minima, each above its chunk's number
    uint32_t hb[8];          // minima per block of 16 columns: of its even columns, and of its odd ones above
    uint32_t d[8];           // minima of places 2k, and of 2k + 1 above

    __device__ __forceinline__ void start(const float (&z)[32], const StageConst &prm)
    {
        zz = squared_norm(z) * prm.scale * prm.scale;
        const float t = prm.emax + sqrtf(zz) * 1.0001f;
        c = __half2float(__float2half_rd(fminf(kPackedRange / (t * t), 16.0f)));
        off = __half2float(__float2half_ru(c * zz + 20.0f));
    }
    // (c c) (c 2048) (off 1) (c 0): what multiplies the norm's three halves, 3072, 1, and a padded column's entries
    __device__ __forceinline__ uint4 row_constants() const
    {
        const uint32_t hc = __half_as_ushort(__float2half_rn(c)), ho = __half_as_ushort(__float2half_rn(off));
        return make_uint4(hc | (hc << 16), hc | (0x6800u << 16), ho | (0x3C00u << 16), hc);
    }
    __device__ __forceinline__ void clear()
    {
        v1 = v2 = v3 = 0xFFFFFFFFu;
#pragma unroll
        for (int q = 0; q < 8; ++q) d[q] = hb[q] = 0xFFFFFFFFu;
    }
    // The minima `low` of chunk k (even columns, odd ones) join the three lowest.
    __device__ __forceinline__ void rank(uint32_t low, int k)
    {
        const uint32_t v = min((low << 16) | (uint32_t)k, (low & 0xFFFF0000u) | (uint32_t)k);
        v3 = min(v3, max(v2, v));
        v2 = min(v2, max(v1, v));
        v1 = min(v1, v);
    }
    __device__ __forceinline__ uint32_t lowest() const { return v1 >> 16; }
    __device__ __forceinline__ uint32_t second() const { return v2 >> 16; }
    __device__ __forceinline__ uint32_t third() const { return v3 >> 16; }
    __device__ __forceinline__ int chunk1() const { return (int)(v1 & 0xFFFFu); }
    __device__ __forceinline__ int chunk2() const { return (int)(v2 & 0xFFFFu); }
};

__device__ __forceinline__ uint32_t threshold8(const PackedSweep &w, uint32_t m1, const StageConst &sb)
{
    const float rz = sqrtf(w.zz) * 1.0001f, nz = w.c * rz, nl = sqrtf(w.ll) * 1.0001f;
    const float d2 = fmaxf(0.5f * (float)m1 - w.off + w.c * w.zz, 0.0f) + 2.0f;
    const float full = window8(nz, nl, sb.emax, w.c, sb) + kPackedCut;
    const float e = fminf(sb.emax, (rz + sqrtf((d2 + full) / w.c)) * 1.0001f);
    const float win = fminf(full, window8(nz, nl, e, w.c, sb) + kPackedCut);
    return min(m1 + (uint32_t)fminf(ceilf(2.0f * (win + 5.4e-6f * (d2 + win))), 65534.0f), 65534u);
}

// 64 columns of scores (half `h` of their chunk) in pairs, folded into the same partitions as in fold_block: 38 minimum
// operations instead of 70.
__device__ __forceinline__ void fold_packed(PackedSweep &w, const uint32_t (&u)[32], int h, uint32_t &chunk)
{
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        w.d[k] = __vimin3_u16x2(w.d[k], u[k], u[k + 8]);
        w.d[k] = __vimin3_u16x2(w.d[k], u[k + 16], u[k + 24]);
    }
    uint32_t m[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const uint32_t *v = u + 8 * b;
        m[b] = __vimin3_u16x2(__vimin3_u16x2(v[0], v[1], v[2]), __vimin3_u16x2(v[3], v[4], v[5]), __vminu2(v[6], v[7]));
        w.hb[4 * h + b] = __vminu2(w.hb[4 * h + b], m[b]);
    }
    chunk = __vimin3_u16x2(__vimin3_u16x2(chunk, m[0], m[1]), m[2], m[3]);
}

// Members whose minimum is at most `limit` (below 65535).
__device__ __forceinline__ Listed listed(const PackedSweep &w, uint32_t limit)
{
    const uint32_t above = (limit + 1u) * 0x10001u;
    // 1 in the half word of a member that is listed
    auto flags = [&](uint32_t v) { return __vminu2(above - __vminu2(v, above), 0x10001u); };
    uint32_t q = 0u, b = 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) q += flags(w.d[k]) << k;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        b += flags(__vminu2(__byte_perm(w.hb[k], w.hb[k + 4], 0x5410), __byte_perm(w.hb[k], w.hb[k + 4], 0x7632))) << k;
    // even places in the low half word, odd ones in the high one: interleaved
    q = (q | (q << 4)) & 0x0F0F0F0Fu;
    q = (q | (q << 2)) & 0x33333333u;
    q = (q | (q << 1)) & 0x55555555u;
    return {(q & 0xFFFFu) | (q >> 15), (b & 0xFu) | (b >> 12)};
}

// 32-byte read-only global load: a codeword row costs four of these, and for
// row-per-lane gathers it is the number of load instructions that the L1 pays for.
__device__ __forceinline__ void ldg256(const float *p, float (&v)[8])
{
    asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
}

__device__ __forceinline__ void load_codeword(const float *__restrict__ e, float (&v)[32])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float part[8];
        ldg256(e + 8 * q, part);
#pragma unroll
        for (int k = 0; k < 8; ++k) v[8 * q + k] = part[k];
    }
}

// Exact squared distance, direct form, same operation order as the scalar kernel.
__device__ __forceinline__ float exact_distance(const float (&z)[32], const float *__restrict__ e)
{
    float acc = 0.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float ev[8];
        ldg256(e + 8 * q, ev);
#pragma unroll
        for (int k = 0; k < 8; ++k) { const float t = z[8 * q + k] - ev[k]; acc = fmaf(t, t, acc); }
    }
    return acc;
}

// Position of set bit number `k` of `bits` (which has that many).
__device__ __forceinline__ int bit_at(uint32_t bits, int k)
{
    for (; k > 0; --k) bits &= bits - 1u;
    return __ffs(bits) - 1;
}

// a / b, rounded down, for 0 <= a < 2^16 and 1 <= b <= 128: the half added keeps the quotient 1 / 256 and more away from a
// whole number, and its error is below 2^-22 of it, 2^-6 at b = 1, where it is a half away.  (An integer division takes some 200 cycles.)
__device__ __forceinline__ int small_quotient(int a, int b) { return (int)(((float)a + 0.5f) * __frcp_rn((float)b)); }

// Exact comparison of the columns listed by `sets` (Listed::word) in `chunks` chunks -- chunk1 and chunk2, or with
// more than two all of a stage --, by `stride` lanes for one row z: lane l takes the l-th column, so that their
// codewords arrive together (one after the other they cost a trip to L2 each: 4400 cycles a row, measured).  The
// lane's best joins (bv, bi).
__device__ __forceinline__ void compare_listed(const float (&z)[32], const float *__restrict__ cbr, int K, int lane, int stride,
                                               uint32_t sets, int chunk1, int chunk2, int chunks, float &bv, int &bi)
{
    const Listed in = listed_of(sets);
    const int nc = __popc(in.places), per = nc * __popc(in.blocks), total = per * chunks;
    for (int l = lane; l < total; l += stride) {
        const int c = small_quotient(l, per), in_chunk = l - c * per, b = small_quotient(in_chunk, nc);
        const int j = (chunks > 2 ? c : c ? chunk2 : chunk1) * 128 + bit_at(in.blocks, b) * 16 +
                      bit_at(in.places, in_chunk - b * nc);
        if (j < K) {
            const float d = exact_distance(z, cbr + (size_t)j * 32);
            if (d < bv || (d == bv && j < bi)) { bv = d; bi = j; }
        }
    }
}

// Exact comparison of all columns.
__device__ __forceinline__ void compare_all(const float (&z)[32], const float *__restrict__ cbr, int K, int lane,
                                            float &bv, int &bi)
{
    for (int j = lane; j < K; j += 32) {
        const float d = exact_distance(z, cbr + (size_t)j * 32);
        if (d < bv) { bv = d; bi = j; }
    }
}

// The best of every `lanes` neighbouring lanes (a power of two), in all of them: smallest distance, lowest index on ties.
__device__ __forceinline__ void best_of(int lanes, float &bv, int &bi)
{
    for (int off = lanes / 2; off > 0; off >>= 1) {
        const float ov = __shfl_xor_sync(0xFFFFFFFFu, bv, off);
        const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, off);
        if (ov < bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
    }
}

// The seven K = 16 steps of one chain: 128 rows (A: TMEM columns a0 ..: 16 of head, 16 of remainder)
// against the 128 codewords of the slot that `bd` describes, scores to the 128 columns from `acc`.  A
// B cell is 128 codewords x 16 bytes = 128 descriptor address units.
__device__ __forceinline__ void issue_chain(uint32_t acc, uint32_t a0, uint64_t bd, uint32_t ones)
{
    mma_f16_ts(acc, a0, bd + 5 * 128, kChainDesc, 0);            // hi[0:16]  . hi cells 5-6
    mma_f16_ts(acc, a0 + 8, bd + 7 * 128, kChainDesc, 1);        // hi[16:32] . hi cells 7-8
    mma_f16_ts(acc, a0, bd, kChainDesc, 1);                      // hi[0:16]  . lo cells 0-1
    mma_f16_ts(acc, a0 + 8, bd + 2 * 128, kChainDesc, 1);        // hi[16:32] . lo cells 2-3
    mma_f16_ts(acc, a0 + 16, bd + 5 * 128, kChainDesc, 1);       // lo[0:16]  . hi cells 5-6
    mma_f16_ts(acc, a0 + 24, bd + 7 * 128, kChainDesc, 1);       // lo[16:32] . hi cells 7-8
    mma_f16_ts(acc, ones, bd + 4 * 128, kChainDesc, 1);     // (1 1 1 0 .. 0) . norm cell 4 (and cell 5 . 0)
}

// The chain with 8-bit corrections, on the last nine cells of a slot: two K = 32 steps of e4m3 (TMEM columns a0 +
// 16 ..: 8 of 64 times the remainder, 8 of a 64th of the head), then heads and norm in half precision.  Five
// steps instead of seven: 327 against 455 cycles (measured).
__device__ __forceinline__ void issue_chain8(uint32_t acc, uint32_t a0, uint64_t bd, uint32_t ones)
{
    mma_e4m3_ts(acc, a0 + 16, bd + 5 * 128, kChainDesc, 0);      // [64 lo]_8    . [e / 64]_8 (cells 9-10 of the slot)
    mma_e4m3_ts(acc, a0 + 24, bd + 7 * 128, kChainDesc, 1);      // [hi / 64]_8  . [64 e_lo]_8 (cells 11-12)
    mma_f16_ts(acc, a0, bd + 1 * 128, kChainDesc, 1);            // hi[0:16]  . hi cells 5-6
    mma_f16_ts(acc, a0 + 8, bd + 3 * 128, kChainDesc, 1);        // hi[16:32] . hi cells 7-8
    mma_f16_ts(acc, ones, bd, kChainDesc, 1);               // (1 1 1 0 .. 0) . norm cell 4 (and cell 5 . 0)
}

// The elements of 16-byte piece `off` of a head vector, widened, to where its group rows stand: element i of group g
// at zv[i * PITCH + g].  PITCH is odd, so that neither the pieces of a vector nor its rows share banks.
template <int PITCH, int N>
__device__ __forceinline__ void scatter_piece(const Shape &s, const float (&val)[N], int off, float *zv)
{
    const int ch = off * N;
    if (s.layout == RVQ_GROUP_CONTIGUOUS) {
        float *p = zv + (ch & 31) * PITCH + (ch >> 5);
#pragma unroll
        for (int u = 0; u < N; ++u) p[u * PITCH] = val[u];
    } else if (s.G == 4) {
        float *p = zv + (ch >> 2) * PITCH;
#pragma unroll
        for (int u = 0; u < N; ++u) p[(u >> 2) * PITCH + (u & 3)] = val[u];
    } else {
        const int lg = __ffs(s.G) - 1;
#pragma unroll
        for (int u = 0; u < N; ++u) zv[((ch + u) >> lg) * PITCH + ((ch + u) & (s.G - 1))] = val[u];
    }
}
template <int PITCH>
__device__ __forceinline__ void scatter_piece(const Shape &s, uint4 raw, int off, float *zv)
{
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
    if (s.dtype == RVQ_F32) {
        const float val[4] = {__uint_as_float(w[0]), __uint_as_float(w[1]), __uint_as_float(w[2]), __uint_as_float(w[3])};
        scatter_piece<PITCH>(s, val, off, zv);
    } else {
        float val[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (s.dtype == RVQ_BF16) {
                val[2 * k] = __uint_as_float(w[k] << 16);
                val[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
            } else {
                const float2 h = __half22float2(*reinterpret_cast<const __half2 *>(&w[k]));
                val[2 * k] = h.x;
                val[2 * k + 1] = h.y;
            }
        }
        scatter_piece<PITCH>(s, val, off, zv);
    }
}
// Piece `off` of head vector v; zeros past the last.
__device__ __forceinline__ uint4 load_piece(const Shape &s, const void *__restrict__ x, int64_t n, int64_t stride,
                                            int64_t v, int off)
{
    if (v >= n) return make_uint4(0u, 0u, 0u, 0u);
    return __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const uint8_t *>(x) + v * stride * s.elem_bytes) + off);
}

// The warp's 32 / G head vectors (1024 elements), from vector v_first on, come in as 16-byte pieces, four loads in
// flight per lane; lane l gets the 32 elements of group l % G of vector l / G, zeros past the last vector.  `rows`:
// element 0 of the warp's first row in a scratch area [32][PITCH].
template <int PITCH>
__device__ __forceinline__ void load_group_rows(const Shape &s, const void *__restrict__ x, int64_t n, int64_t stride,
                                                int64_t v_first, int lane, float *rows, float (&z)[32])
{
    const int lg = __ffs(s.G) - 1, lp = lg + (s.elem_bytes == 4 ? 3 : 2);       // log2 of the pieces of a vector
    for (int c0 = lane; c0 < 32 << (lp - lg); c0 += 128) {
        uint4 raw[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + 32 * u;
            raw[u] = load_piece(s, x, n, stride, v_first + (c >> lp), c & ((1 << lp) - 1));
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + 32 * u;
            scatter_piece<PITCH>(s, raw[u], c & ((1 << lp) - 1), rows + ((c >> lp) << lg));
        }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 32; ++i) z[i] = rows[i * PITCH + lane];
}

// Deviation over the G lanes of this lane's head vector, same summation order as the scalar kernel.
__device__ __forceinline__ float group_deviation(const Shape &s, const float (&z)[32], int lane)
{
    const int base = lane & ~(s.G - 1);                      // (G is a power of two)
    float a = 0.0f;
#pragma unroll
    for (int i = 0; i < 32; ++i) a += z[i];
    float mu = 0.0f;
    for (int k = 0; k < s.G; ++k) mu += __shfl_sync(0xFFFFFFFFu, a, base + k);
    mu /= (float)s.dim;
    float b = 0.0f;
#pragma unroll
    for (int i = 0; i < 32; ++i) b += (z[i] - mu) * (z[i] - mu);
    float ss = 0.0f;
    for (int k = 0; k < s.G; ++k) ss += __shfl_sync(0xFFFFFFFFu, b, base + k);
    return sqrtf(ss / (float)(s.dim - s.ddof));
}

// z[i] / dev, correctly rounded like the scalar kernel's division; zeros for a degenerate row.  Called by a whole
// warp.  With y = RN(1 / dev), a quotient within a few ulps is made exact by q + y (a - q dev), the residual
// being exact in a fused multiply-add (P. Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", 1990), done twice.  That needs every intermediate value to be a normal number;
// rows outside a wide range of exponents are divided one by one, which as a chain of 32 divisions with
// their checks took 3100 cycles.
__device__ __forceinline__ void divide_row(float (&z)[32], float dev, bool deg)
{
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const uint32_t twice = __float_as_uint(z[i]) << 1;               // (the sign gone)
        lo = min(lo, twice - 1u);                                         // (zeros count as large)
        hi = max(hi, twice);
    }
    const bool ordinary = lo >= 2u * 0x21800000u - 1u && hi <= 2u * 0x5D800000u &&
                          dev >= 9.094947e-13f && dev <= 1.0995116e12f;
    if (__all_sync(0xFFFFFFFFu, ordinary || deg)) {                       // 2^-60 .. 2^60 over 2^-40 .. 2^40
        const float b = deg ? 1.0f : dev, y = __frcp_rn(b);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            float q = z[i] * y;
            q = fmaf(fmaf(-q, b, z[i]), y, q);
            q = fmaf(fmaf(-q, b, z[i]), y, q);
            z[i] = deg ? 0.0f : q;
        }
    } else {
#pragma unroll 1
        for (int i = 0; i < 32; ++i) {
            // (rolled: the array is rotated so that its indices stay constants)
            const float q = deg ? 0.0f : z[0] / dev;
#pragma unroll
            for (int k = 0; k < 31; ++k) z[k] = z[k + 1];
            z[31] = q;
        }
    }
}

// A operand row of the residual z: 16 words of half-precision head, 16 of remainder; returns the squared
// norm of the scaled residual.
__device__ __forceinline__ float split_operand(const float (&z)[32], float scale, uint32_t (&ab)[32])
{
    float zz = 0.0f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float z0 = z[2 * i] * scale, z1 = z[2 * i + 1] * scale;
        zz = fmaf(z0, z0, zz); zz = fmaf(z1, z1, zz);
        const __half2 h2 = __floats2half2_rn(z0, z1);
        const float2 hf = __half22float2(h2);
        const __half2 l2 = __floats2half2_rn(z0 - hf.x, z1 - hf.y);
        ab[i] = *reinterpret_cast<const uint32_t *>(&h2);
        ab[16 + i] = *reinterpret_cast<const uint32_t *>(&l2);
    }
    return zz;
}

// The same for the chain with 8-bit corrections: 16 words of head, 8 of 64 times the remainder, 8 of a 64th of the
// head; returns the squared norm of the remainder.
__device__ __forceinline__ uint32_t e4m3x2(__half2 v)
{
    uint16_t d;
    asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(d) : "r"(*reinterpret_cast<const uint32_t *>(&v)));
    return d;
}
__device__ __forceinline__ float split_operand8(const float (&z)[32], float scale, uint32_t (&ab)[32])
{
    float ll = 0.0f;
    const __half2 up = __floats2half2_rn(64.0f, 64.0f), down = __floats2half2_rn(0.015625f, 0.015625f);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        uint32_t lo8[2], hi8[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float z0 = z[4 * i + 2 * h] * scale, z1 = z[4 * i + 2 * h + 1] * scale;
            const __half2 h2 = __floats2half2_rn(z0, z1);
            const float2 hf = __half22float2(h2);
            const float l0 = z0 - hf.x, l1 = z1 - hf.y;
            ll = fmaf(l0, l0, ll); ll = fmaf(l1, l1, ll);
            ab[2 * i + h] = *reinterpret_cast<const uint32_t *>(&h2);
            lo8[h] = e4m3x2(__hmul2(__floats2half2_rn(l0, l1), up));
            hi8[h] = e4m3x2(__hmul2(h2, down));
        }
        ab[16 + i] = __byte_perm(lo8[0], lo8[1], 0x5410);
        ab[24 + i] = __byte_perm(hi8[0], hi8[1], 0x5410);
    }
    return ll;
}

// Codes of the warp's 32 rows (first vector v_first), from codes_s[row of the warp][16], to global memory in
// the configured storage form (Section 3.2).
__device__ __forceinline__ void emit_codes(const Shape &s, const uint16_t *codes_s, int64_t v_first, int64_t n, int lane,
                                           void *__restrict__ codes)
{
    const int G = s.G;
    if (s.bits == 16) {
        const int64_t v = v_first + lane / G;
        if (v < n) {
            uint16_t *o = reinterpret_cast<uint16_t *>(codes) + (v * G + (lane & (G - 1))) * s.R;
            if (s.R == 8) {
                *reinterpret_cast<uint4 *>(o) = *reinterpret_cast<const uint4 *>(codes_s + lane * 16);
            } else {
                for (int r = 0; r < s.R; ++r) o[r] = codes_s[lane * 16 + r];
            }
        }
    } else {
        // the warp holds 32 / G whole head vectors; one 32-bit word per lane and step
        const int words = s.code_bytes / 4, vec_per_warp = 32 / G;
        // quotients as products with 2^20 / d, rounded up: exact while the dividend is below 2^20 / d (here 512 codes
        // of a vector by up to 16 stages, 8192 + 31 bits by up to 16, 256 words by 256); divisions were most of this
        // loop
        const uint32_t by_words = (1u << 20) / (uint32_t)words + 1u, by_bits = (1u << 20) / (uint32_t)s.bits + 1u,
                       by_R = (1u << 20) / (uint32_t)s.R + 1u;
        for (int t = lane; t < vec_per_warp * words; t += 32) {
            const int vl = (int)((uint32_t)t * by_words >> 20), w = t - vl * words;
            const int64_t vv = v_first + vl;
            if (vv >= n) continue;
            uint32_t word = 0;
            const int k_lo = (int)((uint32_t)(32 * w) * by_bits >> 20),
                      k_hi = min(s.per_vector - 1, (int)((uint32_t)(32 * w + 31) * by_bits >> 20));
            for (int k = k_lo; k <= k_hi; ++k) {
                const int gg = (int)((uint32_t)k * by_R >> 20), rr = k - gg * s.R;
                const uint32_t val = codes_s[(vl * G + gg) * 16 + rr];
                const int sh = k * s.bits - 32 * w;
                word |= sh >= 0 ? (val << sh) : (val >> (-sh));
            }
            reinterpret_cast<uint32_t *>(codes)[vv * words + w] = word;
        }
    }
}

}  // namespace rvq
