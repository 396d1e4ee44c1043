// extern "C" boundary of the RVQ library: argument checks on the host, then
// dispatch to the kernels.  No allocation, no synchronisation.  Process-wide
// state: the launch counter below, and what is remembered about each device (its
// SM count) and each context (the shared memory granted to each kernel, resident
// clusters, the address of the built-in scratch array of rvq_ema_update_static).
#include "prepared.cuh"
#include "rvq_selftest.h"

#include <cuda.h>

#include <atomic>

namespace rvq {

static std::atomic<uint64_t> g_launches{0};
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

namespace {

constexpr int kMaxDevices = 64;
std::atomic<int> g_sms[kMaxDevices];

// What has been asked of the runtime about a kernel so far, per context: the largest dynamic shared memory
// granted to it, and how many clusters of 1 .. 8 CTAs run at a time (0: not asked, -1: none).  Open addressing
// by the kernel's address; entries are only ever added.  Threads may race to ask the same thing twice.
struct Grant {
    std::atomic<const void *> kernel{nullptr};
    std::atomic<int> bytes{0};
    std::atomic<int> clusters[9] = {};
};
constexpr int kGrantSlots = 512;                          // (a few times the library's number of kernels)
// A grant is the context's: another context of the same device, or the primary one after a reset, starts without
// any.  Contexts are told apart by the driver's number, which it never gives twice.  A process that has gone
// through more contexts than there is room for asks the runtime on every launch in the further ones.
constexpr int kContexts = 8;
struct Context {
    std::atomic<uint64_t> number{0};                      // the driver's, plus one
    std::atomic<void *> scratch{nullptr};                 // (context_scratch)
    Grant grants[kGrantSlots];
};
Context g_contexts[kContexts];

// The calling thread's context, as the driver's number for it plus one; 0 if it has none yet.
uint64_t current_context()
{
    using GetId = CUresult (*)(CUcontext, unsigned long long *);
    static const GetId get_id = [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        const bool ok = cudaGetDriverEntryPoint("cuCtxGetId", &fn, cudaEnableDefault, &found) == cudaSuccess && found == cudaDriverEntryPointSuccess;
        if (!ok) cudaGetLastError();
        return ok ? reinterpret_cast<GetId>(fn) : nullptr;
    }();
    unsigned long long number = 0;
    return get_id && get_id(nullptr, &number) == CUDA_SUCCESS ? (uint64_t)number + 1 : 0;
}

// What is remembered about it; null: nothing can be.
Context *context()
{
    const uint64_t number = current_context();
    if (number == 0) return nullptr;
    for (Context &c : g_contexts) {
        uint64_t have = c.number.load(std::memory_order_acquire);
        if (have == 0 && c.number.compare_exchange_strong(have, number)) have = number;
        if (have == number) return &c;
    }
    return nullptr;
}

Grant *grant_of(const void *kernel)
{
    Context *const c = context();
    if (!c) return nullptr;
    const uint32_t h = (uint32_t)((reinterpret_cast<uintptr_t>(kernel) >> 4) * 2654435761u) >> 7;
    for (uint32_t k = 0; k < (uint32_t)kGrantSlots; ++k) {
        Grant &g = c->grants[(h + k) % kGrantSlots];
        const void *have = g.kernel.load(std::memory_order_acquire);
        if (have == nullptr && g.kernel.compare_exchange_strong(have, kernel)) have = kernel;
        if (have == kernel) return &g;
    }
    return nullptr;
}

}  // namespace

std::atomic<void *> *context_scratch()
{
    Context *const c = context();
    return c ? &c->scratch : nullptr;
}

int sm_count()
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
    int sms = dev < kMaxDevices ? g_sms[dev].load(std::memory_order_relaxed) : 0;
    if (sms > 0) return sms;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (dev < kMaxDevices) g_sms[dev].store(sms, std::memory_order_relaxed);
    return sms;
}

bool allow_shared_memory(const void *kernel, int bytes)
{
    Grant *g = grant_of(kernel);
    if (g && g->bytes.load(std::memory_order_acquire) >= bytes) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    if (g) {
        int old = g->bytes.load(std::memory_order_relaxed);
        while (old < bytes && !g->bytes.compare_exchange_weak(old, bytes, std::memory_order_release)) {}
    }
    return true;
}

static cudaLaunchConfig_t cluster_config(int clusters, int ctas, int threads, int smem, cudaStream_t stream, cudaLaunchAttribute *attr)
{
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = 1; attr->val.clusterDim.y = (unsigned)ctas; attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)clusters, (unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cfg;
}

int resident_clusters(const void *kernel, int ctas, int threads, int smem)
{
    if (ctas < 1 || ctas > 8) return 0;
    Grant *g = grant_of(kernel);
    int have = g ? g->clusters[ctas].load(std::memory_order_acquire) : 0;
    if (have == 0) {
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = cluster_config(1, ctas, threads, smem, nullptr, &attr);
        if (!allow_shared_memory(kernel, smem) || cudaOccupancyMaxActiveClusters(&have, kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            have = 0;
        }
        if (have <= 0) have = -1;
        if (g) g->clusters[ctas].store(have, std::memory_order_release);
    }
    return have < 0 ? 0 : have;
}

int launch_clusters(const void *kernel, int clusters, int ctas, int threads, int smem, cudaStream_t stream, void **args)
{
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config(clusters, ctas, threads, smem, stream, &attr);
    const cudaError_t e = cudaLaunchKernelExC(&cfg, kernel, args);
    const int rc = check_launch();
    return e == cudaSuccess ? rc : RVQ_ERR_LAUNCH;
}

static int ceil_log2(int k)
{
    int b = 0;
    while ((1 << b) < k) ++b;
    return b < 1 ? 1 : b;
}

int make_shape(const rvq_config *c, Shape *s)
{
    if (!c) return RVQ_ERR_BADARG;
    if (c->group_dim != 8 && c->group_dim != 16 && c->group_dim != 32 && c->group_dim != 64)
        return RVQ_ERR_UNSUPPORTED;
    if (c->dim < c->group_dim || c->dim > 1024 || c->dim % c->group_dim) return RVQ_ERR_BADARG;
    if (c->layout != RVQ_GROUP_CONTIGUOUS && c->layout != RVQ_GROUP_STRIDED) return RVQ_ERR_BADARG;
    if (c->depth < 1 || c->depth > 16) return RVQ_ERR_BADARG;
    if (c->codebook_size < 2 || c->codebook_size > 65536) return RVQ_ERR_BADARG;
    if (c->code_bits != 16 && c->code_bits != ceil_log2(c->codebook_size)) return RVQ_ERR_BADARG;
    if (c->x_dtype < RVQ_F32 || c->x_dtype > RVQ_F16) return RVQ_ERR_BADARG;
    if (c->std_ddof != 0 && c->std_ddof != 1) return RVQ_ERR_BADARG;
    s->dim = c->dim; s->gd = c->group_dim; s->G = c->dim / c->group_dim; s->layout = c->layout;
    s->R = c->depth; s->K = c->codebook_size; s->bits = c->code_bits; s->dtype = c->x_dtype;
    s->ddof = c->std_ddof;
    if (s->G > 128 || s->dim - s->ddof <= 0) return RVQ_ERR_UNSUPPORTED;
    s->per_vector = s->G * s->R;
    s->code_bytes = s->bits == 16 ? s->per_vector * 2 : (s->per_vector * s->bits + 31) / 32 * 4;
    s->elem_bytes = c->x_dtype == RVQ_F32 ? 4 : 2;
    s->raw = 0;
    return RVQ_OK;
}

static int check_rows(const Shape &s, const void *p, int64_t n, int64_t stride)
{
    if (n < 0 || stride < s.dim) return RVQ_ERR_BADARG;
    if (n > 0 && !p) return RVQ_ERR_BADARG;
    if (!aligned16(p) || (stride * s.elem_bytes) % 16) return RVQ_ERR_ALIGN;
    return RVQ_OK;
}

}  // namespace rvq

using namespace rvq;

extern "C" {

const char *rvq_status_string(int code)
{
    switch (code) {
    case RVQ_OK: return "ok";
    case RVQ_ERR_BADARG: return "bad argument";
    case RVQ_ERR_ALIGN: return "pointer or stride not 16-byte aligned";
    case RVQ_ERR_UNSUPPORTED: return "unsupported shape";
    case RVQ_ERR_WORKSPACE: return "workspace too small";
    case RVQ_ERR_LAUNCH: return "CUDA launch failed";
    case RVQ_ERR_DEVICE: return "no sm_100 device";
    case RVQ_ERR_STATIC_LIMIT: return "shape needs more scratch than the library's built-in array holds";
    default: return "unknown error";
    }
}

int rvq_version(void) { return 1000; }

uint64_t rvq_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

size_t rvq_code_bytes(const rvq_config *cfg)
{
    Shape s;
    return make_shape(cfg, &s) == RVQ_OK ? (size_t)s.code_bytes : 0;
}

size_t rvq_prepared_bytes(const rvq_config *cfg)
{
    Shape s;
    return make_shape(cfg, &s) == RVQ_OK ? prepared_bytes(s) : 0;
}

int rvq_prepare_codebooks(const rvq_config *cfg, const float *codebooks, void *prepared, void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if (!codebooks || !prepared) return RVQ_ERR_BADARG;
    if (!aligned16(codebooks) || !aligned256(prepared)) return RVQ_ERR_ALIGN;
    return launch_prepare(s, codebooks, prepared, (cudaStream_t)stream);
}

size_t rvq_workspace_bytes(const rvq_config *cfg, int64_t n)
{
    Shape s;
    (void)n;
    return make_shape(cfg, &s) == RVQ_OK ? ema_workspace_bytes(s) : 0;
}

static int encode_common(const rvq_config *cfg, const void *x, int64_t n, int64_t x_row_stride,
                         const float *codebooks, const void *prepared, void *codes, uint16_t *std_f16,
                         float *stage_energy, rvq_status *status, void *stream, bool allow_tensor,
                         uint32_t *stat_cnt = nullptr, float *stat_sum = nullptr)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if ((rc = check_rows(s, x, n, x_row_stride)) != RVQ_OK) return rc;
    if (!codebooks || !prepared || (n > 0 && (!codes || !std_f16))) return RVQ_ERR_BADARG;
    if (!aligned16(codebooks) || !aligned16(codes) || !aligned256(prepared)) return RVQ_ERR_ALIGN;
    if (stage_energy && cudaMemsetAsync(stage_energy, 0, (size_t)s.R * sizeof(float), (cudaStream_t)stream) != cudaSuccess)
        return RVQ_ERR_LAUNCH;
    if (allow_tensor && !stat_sum && encode_small_wanted(s, n))
        return launch_encode_small(s, x, n, x_row_stride, prepared, codes, std_f16, status, (cudaStream_t)stream, stage_energy);
    if (allow_tensor && !stat_sum && encode_split_wanted(s, n))
        return launch_encode_split(s, x, n, x_row_stride, codebooks, prepared, codes, std_f16, status, (cudaStream_t)stream, stage_energy);
    if (allow_tensor && encode_tensor_supported(s))
        return launch_encode_tensor(s, x, n, x_row_stride, codebooks, prepared, codes, std_f16, status,
                                    (cudaStream_t)stream, stat_cnt, stat_sum, stage_energy);
    return launch_encode_scalar(s, x, n, x_row_stride, codebooks, codes, std_f16, status, (cudaStream_t)stream,
                                stage_energy);
}

int rvq_encode(const rvq_config *cfg, const void *x, int64_t n, int64_t x_row_stride,
               const float *codebooks, const void *prepared, void *codes, uint16_t *std_f16,
               float *stage_energy, void *workspace, size_t workspace_bytes, rvq_status *status, void *stream)
{
    (void)workspace; (void)workspace_bytes;
    return encode_common(cfg, x, n, x_row_stride, codebooks, prepared, codes, std_f16, stage_energy, status, stream, true);
}

// Whether the batch's statistics are taken by a pass of their own after the encode, or fused into the throughput kernel
// (us of rvq_encode_stats, fused / apart).
//   - Batches that the encoders for few tiles take (up to one tile per SM): apart, those encoders can run, but the pass costs
//     its time per row, while the throughput kernel takes as long for one row as for all tiles of such a batch, and
//     longer with more codes.  So apart up to a number of group rows that grows with the codes, and with how fast the
//     pass is (depth 8 but where said otherwise):
//     four rows of a warp, 16 K: 512 codes 8192 rows 50 / 48, 16384 54 / 58; 700 codes 8192 60 / 54, 16384 61 / 66; 1024 codes 8192 69 / 56, 16384
//     70 / 71, 18944 70 / 73; 2048 codes 18944 107 / 99 (depth 4, 512 codes 8192 32 / 35, 1024 codes 16384 42 / 46, 2048 codes 18944 61 / 61);
//     one row of a warp, 8 K: 512 codes 4096 rows 51 / 50, 8192 52 / 54; 1024 codes 8192 69 / 61, 16384 70 / 77; 2048 codes 16384 107 / 105;
//     a thread per row, 4 K from 1024 codes on: 512 codes lose at any size (256 rows 50 / 55); 1024 codes, 16 groups 4096 69 / 70, 8192 69 / 76,
//     depth 12 4096 96 / 90, 8192 96 / 98; 2048 codes 8192 106 / 89, 16384 106 / 113.
//   - More tiles with codebooks too small to hide the additions behind (fused, the epilogue waits for them), with four
//     groups or eight.  A learning step: 32000 vectors and 256 codes 193 / 175, 240000 940 / 944, 1M 4050 / 4100 (all
//     rows meet in a few bins either way); 512 codes 80000 426 / 416, 480000 2312 / 2222.
static bool statistics_apart(const Shape &s, int64_t n)
{
    const StatsPass pass = ema_stats_pass(s);
    const int64_t rows = n * s.G;
    if (encode_small_wanted(s, n) || encode_split_wanted(s, n))
        return rows <= (pass == StatsPass::kQuad ? 16 : pass == StatsPass::kWarp ? 8 : s.K >= 1024 ? 4 : 0) * (int64_t)s.K;
    return encode_tensor_deferred_stages(s) == 0 && pass == StatsPass::kQuad && (s.K > 256 || rows <= (1 << 19));
}

int rvq_encode_stats(const rvq_config *cfg, const void *x, int64_t n, int64_t x_row_stride,
                     const float *codebooks, const void *prepared, void *codes, uint16_t *std_f16,
                     float *stage_energy, float *batch_count, float *batch_sum, void *workspace,
                     size_t workspace_bytes, rvq_status *status, void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if (!batch_count || !batch_sum || !workspace) return RVQ_ERR_BADARG;
    if (!aligned16(batch_sum) || !aligned256(workspace)) return RVQ_ERR_ALIGN;
    if (workspace_bytes < ema_stats_scratch_bytes(s)) return RVQ_ERR_WORKSPACE;
    if (!encode_tensor_supported(s) || statistics_apart(s, n)) {
        rc = encode_common(cfg, x, n, x_row_stride, codebooks, prepared, codes, std_f16, stage_energy, status, stream, true);
        if (rc != RVQ_OK) return rc;
        return launch_ema_stats(s, x, n, x_row_stride, codes, codebooks, batch_count, batch_sum, workspace,
                                status, (cudaStream_t)stream);
    }
    if ((rc = check_rows(s, x, n, x_row_stride)) != RVQ_OK) return rc;
    if (!codebooks || !prepared || (n > 0 && (!codes || !std_f16))) return RVQ_ERR_BADARG;
    if (!aligned16(codebooks) || !aligned16(codes) || !aligned256(prepared)) return RVQ_ERR_ALIGN;
    uint32_t *cnt = reinterpret_cast<uint32_t *>(workspace);
    const int bins = s.R * s.K;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(cnt, 0, (size_t)bins * sizeof(uint32_t), st) != cudaSuccess ||
        cudaMemsetAsync(batch_sum, 0, (size_t)bins * s.gd * sizeof(float), st) != cudaSuccess)
        return RVQ_ERR_LAUNCH;
    rc = encode_common(cfg, x, n, x_row_stride, codebooks, prepared, codes, std_f16, stage_energy, status, stream, true,
                       cnt, batch_sum);
    if (rc != RVQ_OK) return rc;
    return launch_stats_finish(s, cnt, codebooks, batch_sum, batch_count, encode_tensor_deferred_stages(s), st);
}

int rvq_selftest_encode_timeout(const rvq_config *cfg, const void *x, int64_t n, int64_t x_row_stride,
                                const float *codebooks, const void *prepared, void *codes, uint16_t *std_f16,
                                uint32_t wait_polls, rvq_status *status, void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if ((rc = check_rows(s, x, n, x_row_stride)) != RVQ_OK) return rc;
    if (!codebooks || !prepared || !status || (n > 0 && (!codes || !std_f16))) return RVQ_ERR_BADARG;
    if (!aligned16(codebooks) || !aligned16(codes) || !aligned256(prepared)) return RVQ_ERR_ALIGN;
    if (!encode_tensor_supported(s) || wait_polls < 1024u) return RVQ_ERR_UNSUPPORTED;
    return launch_encode_tensor(s, x, n, x_row_stride, codebooks, prepared, codes, std_f16, status,
                                (cudaStream_t)stream, nullptr, nullptr, nullptr, wait_polls, 1);
}

int rvq_encode_exact(const rvq_config *cfg, const void *x, int64_t n, int64_t x_row_stride,
                     const float *codebooks, const void *prepared, void *codes, uint16_t *std_f16,
                     float *stage_energy, rvq_status *status, void *stream)
{
    return encode_common(cfg, x, n, x_row_stride, codebooks, prepared, codes, std_f16, stage_energy, status, stream, false);
}

int rvq_decode(const rvq_config *cfg, const void *codes, const uint16_t *std_f16, int64_t n,
               const float *codebooks, const void *prepared, void *x_out, int64_t out_row_stride,
               rvq_status *status, void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if ((rc = check_rows(s, x_out, n, out_row_stride)) != RVQ_OK) return rc;
    if (!codebooks || !prepared || (n > 0 && (!codes || !std_f16))) return RVQ_ERR_BADARG;
    if (!aligned16(codebooks) || !aligned16(codes) || !aligned256(prepared)) return RVQ_ERR_ALIGN;
    if (decode_direct_wanted(s, n, false, true))
        return launch_decode_direct(s, codes, std_f16, n, codebooks, x_out, out_row_stride, status, (cudaStream_t)stream);
    if (decode_sliced_supported(s))
        return launch_decode_sliced(s, codes, std_f16, n, codebooks, prepared, x_out, out_row_stride, status, (cudaStream_t)stream);
    return launch_decode_gather(s, codes, std_f16, n, codebooks, x_out, out_row_stride, status, (cudaStream_t)stream);
}

int rvq_rope_table(int32_t dim, double base, int32_t positions, float *cos_sin, void *stream)
{
    if (dim < 2 || dim > 1024 || (dim & 1) || !(base > 1.0) || positions < 0 || (positions > 0 && !cos_sin))
        return RVQ_ERR_BADARG;
    if (!aligned16(cos_sin)) return RVQ_ERR_ALIGN;
    return launch_rope_table(dim, base, positions, cos_sin, (cudaStream_t)stream);
}

int rvq_decode_rope(const rvq_config *cfg, const void *codes, const uint16_t *std_f16, int64_t n,
                    const float *codebooks, const void *prepared, const int32_t *position,
                    int32_t vectors_per_position,
                    const float *cos_sin, int32_t positions, int32_t pairing, void *x_out,
                    int64_t out_row_stride, rvq_status *status, void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if ((rc = check_rows(s, x_out, n, out_row_stride)) != RVQ_OK) return rc;
    if (!codebooks || (n > 0 && (!codes || !std_f16 || !position || !cos_sin))) return RVQ_ERR_BADARG;
    if (vectors_per_position < 1 || positions < 1 || (pairing != RVQ_ROPE_HALVES && pairing != RVQ_ROPE_ADJACENT))
        return RVQ_ERR_BADARG;
    if (s.dim & 1) return RVQ_ERR_UNSUPPORTED;
    if (!aligned16(codebooks) || !aligned16(codes) || !aligned16(cos_sin) || !aligned256(prepared)) return RVQ_ERR_ALIGN;
    if (decode_direct_wanted(s, n, true, prepared != nullptr))
        return launch_decode_direct(s, codes, std_f16, n, codebooks, x_out, out_row_stride, status, (cudaStream_t)stream, position,
                                    vectors_per_position, cos_sin, positions, pairing);
    return launch_decode_rope(s, codes, std_f16, n, codebooks, prepared, position, vectors_per_position, cos_sin, positions,
                              pairing, x_out, out_row_stride, status, (cudaStream_t)stream);
}

size_t rvq_attention_workspace_bytes(int64_t tokens, int32_t q_heads)
{
    if (tokens < 1 || q_heads < 1 || q_heads > 32) return 0;
    return attention_workspace_bytes(tokens, q_heads);
}

int rvq_attention_decode(const rvq_config *cfg_k, const rvq_config *cfg_v, const float *q, int32_t q_heads,
                         const void *codes_k, const uint16_t *std_k, const void *codes_v, const uint16_t *std_v,
                         int64_t tokens, int32_t kv_heads, const float *codebooks_k, const float *codebooks_v,
                         const int32_t *position, const float *cos_sin, int32_t positions, int32_t pairing,
                         float scale, float *out, void *workspace, size_t workspace_bytes, rvq_status *status,
                         void *stream)
{
    Shape sk, sv;
    int rc = make_shape(cfg_k, &sk);
    if (rc != RVQ_OK) return rc;
    if ((rc = make_shape(cfg_v, &sv)) != RVQ_OK) return rc;
    if (!q || !codes_k || !std_k || !codes_v || !std_v || !codebooks_k || !codebooks_v || !out || !workspace)
        return RVQ_ERR_BADARG;
    if (tokens < 1 || q_heads < 1 || kv_heads < 1 || !(scale == scale)) return RVQ_ERR_BADARG;
    if (cos_sin && (positions < 1 || (pairing != RVQ_ROPE_HALVES && pairing != RVQ_ROPE_ADJACENT))) return RVQ_ERR_BADARG;
    if (!attention_supported(sk, sv, kv_heads, q_heads, tokens)) return RVQ_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(codes_k) || !aligned16(codes_v) || !aligned16(codebooks_k) || !aligned16(codebooks_v) ||
        !aligned16(cos_sin) || !aligned16(out) || !aligned256(workspace))
        return RVQ_ERR_ALIGN;
    if (workspace_bytes < attention_workspace_bytes(tokens, q_heads)) return RVQ_ERR_WORKSPACE;
    return launch_attention_decode(sk, sv, q, q_heads, codes_k, std_k, codes_v, std_v, tokens, codebooks_k, codebooks_v,
                                   position, cos_sin, positions, pairing, scale, out, workspace, status,
                                   (cudaStream_t)stream);
}

static int check_ema_common(const Shape &s, const void *x, int64_t n, int64_t stride, const void *codes,
                            const float *codebooks)
{
    int rc = check_rows(s, x, n, stride);
    if (rc != RVQ_OK) return rc;
    if (!codebooks || (n > 0 && !codes)) return RVQ_ERR_BADARG;
    if (!aligned16(codebooks) || !aligned16(codes)) return RVQ_ERR_ALIGN;
    return RVQ_OK;
}

int rvq_ema_stats(const rvq_config *cfg, const void *x, int64_t n, int64_t x_row_stride,
                  const void *codes, const float *codebooks, float *batch_count, float *batch_sum,
                  void *workspace, size_t workspace_bytes, rvq_status *status, void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if ((rc = check_ema_common(s, x, n, x_row_stride, codes, codebooks)) != RVQ_OK) return rc;
    if (!batch_count || !batch_sum || !workspace) return RVQ_ERR_BADARG;
    if (!aligned16(batch_sum) || !aligned256(workspace)) return RVQ_ERR_ALIGN;
    if (workspace_bytes < ema_stats_scratch_bytes(s)) return RVQ_ERR_WORKSPACE;
    return launch_ema_stats(s, x, n, x_row_stride, codes, codebooks, batch_count, batch_sum, workspace,
                            status, (cudaStream_t)stream);
}

int rvq_ema_apply(const rvq_config *cfg, const float *batch_count, const float *batch_sum,
                  float *codebooks, float *ema_count, float *ema_sum, float decay, float eps,
                  void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if (!batch_count || !batch_sum || !codebooks || !ema_count || !ema_sum) return RVQ_ERR_BADARG;
    if (!(decay >= 0.0f && decay <= 1.0f) || !(eps >= 0.0f)) return RVQ_ERR_BADARG;
    return launch_ema_apply(s, batch_count, batch_sum, codebooks, ema_count, ema_sum, decay, eps,
                            (cudaStream_t)stream);
}

int rvq_ema_update(const rvq_config *cfg, const void *x, int64_t n, int64_t x_row_stride,
                   const void *codes, float *codebooks, float *ema_count, float *ema_sum,
                   float *batch_count, float decay, float eps, void *workspace,
                   size_t workspace_bytes, rvq_status *status, void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if ((rc = check_ema_common(s, x, n, x_row_stride, codes, codebooks)) != RVQ_OK) return rc;
    if (!ema_count || !ema_sum || !workspace) return RVQ_ERR_BADARG;
    if (!(decay >= 0.0f && decay <= 1.0f) || !(eps >= 0.0f)) return RVQ_ERR_BADARG;
    if (!aligned16(ema_sum) || !aligned256(workspace)) return RVQ_ERR_ALIGN;
    if (workspace_bytes < ema_workspace_bytes(s)) return RVQ_ERR_WORKSPACE;
    uint8_t *ws = reinterpret_cast<uint8_t *>(workspace);
    float *bc = reinterpret_cast<float *>(ws + ema_stats_scratch_bytes(s));
    float *bs = reinterpret_cast<float *>(ws + ema_stats_scratch_bytes(s) +
                                          ((size_t)s.R * s.K * sizeof(float) + 255) / 256 * 256);
    rc = launch_ema_stats(s, x, n, x_row_stride, codes, codebooks, bc, bs, workspace, status, (cudaStream_t)stream);
    if (rc != RVQ_OK) return rc;
    if (batch_count &&
        cudaMemcpyAsync(batch_count, bc, (size_t)s.R * s.K * sizeof(float), cudaMemcpyDeviceToDevice,
                        (cudaStream_t)stream) != cudaSuccess)
        return RVQ_ERR_LAUNCH;
    return launch_ema_apply(s, bc, bs, codebooks, ema_count, ema_sum, decay, eps, (cudaStream_t)stream);
}

int rvq_learn_step(const rvq_config *cfg, const void *x, int64_t n, int64_t x_row_stride,
                   float *codebooks, void *prepared, float *ema_count, float *ema_sum, void *codes,
                   uint16_t *std_f16, float *stage_energy, float decay, float eps, void *workspace,
                   size_t workspace_bytes, rvq_status *status, void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if (!ema_count || !ema_sum || !workspace || !codebooks || !prepared) return RVQ_ERR_BADARG;
    if (!(decay >= 0.0f && decay <= 1.0f) || !(eps >= 0.0f)) return RVQ_ERR_BADARG;
    if (!aligned16(ema_sum) || !aligned256(workspace)) return RVQ_ERR_ALIGN;
    if (workspace_bytes < ema_workspace_bytes(s)) return RVQ_ERR_WORKSPACE;
    // same carving as rvq_ema_update: counts | batch counts | batch sums
    uint8_t *ws = reinterpret_cast<uint8_t *>(workspace);
    float *bc = reinterpret_cast<float *>(ws + ema_stats_scratch_bytes(s));
    float *bs = reinterpret_cast<float *>(ws + ema_stats_scratch_bytes(s) +
                                          ((size_t)s.R * s.K * sizeof(float) + 255) / 256 * 256);
    rc = rvq_encode_stats(cfg, x, n, x_row_stride, codebooks, prepared, codes, std_f16, stage_energy, bc, bs,
                          workspace, workspace_bytes, status, stream);
    if (rc != RVQ_OK) return rc;
    // (this call's kernels follow one another: their launches overlap)
    rc = launch_ema_apply(s, bc, bs, codebooks, ema_count, ema_sum, decay, eps, (cudaStream_t)stream, true);
    if (rc != RVQ_OK) return rc;
    return launch_prepare(s, codebooks, prepared, (cudaStream_t)stream, true);
}

size_t rvq_kmeans_workspace_bytes(const rvq_config *cfg, int64_t n)
{
    Shape s;
    return make_shape(cfg, &s) == RVQ_OK ? kmeans_workspace_bytes(s, n) : 0;
}

int rvq_kmeans_init(const rvq_config *cfg, const void *x, int64_t n, int64_t x_row_stride,
                    const int64_t *seed_rows, int32_t iterations, float *codebooks, void *prepared,
                    void *workspace, size_t workspace_bytes, rvq_status *status, void *stream)
{
    Shape s;
    int rc = make_shape(cfg, &s);
    if (rc != RVQ_OK) return rc;
    if (!encode_tensor_supported(s)) return RVQ_ERR_UNSUPPORTED;
    if ((rc = check_rows(s, x, n, x_row_stride)) != RVQ_OK) return rc;
    if (n < 1 || !seed_rows || !codebooks || !prepared || !workspace) return RVQ_ERR_BADARG;
    if (iterations < 0 || iterations > 1000) return RVQ_ERR_BADARG;
    if (!aligned16(codebooks) || !aligned256(prepared) || !aligned256(workspace)) return RVQ_ERR_ALIGN;
    if (workspace_bytes < kmeans_workspace_bytes(s, n)) return RVQ_ERR_WORKSPACE;
    return launch_kmeans(s, x, n, x_row_stride, seed_rows, iterations, codebooks, prepared, workspace, status,
                         (cudaStream_t)stream);
}

}  // extern "C"
