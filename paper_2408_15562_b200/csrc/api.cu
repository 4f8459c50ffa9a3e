// C ABI of libfspad.so: context management, argument validation and the
// host-buffer entry point.  All arithmetic of the verify step lives in the
// kernel translation units; nothing here computes on the host.
#include <climits>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <new>

#include <cuda.h>

#include "common.cuh"

namespace {

inline bool misaligned(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; }

template <typename T>
bool dev_alloc(T **p, size_t count)
{
    *p = nullptr;
    if (count == 0) count = 1;
    return cudaMalloc(reinterpret_cast<void **>(p), count * sizeof(T)) == cudaSuccess;
}

int check_common(const fspad_ctx *ctx, int n_nodes, int batch)
{
    if (!ctx) return FSPAD_ERR_NULL;
    if (n_nodes > FSPAD_MAX_NODES_WIDE || n_nodes > ctx->cfg.max_nodes) return FSPAD_ERR_TREE_TOO_LARGE;
    if (n_nodes < 1 || batch < 0 || batch > ctx->cfg.max_batch) return FSPAD_ERR_SHAPE;
    return FSPAD_OK;
}

// Device address of host memory [p, p + bytes) if all of it is page-locked and mapped in one piece, else NULL.  The first
// byte alone says nothing about the rest: of a buffer whose front part only is registered a kernel would read past the mapping.
const void *mapped_whole(const void *p, size_t bytes)
{
    typedef CUresult (*AttrFn)(void *, CUpointer_attribute, CUdeviceptr);
    static const AttrFn attr = [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        const bool ok = cudaGetDriverEntryPoint("cuPointerGetAttribute", &fn, cudaEnableDefault, &q) == cudaSuccess &&
                        q == cudaDriverEntryPointSuccess;
        (void)cudaGetLastError();
        return ok ? reinterpret_cast<AttrFn>(fn) : nullptr;
    }();
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    if (at.type != cudaMemoryTypeHost || at.devicePointer == nullptr || attr == nullptr) return nullptr;
    CUdeviceptr lo = 0;
    size_t size = 0;
    const CUdeviceptr first = reinterpret_cast<CUdeviceptr>(at.devicePointer);
    if (attr(&lo, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, first) != CUDA_SUCCESS ||
        attr(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, first) != CUDA_SUCCESS)
        return nullptr;
    return first >= lo && first - lo <= size && size - (first - lo) >= bytes ? at.devicePointer : nullptr;
}

// Whether the host can look at p: a caller's mistake (a device array for a host one) is the copy's to report.
bool on_host(const void *p)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) == cudaSuccess) return at.type != cudaMemoryTypeDevice;
    (void)cudaGetLastError();
    return true;
}

// Rows [batch][nodes] of the nodes that have children, and of the roots: what the scan by the trees reads.
int rows_with_children(const int32_t *parent, int nodes, int batch)
{
    int n = 0;
    for (int b = 0; b < batch; ++b, parent += nodes) {
        unsigned long long mark[(FSPAD_MAX_NODES_WIDE + 63) / 64] = {1ull};
        for (int c = 1; c < nodes; ++c) {
            const unsigned p = (unsigned)parent[c];
            if (p < (unsigned)c) mark[p >> 6] |= 1ull << (p & 63);
        }
        for (unsigned long long m : mark) n += __builtin_popcountll(m);
    }
    return n;
}

// How a step's attention shares the SMs with its acceptance.  Both entry points take it from here: the number of key ranges
// follows from attn_sms, and with it which reference a probability is rounded against, so that they give the same bits.
struct StepPlan {
    bool chain;                 // one stream: scan, walk, and the attention launched beside the walk
    bool scan_first;            // two streams: the scan goes first on all SMs, the attention behind it beside the walk
    int attn_sms;               // SMs the attention may fill (0: all)
    bool compact_far;           // a compaction kernel would come behind a long attention
};
// A call that is being captured into a graph: its events cost nothing there.
bool capturing(cudaStream_t st)
{
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &s) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return s == cudaStreamCaptureStatusActive;
}
// captured: decides on the order alone, never on attn_sms.
StepPlan step_plan(fspad_ctx *ctx, int n_nodes, int batch, bool may_sample, bool captured)
{
    // Which of the two goes first.  The acceptance is a streaming scan over every SM followed by a walk
    // that one cluster per sampling sequence carries out; the attention is one CTA per SM.  Where the walk's clusters
    // leave half of the SMs free and the attention is long, the scan goes first on all SMs and the walk and the attention, sized
    // for the SMs the walk leaves, follow it in the same stream as programmatic dependents: the attention's CTAs come when every
    // CTA of the walk has its SM.  (On a second stream behind an event the attention was there 3 to 5 us later, or now and then
    // ahead of a cluster, which then had no 16 SMs side by side before the attention had left: 80 us in place of 38 on 52 heads.
    // One B200, us a step, two streams against one: 50.7 and 38.1 on 52 heads and 4 K keys, 44.2 and 42.4 on 8 x 8 and 8 K,
    // both 17 chunks a CTA.)  What is known here is how long the sequences may be, not how long they are; so the merge of the key ranges
    // waits for the attention alone, not for the walk (when it did, a 2 K sequence in a context of 12 K rows or more took 37.1 us, two
    // streams 34.2, and 31.1 now; 52 heads and 4 K keys 38.6 -> 39.0).  On larger arrays of logits one stream is the better way for an
    // attention of any length (`any_attn`): called one by one, 8 KV heads and 60 x 128256 at 1 K, 2 K and 4 K keys 31.2 -> 27.6, 32.2 -> 28.9
    // and 32.3 -> 28.8, 64 heads at 2 K 32.1 -> 28.5, two sequences 35.1 -> 33.8, all behind a scan by the trees; behind a scan of all rows
    // 60 x 50257 32.3 -> 27.4, 24 x 128256 28.9 -> 24.1, 24 x 50257 twice 26.6 -> 24.6.  (The line lies higher than it need: 60 x 32000, below it, takes
    // 28.3 us in two streams and 25.2 in one.)  Captured, such a step forks only where the scan goes first: beside an attention on most SMs
    // it is the longer way (52 heads and 1 K keys 38.7).
    // In a graph, where events cost nothing, the fork is the better way if the attention's CTAs find room beside the walk's: 29.7 against
    // 30.4 us (one stream) on the 2 K sequence, 37.8 and 38.4 on 52 heads, 17.3 and 18.1 at 580 keys, 45.3 and 46.5 on two such
    // sequences; where they do not, four short sequences of 32 heads take 33.8 in one stream and 44.8 forked.  A walk of single CTAs (less than 4096
    // tokens) has next to no scan before it and goes beside the attention from the start: 12.8 against 14.2 (one stream) and 16.2 (scan first).
    // Otherwise, and with more clusters, the attention is forked behind the scan onto the second stream.
    const fspad_config &c = ctx->cfg;
    const int sms = ctx->sm_count;
    auto ctas_on = [&](int n) {
        return (long long)batch * c.n_kv_heads * fspad_attn_mtiles(ctx, n_nodes, batch, n) * fspad_attn_umma_splits(ctx, n_nodes, batch, n);
    };
    const long long attn_ctas = ctas_on(sms);
    StepPlan p = {false, false, 0, false};
    if (may_sample) {
        const int walk = fspad_walk_ctas(ctx, batch, c.vocab);
        const int beside = sms - (walk < sms / 2 ? walk : sms / 2), ranges = fspad_attn_umma_splits(ctx, n_nodes, batch, beside);
        const bool long_attn = ranges == 1 || (c.max_len + 127) / 128 >= 12 * ranges;
        const int rows = batch * n_nodes;
        const bool any_attn = (long long)rows * c.vocab >= (n_nodes >= 16 ? 1 << 21 : 1 << 23) || (c.vocab > 98304 && rows <= 32);
        const bool one_stream = walk <= sms / 2 && (long_attn || any_attn);
        const bool scan_first = walk <= sms / 2 && long_attn ? walk > batch : sms - attn_ctas < sms / 4;
        const bool fork = !one_stream || (captured && ctas_on(beside) <= beside && (long_attn || scan_first));
        p.chain = !fork;
        p.scan_first = fork && scan_first;
        p.compact_far = p.chain && long_attn;
        if (scan_first || (walk <= sms / 2 && long_attn)) p.attn_sms = beside;
    } else {
        // An all-greedy acceptance is a scan and a one-CTA walk: beside an attention that holds most SMs the
        // scan's CTAs only get going when the attention's leave.  Where the context is short enough for the
        // attention to stay short on half the SMs (at most 8 chunks per CTA by the context's max_len), it
        // gets half and the two really run side by side (17.2 against 20.5 us on the 26-node greedy workload); and where the scan
        // is short, too (8 MB: 1.3 us of HBM, 3.6 us in all), and the step is called and not captured, the scan goes first and the attention
        // follows in the same stream: four launches without an event between them, 16.5 -> 12.7 us on that workload (in one range; in two,
        // with 1024 rows, 16.5 -> 13.9).  With one key range (no merge) that holds for an attention of few CTAs, too: 8 KV heads called one
        // by one 16.5 -> 12.4 us.  From a graph the two streams take 11.4 us on that workload against 12.8 in one (1024 rows: 12.2 and 13.7;
        // 8 KV heads: 11.4 and 12.4).
        const int s_half = fspad_attn_umma_splits(ctx, n_nodes, batch, sms / 2);
        const int max_chunks = (c.max_len + 127) / 128;
        const bool short_attn = (max_chunks + s_half - 1) / s_half <= 8;
        if (short_attn && attn_ctas > sms / 2) p.attn_sms = sms / 2;
        p.chain = !captured && short_attn && (attn_ctas > sms / 2 || fspad_attn_umma_splits(ctx, n_nodes, batch) == 1) &&
                  (long long)batch * n_nodes * c.vocab <= 2 << 20;
    }
    return p;
}

}  // namespace

extern "C" {

const char *fspad_strerror(int err)
{
    switch (err) {
    case FSPAD_OK: return "ok";
    case FSPAD_ERR_NULL: return "required pointer is NULL";
    case FSPAD_ERR_ALIGN: return "pointer is not 16-byte aligned";
    case FSPAD_ERR_SHAPE: return "sizes inconsistent with the context";
    case FSPAD_ERR_TREE_TOO_LARGE: return "tree has more nodes than supported";
    case FSPAD_ERR_RANGE: return "value out of range (prefix length, token id, temperature or path)";
    case FSPAD_ERR_CUDA: return "CUDA runtime call failed";
    case FSPAD_ERR_TIMEOUT: return "bounded device-side wait ran out";
    case FSPAD_ERR_BAD_TREE: return "parent[] is not a topologically ordered tree rooted at node 0";
    case FSPAD_ERR_NOMEM: return "allocation failed";
    case FSPAD_ERR_TOO_LARGE: return "size exceeds the fixed capacity of the no-allocation entry point";
    default: return "unknown error";
    }
}

int fspad_create(const fspad_config *cfg, fspad_ctx **out)
{
    if (!out) return FSPAD_ERR_NULL;
    *out = nullptr;
    if (!cfg) return FSPAD_ERR_NULL;
    if (cfg->head_dim != FSPAD_HEAD_DIM || cfg->n_kv_heads < 1 || cfg->n_q_heads < 1 ||
        cfg->n_q_heads % cfg->n_kv_heads != 0 || cfg->vocab < 1 || cfg->n_layers < 1 ||
        cfg->max_len < 1 || cfg->max_batch < 1 || cfg->max_nodes < 1)
        return FSPAD_ERR_SHAPE;
    if (cfg->max_nodes > FSPAD_MAX_NODES_WIDE) return FSPAD_ERR_TREE_TOO_LARGE;
    if (cfg->max_nodes > cfg->max_len) return FSPAD_ERR_RANGE;
    if (!(cfg->softmax_scale >= 0.0f)) return FSPAD_ERR_RANGE;

    fspad_ctx *ctx = new (std::nothrow) fspad_ctx();
    if (!ctx) return FSPAD_ERR_NOMEM;
    std::memset(ctx, 0, sizeof(*ctx));
    ctx->cfg = *cfg;
    ctx->scale = cfg->softmax_scale > 0.0f ? cfg->softmax_scale : 1.0f / std::sqrt((float)cfg->head_dim);
    if (cudaGetDevice(&ctx->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess) {
        delete ctx;
        return FSPAD_ERR_CUDA;
    }

    const int G = cfg->n_q_heads / cfg->n_kv_heads;
    const size_t B = (size_t)cfg->max_batch, Nmax = (size_t)cfg->max_nodes;
    // split-KV partials: worst case over every (n_nodes, batch) a call may pass, and any length of a paged call's table
    size_t part_rows = 0;
    int max_splits = 1;
    for (int n = 1; n <= cfg->max_nodes; ++n)
        for (int b = 1; b <= cfg->max_batch; ++b) {
            const int s = fspad_attn_ranges(ctx, n, b, 0, INT_MAX, true);
            const size_t rows = (size_t)b * cfg->n_kv_heads * s * n * G;
            if (rows > part_rows) part_rows = rows;
            if (s > max_splits) max_splits = s;
        }
    ctx->attn_max_splits = max_splits;
    const size_t rows = B * Nmax;
    ctx->stats_slots = 64;

    bool ok = dev_alloc(&ctx->d_status, 1);
    ok = ok && dev_alloc(&ctx->part_o, part_rows * FSPAD_HEAD_DIM);
    ok = ok && dev_alloc(&ctx->part_ml, part_rows * 2);
    ok = ok && dev_alloc(&ctx->attn_done, 1);
    ok = ok && dev_alloc(&ctx->st_part, rows * ctx->stats_slots);
    ok = ok && dev_alloc(&ctx->row_max, rows);
    ok = ok && dev_alloc(&ctx->row_sum, rows);
    ok = ok && dev_alloc(&ctx->row_arg, rows);
    {
        uint2 *dx = nullptr;
        ok = ok && dev_alloc(&dx, B * FSPAD_MAX_FRONTIER * (size_t)fspad_draft_expand_pieces(cfg->vocab) * FSPAD_MAX_FRONTIER);
        ctx->dx_part = dx;
    }
    ok = ok && dev_alloc(&ctx->dx_done, B);
    ok = ok && dev_alloc(&ctx->dx_front, 2 * B * FSPAD_MAX_FRONTIER);
    ok = ok && dev_alloc(&ctx->lm_parts, (rows < FSPAD_LM_SLAB_ROWS ? rows : (size_t)FSPAD_LM_SLAB_ROWS) * fspad_lm_head_tiles(cfg->vocab));
    ok = ok && cudaStreamCreateWithFlags(&ctx->side, cudaStreamNonBlocking) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&ctx->ev_join, cudaEventDisableTiming) == cudaSuccess;
    if (ok) {
        ok = cudaMemset(ctx->d_status, 0, sizeof(int)) == cudaSuccess &&
             cudaMemset(ctx->attn_done, 0, sizeof(int)) == cudaSuccess &&
             cudaMemset(ctx->dx_done, 0, B * sizeof(int)) == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess;
    }
    if (!ok) {
        fspad_destroy(ctx);
        return FSPAD_ERR_NOMEM;
    }
    *out = ctx;
    return FSPAD_OK;
}

void fspad_destroy(fspad_ctx *ctx)
{
    if (!ctx) return;
    cudaDeviceSynchronize();
    void *ptrs[] = {ctx->lm_parts, ctx->dx_part, ctx->dx_done, ctx->dx_front, ctx->d_status, ctx->part_o, ctx->part_ml, ctx->attn_done, ctx->st_part, ctx->row_max, ctx->row_sum, ctx->row_arg, ctx->h_q, ctx->h_tk,
                    ctx->h_tv, ctx->h_out, ctx->h_parent, ctx->h_prefix, ctx->h_tokens, ctx->h_path,
                    ctx->h_nacc, ctx->h_bonus, ctx->h_newlen, ctx->h_logits, ctx->h_draft, ctx->h_temp,
                    ctx->h_unif};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    if (ctx->ev_fork) cudaEventDestroy(ctx->ev_fork);
    if (ctx->ev_join) cudaEventDestroy(ctx->ev_join);
    if (ctx->side) cudaStreamDestroy(ctx->side);
    delete ctx;
}

int fspad_status(fspad_ctx *ctx, void *stream)
{
    if (!ctx) return FSPAD_ERR_NULL;
    cudaStream_t st = fspad_stream(stream);
    int h = 0;
    if (cudaMemcpyAsync(&h, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return FSPAD_ERR_CUDA;
    if (h != 0) {
        if (cudaMemsetAsync(ctx->d_status, 0, sizeof(int), st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return FSPAD_ERR_CUDA;
    }
    return h;
}

long long fspad_launch_count(const fspad_ctx *ctx) { return ctx ? ctx->launches : 0; }

int fspad_selftest_wait_timeout(fspad_ctx *ctx, int polls, void *stream)
{
    if (!ctx) return FSPAD_ERR_NULL;
    if (polls < 1 || polls > 4096) return FSPAD_ERR_RANGE;
    return fspad_launch_wait_selftest(ctx, polls, fspad_stream(stream)) == cudaSuccess &&
                   fspad_launch_walk_wait_selftest(ctx, polls, fspad_stream(stream)) == cudaSuccess
               ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_tree_attn(fspad_ctx *ctx, const fspad_bf16 *q, const fspad_bf16 *k_cache,
                    const fspad_bf16 *v_cache, const fspad_bf16 *tree_k, const fspad_bf16 *tree_v,
                    const int32_t *parent, const int32_t *prefix_len, int n_nodes, int batch,
                    fspad_bf16 *out, void *stream)
{
    int rc = check_common(ctx, n_nodes, batch);
    if (rc) return rc;
    if (!q || !k_cache || !v_cache || !parent || !prefix_len || !out) return FSPAD_ERR_NULL;
    if ((tree_k == nullptr) != (tree_v == nullptr)) return FSPAD_ERR_NULL;
    if (misaligned(q) || misaligned(k_cache) || misaligned(v_cache) || misaligned(tree_k) ||
        misaligned(tree_v) || misaligned(out))
        return FSPAD_ERR_ALIGN;
    if (n_nodes > ctx->cfg.max_len) return FSPAD_ERR_RANGE;
    if (batch == 0) return FSPAD_OK;
    cudaError_t e = fspad_launch_tree_attn(ctx, q, k_cache, v_cache, tree_k, tree_v, parent, prefix_len,
                                           n_nodes, batch, out, fspad_stream(stream), 0, FspadPaged{nullptr, 0, 0, false, true});
    return e == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_accept_stats(fspad_ctx *ctx, const float *logits, const float *temperature, int rows,
                       int rows_per_seq, float *row_max, double *row_sum, int32_t *row_arg,
                       void *stream)
{
    if (!ctx) return FSPAD_ERR_NULL;
    const bool scan_only = !row_max && !row_sum && !row_arg;
    if (!logits || (!scan_only && (!row_max || !row_sum || !row_arg))) return FSPAD_ERR_NULL;
    if (rows < 0 || rows_per_seq < 1 || rows > ctx->cfg.max_batch * ctx->cfg.max_nodes)
        return FSPAD_ERR_SHAPE;
    if (rows == 0) return FSPAD_OK;
    if (scan_only) {
        FspadStatsGeom geom;
        return fspad_launch_stats_partials(ctx, logits, temperature, rows, rows_per_seq, ctx->cfg.vocab, &geom,
                                           fspad_stream(stream)) == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
    }
    cudaError_t e = fspad_launch_accept_stats(ctx, logits, temperature, rows, rows_per_seq, ctx->cfg.vocab,
                                              row_max, row_sum, row_arg, fspad_stream(stream));
    return e == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_tree_accept(fspad_ctx *ctx, const float *target_logits, const float *draft_probs,
                      const int32_t *draft_tokens, const int32_t *parent, const float *temperature,
                      const float *uniforms, int n_nodes, int batch, int32_t *accepted_path,
                      int32_t *n_accepted, int32_t *bonus_token, void *stream)
{
    int rc = check_common(ctx, n_nodes, batch);
    if (rc) return rc;
    if (!target_logits || !draft_tokens || !parent || !temperature || !accepted_path || !n_accepted ||
        !bonus_token)
        return FSPAD_ERR_NULL;
    if ((draft_probs == nullptr) != (uniforms == nullptr)) return FSPAD_ERR_NULL;
    if (misaligned(target_logits) || misaligned(draft_probs)) return FSPAD_ERR_ALIGN;
    if (batch == 0) return FSPAD_OK;
    cudaStream_t st = fspad_stream(stream);
    FspadStatsGeom geom;
    if (fspad_scan_inner(ctx->sm_count, batch * n_nodes, n_nodes, ctx->cfg.vocab, draft_probs != nullptr, true)) geom.parent = parent;
    cudaError_t e = fspad_launch_stats_partials(ctx, target_logits, temperature, batch * n_nodes, n_nodes,
                                                ctx->cfg.vocab, &geom, st);
    if (e != cudaSuccess) return FSPAD_ERR_CUDA;
    e = fspad_launch_accept_walk(ctx, target_logits, draft_probs, draft_tokens, parent, temperature,
                                 uniforms, geom, n_nodes, batch, ctx->cfg.vocab, accepted_path, n_accepted,
                                 bonus_token, st);
    return e == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_lm_head_stats(fspad_ctx *ctx, const fspad_bf16 *hidden, const fspad_bf16 *lm_head, int hidden_dim, int rows,
                        int rows_per_seq, const float *temperature, float *logits_out, float *row_max, double *row_sum,
                        int32_t *row_arg, void *stream)
{
    if (!ctx) return FSPAD_ERR_NULL;
    if (!hidden || !lm_head || !row_max || !row_sum || !row_arg) return FSPAD_ERR_NULL;
    if (misaligned(hidden) || misaligned(lm_head) || misaligned(logits_out)) return FSPAD_ERR_ALIGN;
    if (hidden_dim < 8 || hidden_dim % 8 != 0 || rows < 0 || rows_per_seq < 1 ||
        rows > ctx->cfg.max_batch * ctx->cfg.max_nodes)
        return FSPAD_ERR_SHAPE;
    if (rows == 0) return FSPAD_OK;
    return fspad_launch_lm_head(ctx, hidden, lm_head, hidden_dim, rows, rows_per_seq, temperature, logits_out, nullptr,
                                row_max, row_sum, row_arg, fspad_stream(stream)) == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_lm_head_accept(fspad_ctx *ctx, const fspad_bf16 *hidden, const fspad_bf16 *lm_head, int hidden_dim,
                         const float *draft_probs, const int32_t *draft_tokens, const int32_t *parent,
                         const float *temperature, const float *uniforms, int n_nodes, int batch, float *logits,
                         int32_t *accepted_path, int32_t *n_accepted, int32_t *bonus_token, void *stream)
{
    int rc = check_common(ctx, n_nodes, batch);
    if (rc) return rc;
    if (!hidden || !lm_head || !draft_tokens || !parent || !temperature || !accepted_path || !n_accepted || !bonus_token)
        return FSPAD_ERR_NULL;
    if ((draft_probs == nullptr) != (uniforms == nullptr)) return FSPAD_ERR_NULL;
    if (draft_probs != nullptr && logits == nullptr) return FSPAD_ERR_NULL;     // the sampling walk reads logits rows
    if (misaligned(hidden) || misaligned(lm_head) || misaligned(logits) || misaligned(draft_probs)) return FSPAD_ERR_ALIGN;
    if (hidden_dim < 8 || hidden_dim % 8 != 0) return FSPAD_ERR_SHAPE;
    if (batch == 0) return FSPAD_OK;
    cudaStream_t st = fspad_stream(stream);
    const int V = ctx->cfg.vocab, rows = batch * n_nodes;
    const bool vec = (V % 4 == 0);          // logits and draft rows are 16-byte aligned (checked above)
    const FspadStatsGeom geom = fspad_lm_head_geom(rows, V, vec, ctx->stats_slots);
    if (fspad_launch_lm_head(ctx, hidden, lm_head, hidden_dim, rows, n_nodes, temperature, logits, &geom, nullptr, nullptr,
                             nullptr, st) != cudaSuccess)
        return FSPAD_ERR_CUDA;
    // a greedy walk needs only the partials; logits may be NULL then, and the walk never reads them
    return fspad_launch_accept_walk(ctx, logits, draft_probs, draft_tokens, parent, temperature, uniforms, geom, n_nodes,
                                    batch, V, accepted_path, n_accepted, bonus_token, st) == cudaSuccess
               ? FSPAD_OK : FSPAD_ERR_CUDA;
}

size_t fspad_feature_sampler_workspace_bytes(int rows, int hidden_dim, int inter_dim)
{
    if (rows < 1 || hidden_dim < 1 || inter_dim < 1) return 0;
    return fspad_feature_sampler_scratch_floats(rows, hidden_dim, inter_dim) * sizeof(float);
}

int fspad_feature_sampler(fspad_ctx *ctx, const fspad_bf16 *f, const fspad_bf16 *e, const fspad_bf16 *w_up,
                          const fspad_bf16 *w_gate, const fspad_bf16 *w_down, int rows, int hidden_dim, int inter_dim,
                          fspad_bf16 *inter, fspad_bf16 *eta, void *workspace, size_t workspace_bytes, void *stream)
{
    if (!ctx) return FSPAD_ERR_NULL;
    if (!f || !e || !w_up || !w_gate || !w_down || !inter || !eta || !workspace) return FSPAD_ERR_NULL;
    if (misaligned(f) || misaligned(e) || misaligned(w_up) || misaligned(w_gate) || misaligned(w_down) || misaligned(inter) ||
        misaligned(eta) || misaligned(workspace))
        return FSPAD_ERR_ALIGN;
    if (rows < 0 || rows > 128 || hidden_dim < 8 || hidden_dim % 8 != 0 || inter_dim < 8 || inter_dim % 8 != 0)
        return FSPAD_ERR_SHAPE;
    if (rows == 0) return FSPAD_OK;
    if (workspace_bytes < fspad_feature_sampler_workspace_bytes(rows, hidden_dim, inter_dim)) return FSPAD_ERR_RANGE;
    return fspad_launch_feature_sampler(ctx, f, e, w_up, w_gate, w_down, rows, hidden_dim, inter_dim, inter, eta,
                                        static_cast<float *>(workspace), fspad_stream(stream)) == cudaSuccess
               ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_tree_attn_paged(fspad_ctx *ctx, const fspad_bf16 *q, const fspad_bf16 *k_pool, const fspad_bf16 *v_pool,
                          const int32_t *block_table, int blocks_per_seq, int n_blocks, const fspad_bf16 *tree_k,
                          const fspad_bf16 *tree_v, const int32_t *parent, const int32_t *prefix_len, int n_nodes,
                          int batch, fspad_bf16 *out, void *stream)
{
    int rc = check_common(ctx, n_nodes, batch);
    if (rc) return rc;
    if (!q || !k_pool || !v_pool || !block_table || !parent || !prefix_len || !out) return FSPAD_ERR_NULL;
    if ((tree_k == nullptr) != (tree_v == nullptr)) return FSPAD_ERR_NULL;
    if (misaligned(q) || misaligned(k_pool) || misaligned(v_pool) || misaligned(tree_k) || misaligned(tree_v) || misaligned(out))
        return FSPAD_ERR_ALIGN;
    if (blocks_per_seq < 1 || n_blocks < 1 || (long long)blocks_per_seq * 128 < n_nodes) return FSPAD_ERR_SHAPE;
    if (batch == 0) return FSPAD_OK;
    if (blocks_per_seq > INT_MAX / 128) return FSPAD_ERR_TOO_LARGE;      // rows are counted in 32 bits
    const FspadPaged pg{block_table, blocks_per_seq, n_blocks, false, true};
    return fspad_launch_tree_attn(ctx, q, k_pool, v_pool, tree_k, tree_v, parent, prefix_len, n_nodes, batch, out,
                                  fspad_stream(stream), 0, pg) == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_kv_compact_paged(fspad_ctx *ctx, fspad_bf16 *pool, const int32_t *block_table, int blocks_per_seq, int n_blocks,
                           const int32_t *accepted_path, const int32_t *n_accepted, const int32_t *prefix_len, int batch,
                           int32_t *new_len, void *stream)
{
    if (!ctx) return FSPAD_ERR_NULL;
    if (!pool || !block_table || !accepted_path || !n_accepted || !prefix_len) return FSPAD_ERR_NULL;
    if (misaligned(pool)) return FSPAD_ERR_ALIGN;
    if (batch < 0 || batch > ctx->cfg.max_batch || blocks_per_seq < 1 || n_blocks < 1) return FSPAD_ERR_SHAPE;
    if (batch == 0) return FSPAD_OK;
    const FspadPaged pg{block_table, blocks_per_seq, n_blocks};
    return fspad_launch_kv_compact_paged(ctx, pool, pg, accepted_path, n_accepted, prefix_len, batch, new_len,
                                         fspad_stream(stream)) == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_kv_compact(fspad_ctx *ctx, fspad_bf16 *cache, const int32_t *accepted_path,
                     const int32_t *n_accepted, const int32_t *prefix_len, int batch,
                     int32_t *new_len, void *stream)
{
    if (!ctx) return FSPAD_ERR_NULL;
    if (!cache || !accepted_path || !n_accepted || !prefix_len) return FSPAD_ERR_NULL;
    if (misaligned(cache)) return FSPAD_ERR_ALIGN;
    if (batch < 0 || batch > ctx->cfg.max_batch) return FSPAD_ERR_SHAPE;
    if (batch == 0) return FSPAD_OK;
    cudaError_t e = fspad_launch_kv_compact(ctx, cache, accepted_path, n_accepted, prefix_len, batch,
                                            new_len, fspad_stream(stream));
    return e == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_kv_append(fspad_ctx *ctx, fspad_bf16 *cache, const fspad_bf16 *tree_kv, const int32_t *accepted_path,
                    const int32_t *n_accepted, const int32_t *prefix_len, int n_nodes, int batch, int32_t *new_len,
                    void *stream)
{
    int rc = check_common(ctx, n_nodes, batch);
    if (rc) return rc;
    if (!cache || !tree_kv || !accepted_path || !n_accepted || !prefix_len) return FSPAD_ERR_NULL;
    if (misaligned(cache) || misaligned(tree_kv)) return FSPAD_ERR_ALIGN;
    if (batch == 0) return FSPAD_OK;
    cudaError_t e = fspad_launch_kv_append(ctx, cache, tree_kv, accepted_path, n_accepted, prefix_len, n_nodes, batch,
                                           new_len, fspad_stream(stream));
    return e == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_tree_build(fspad_ctx *ctx, const int32_t *cand_parent, const int32_t *cand_token,
                     const float *cand_logp, const int32_t *root_token, int n_cand, int n_nodes, int batch,
                     int32_t *parent_out, int32_t *token_out, int32_t *cand_out, uint64_t *anc_out,
                     int32_t *n_out, void *stream)
{
    int rc = check_common(ctx, n_nodes, batch);
    if (rc) return rc;
    if (!cand_parent || !cand_token || !cand_logp || !root_token || !parent_out || !token_out || !cand_out || !n_out)
        return FSPAD_ERR_NULL;
    if (n_nodes > FSPAD_MAX_NODES) return FSPAD_ERR_TREE_TOO_LARGE;      // the builder's masks are one word per node
    if (n_cand < 1 || n_cand > FSPAD_MAX_CANDIDATES) return FSPAD_ERR_SHAPE;
    if (batch == 0) return FSPAD_OK;
    cudaError_t e = fspad_launch_tree_build(ctx, cand_parent, cand_token, cand_logp, root_token, n_cand, n_nodes,
                                            batch, parent_out, token_out, cand_out,
                                            reinterpret_cast<unsigned long long *>(anc_out), n_out, fspad_stream(stream));
    return e == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_draft_expand(fspad_ctx *ctx, const float *logprobs, const float *frontier_logp,
                       const int32_t *frontier_cand, int n_frontier, int top_k, int width, int base, int n_cand_cap,
                       int batch, int32_t *cand_parent, int32_t *cand_token, float *cand_logp, int32_t *next_cand,
                       float *next_logp, void *stream)
{
    if (!ctx) return FSPAD_ERR_NULL;
    if (!logprobs || !frontier_logp || !frontier_cand || !cand_parent || !cand_token || !cand_logp || !next_cand ||
        !next_logp)
        return FSPAD_ERR_NULL;
    if (batch < 0 || batch > ctx->cfg.max_batch) return FSPAD_ERR_SHAPE;
    if (n_frontier < 1 || n_frontier > FSPAD_MAX_FRONTIER || top_k < 1 || top_k > FSPAD_MAX_FRONTIER ||
        top_k > ctx->cfg.vocab)
        return FSPAD_ERR_SHAPE;
    if (width < 1 || width > n_frontier * top_k || base < 0 || base + n_frontier * top_k > n_cand_cap)
        return FSPAD_ERR_SHAPE;
    if ((long long)fspad_draft_expand_pieces(ctx->cfg.vocab) * top_k > FSPAD_MAX_CANDIDATES) return FSPAD_ERR_TOO_LARGE;
    if (batch == 0) return FSPAD_OK;
    cudaError_t e = fspad_launch_draft_expand(ctx, logprobs, frontier_logp, frontier_cand, n_frontier, top_k, width,
                                              base, n_cand_cap, batch, cand_parent, cand_token, cand_logp, next_cand,
                                              next_logp, fspad_stream(stream));
    return e == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_verify_step(fspad_ctx *ctx, fspad_bf16 *cache, int attn_layer, const fspad_bf16 *q,
                      const fspad_bf16 *tree_k, const fspad_bf16 *tree_v, const int32_t *parent,
                      const int32_t *prefix_len, const float *target_logits, const float *draft_probs,
                      const int32_t *draft_tokens, const float *temperature, const float *uniforms,
                      int n_nodes, int batch, fspad_bf16 *attn_out, int32_t *accepted_path,
                      int32_t *n_accepted, int32_t *bonus_token, int32_t *new_len, void *stream)
{
    int rc = check_common(ctx, n_nodes, batch);
    if (rc) return rc;
    if (!cache || !q || !parent || !prefix_len || !target_logits || !draft_tokens || !temperature || !attn_out ||
        !accepted_path || !n_accepted || !bonus_token)
        return FSPAD_ERR_NULL;
    if ((tree_k == nullptr) != (tree_v == nullptr)) return FSPAD_ERR_NULL;
    if ((draft_probs == nullptr) != (uniforms == nullptr)) return FSPAD_ERR_NULL;
    if (misaligned(cache) || misaligned(q) || misaligned(tree_k) || misaligned(tree_v) || misaligned(attn_out) ||
        misaligned(target_logits) || misaligned(draft_probs))
        return FSPAD_ERR_ALIGN;
    if (attn_layer < 0 || attn_layer >= ctx->cfg.n_layers) return FSPAD_ERR_SHAPE;
    if (n_nodes > ctx->cfg.max_len) return FSPAD_ERR_RANGE;
    if (batch == 0) return FSPAD_OK;
    const fspad_config &c = ctx->cfg;
    cudaStream_t st = fspad_stream(stream);
    const size_t plane = (size_t)batch * c.n_kv_heads * (size_t)c.max_len * FSPAD_HEAD_DIM;
    const fspad_bf16 *kc = cache + (size_t)attn_layer * 2 * plane, *vc = kc + plane;

    const int sms = ctx->sm_count;
    const bool may_sample = draft_probs != nullptr;
    const StepPlan plan = step_plan(ctx, n_nodes, batch, may_sample, capturing(st));
    const bool scan_first = plan.scan_first;
    const int attn_sms = plan.attn_sms;
    cudaError_t ce = cudaSuccess;
    FspadStatsGeom geom;
    const int rows = batch * n_nodes;
    if (fspad_scan_inner(sms, rows, n_nodes, c.vocab, may_sample, false)) geom.parent = parent;
    // With the tree rows given apart from the cache the compaction depends on the walk alone, and when the
    // sequence's slices are few (a warp takes one after another: four each for the 16 warps of a greedy walk's CTA) the walk makes the moves itself at its end: one dependent launch less on the step's
    // longest chain (all-greedy step of 26 nodes and 64 slices: 29.3 -> 23.7 us called one by one, 13.1 against 13.3 from a graph).
    // In one stream, where the compaction kernel would come behind the attention, that pays up to two slices a warp of the cluster's CTAs, 16
    // warps each: 256 slices at 32000 tokens (eight CTAs) 22.3 us against 23.5 with the kernel, at 128256 (16) 28.5 and 30.7; a single CTA
    // (4000 tokens) 29.4 and 24.9.  A sequence of temperature 0 among them has one CTA whatever the cluster: 256 slices 23 us and 22.4.
    const bool aliased = tree_k == nullptr;      // attention reads the cache rows that compaction rewrites
    int most_slices = 64;
    if (plan.compact_far) {
        const int by_cluster = 32 * (fspad_walk_ctas(ctx, batch, c.vocab) / batch);
        most_slices = by_cluster < 64 ? 64 : by_cluster > 256 ? 256 : by_cluster;
    }
    const bool walk_compacts = !aliased && c.n_layers * 2 * c.n_kv_heads <= most_slices;
    FspadWalkCompact kv;
    if (walk_compacts) { kv.cache = cache; kv.prefix_len = prefix_len; kv.new_len = new_len; }
    if (plan.chain) {
        // Every kernel's end waits for its predecessor's: what follows this call finds all of it complete.
        ce = fspad_launch_stats_partials(ctx, target_logits, temperature, rows, n_nodes, c.vocab, &geom, st);
        if (ce == cudaSuccess)
            ce = fspad_launch_accept_walk(ctx, target_logits, draft_probs, draft_tokens, parent, temperature, uniforms, geom,
                                          n_nodes, batch, c.vocab, accepted_path, n_accepted, bonus_token, st, kv);
        if (ce == cudaSuccess)
            ce = fspad_launch_tree_attn(ctx, q, kc, vc, tree_k, tree_v, parent, prefix_len, n_nodes, batch, attn_out, st, attn_sms,
                                        FspadPaged{nullptr, 0, 0, true});
        if (ce == cudaSuccess && !walk_compacts)
            ce = fspad_launch_kv_compact(ctx, cache, accepted_path, n_accepted, prefix_len, batch, new_len, st);
        return ce == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
    }
    if (scan_first)
        ce = fspad_launch_stats_partials(ctx, target_logits, temperature, rows, n_nodes, c.vocab, &geom, st);
    // fork: the attention of this step on the context's second stream
    if (ce != cudaSuccess || cudaEventRecord(ctx->ev_fork, st) != cudaSuccess ||
        cudaStreamWaitEvent(ctx->side, ctx->ev_fork, 0) != cudaSuccess)
        return FSPAD_ERR_CUDA;
    int rc_attn = FSPAD_OK;
    if (!scan_first) {
        rc_attn = fspad_launch_tree_attn(ctx, q, kc, vc, tree_k, tree_v, parent, prefix_len, n_nodes, batch, attn_out,
                                         ctx->side, attn_sms) == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
        // Here the scan is launched as a plain dependent: as a programmatic dependent of the previous
        // step's last kernel it was seen to hold the forked attention back behind the whole acceptance
        // (steps replayed from one CUDA graph: 72.5 us per step against 48.8 on the 52-head shape).
        // Where the acceptance is the longer chain (a sampling walk follows, or the attention is the short
        // one above), the scan is cut for the SMs the attention leaves free - one wave of two CTAs per SM
        // there: cut for the whole chip its CTAs queue for those few SMs in several waves, each with a
        // launch's fixed cost (45.5 -> 41.2 us on the 52-head sampling workload, 17.1 -> 14.7 us on the
        // 26-node greedy one).  Under a long attention with a greedy walk the short-lived CTAs of the
        // full-size scan are the better neighbours (37.6 against 39.0 us): an attention CTA that finds
        // its SM taken waits for a scan CTA's whole life.
        int scan_sms = 0;
        if (may_sample || attn_sms > 0) {
            const long long attn_now = (long long)batch * c.n_kv_heads * fspad_attn_mtiles(ctx, n_nodes, batch, attn_sms) *
                                       fspad_attn_umma_splits(ctx, n_nodes, batch, attn_sms);
            scan_sms = sms - (int)(attn_now < sms ? attn_now : sms);
            if (scan_sms < sms / 8) scan_sms = sms / 8;
        }
        ce = fspad_launch_stats_partials(ctx, target_logits, temperature, rows, n_nodes, c.vocab, &geom, st, false, scan_sms);
    }
    if (ce == cudaSuccess)
        ce = fspad_launch_accept_walk(ctx, target_logits, draft_probs, draft_tokens, parent, temperature, uniforms, geom,
                                      n_nodes, batch, c.vocab, accepted_path, n_accepted, bonus_token, st, kv);
    rc = ce == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
    if (scan_first) {
        // When the walk's clusters need more than one wave, merge CTAs that sit resident waiting for the
        // attention would keep the later clusters off their SMs (244 against 224 us on the ragged batch):
        // the merge kernel is then a plain dependent.
        const bool walk_one_wave = fspad_walk_ctas(ctx, batch, c.vocab) <= sms / 2;   // the attention was sized to leave that many free
        rc_attn = fspad_launch_tree_attn(ctx, q, kc, vc, tree_k, tree_v, parent, prefix_len, n_nodes, batch, attn_out,
                                         ctx->side, attn_sms, FspadPaged{nullptr, 0, 0}, walk_one_wave) == cudaSuccess
                      ? FSPAD_OK : FSPAD_ERR_CUDA;
    }
    // the join is queued whatever happened in between, so that a capture of `stream` never ends
    // with the second stream left unjoined
    const bool ev_ok = cudaEventRecord(ctx->ev_join, ctx->side) == cudaSuccess;
    bool joined = false;
    if (aliased) joined = cudaStreamWaitEvent(st, ctx->ev_join, 0) == cudaSuccess;
    if (rc == FSPAD_OK && rc_attn == FSPAD_OK && !walk_compacts) {
        // behind a join the compaction has two predecessors, so it is launched as a plain dependent
        cudaError_t e = fspad_launch_kv_compact(ctx, cache, accepted_path, n_accepted, prefix_len, batch, new_len, st,
                                                !aliased);
        if (e != cudaSuccess) rc = FSPAD_ERR_CUDA;
    }
    if (!aliased) joined = cudaStreamWaitEvent(st, ctx->ev_join, 0) == cudaSuccess;
    if (rc_attn) return rc_attn;
    if (rc) return rc;
    return (ev_ok && joined) ? FSPAD_OK : FSPAD_ERR_CUDA;
}

int fspad_verify_step_host(fspad_ctx *ctx, fspad_bf16 *cache, const fspad_bf16 *q,
                           const fspad_bf16 *tree_k, const fspad_bf16 *tree_v, const int32_t *parent,
                           const int32_t *prefix_len, const float *target_logits,
                           const float *draft_probs, const int32_t *draft_tokens,
                           const float *temperature, const float *uniforms, int n_nodes, int batch,
                           fspad_bf16 *attn_out, int32_t *accepted_path, int32_t *n_accepted,
                           int32_t *bonus_token, int32_t *new_len, void *stream)
{
    int rc = check_common(ctx, n_nodes, batch);
    if (rc) return rc;
    if (!cache || !q || !tree_k || !tree_v || !parent || !prefix_len || !target_logits || !draft_tokens ||
        !temperature || !attn_out || !accepted_path || !n_accepted || !bonus_token || !new_len)
        return FSPAD_ERR_NULL;
    if ((draft_probs == nullptr) != (uniforms == nullptr)) return FSPAD_ERR_NULL;
    if (misaligned(cache)) return FSPAD_ERR_ALIGN;
    if (n_nodes > ctx->cfg.max_len) return FSPAD_ERR_RANGE;
    if (batch == 0) return FSPAD_OK;
    const fspad_config &c = ctx->cfg;
    cudaStream_t st = fspad_stream(stream);

    // staging buffers are created by the first call, sized for the context's maxima; a failed
    // attempt frees what it got, so that a later call starts over instead of using half a set
    if (!ctx->h_ready) {
        const size_t B = (size_t)c.max_batch, N = (size_t)c.max_nodes;
        bool ok = dev_alloc(&ctx->h_q, B * N * c.n_q_heads * FSPAD_HEAD_DIM);
        ok = ok && dev_alloc(&ctx->h_out, B * N * c.n_q_heads * FSPAD_HEAD_DIM);
        ok = ok && dev_alloc(&ctx->h_tk, B * c.n_kv_heads * N * FSPAD_HEAD_DIM);
        ok = ok && dev_alloc(&ctx->h_tv, B * c.n_kv_heads * N * FSPAD_HEAD_DIM);
        ok = ok && dev_alloc(&ctx->h_parent, B * N) && dev_alloc(&ctx->h_tokens, B * N);
        ok = ok && dev_alloc(&ctx->h_prefix, B) && dev_alloc(&ctx->h_nacc, B);
        ok = ok && dev_alloc(&ctx->h_bonus, B) && dev_alloc(&ctx->h_newlen, B);
        ok = ok && dev_alloc(&ctx->h_path, B * N) && dev_alloc(&ctx->h_temp, B);
        ok = ok && dev_alloc(&ctx->h_unif, B * (N + 1));
        ok = ok && dev_alloc(&ctx->h_logits, B * N * c.vocab);
        ok = ok && dev_alloc(&ctx->h_draft, B * N * c.vocab);
        if (!ok) {
            void **slots[] = {(void **)&ctx->h_q, (void **)&ctx->h_out, (void **)&ctx->h_tk, (void **)&ctx->h_tv,
                              (void **)&ctx->h_parent, (void **)&ctx->h_tokens, (void **)&ctx->h_prefix,
                              (void **)&ctx->h_nacc, (void **)&ctx->h_bonus, (void **)&ctx->h_newlen,
                              (void **)&ctx->h_path, (void **)&ctx->h_temp, (void **)&ctx->h_unif,
                              (void **)&ctx->h_logits, (void **)&ctx->h_draft};
            for (void **sl : slots) {
                if (*sl) cudaFree(*sl);
                *sl = nullptr;
            }
            (void)cudaGetLastError();
            return FSPAD_ERR_NOMEM;
        }
        ctx->h_ready = 1;
    }
    const size_t B = (size_t)batch, N = (size_t)n_nodes;
    const size_t q_bytes = B * N * c.n_q_heads * FSPAD_HEAD_DIM * sizeof(fspad_bf16);
    const size_t t_bytes = B * c.n_kv_heads * N * FSPAD_HEAD_DIM * sizeof(fspad_bf16);
    const size_t lg_bytes = B * N * c.vocab * sizeof(float);
    bool ok = true;
    auto h2d = [&](void *dst, const void *src, size_t bytes) {
        ok = ok && cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st) == cudaSuccess;
    };
    auto d2h = [&](void *dst, const void *src, size_t bytes) {
        ok = ok && cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    };
    // The caller's memory is read and written by what is queued, the draft rows by the walk itself: an error, too, is returned only
    // when nothing of it is still under way.
    auto give_up = [&](int err) {
        (void)cudaStreamSynchronize(ctx->side);
        (void)cudaStreamSynchronize(st);
        return err;
    };
    // The walk reads draft rows only where it rejects, and one probability per node: page-locked draft rows are left where they
    // are and read over the link by the kernel (60 rows of 128256 copied whole took 557 us, as long as the logits).  The
    // kernel wants them on a 16-byte boundary, and pageable ones have to be copied.
    const float *draft = draft_probs ? static_cast<const float *>(mapped_whole(draft_probs, lg_bytes)) : nullptr;
    if (misaligned(draft)) draft = nullptr;
    const bool draft_in_place = draft != nullptr;
    // Of the logits the scan by the trees reads the rows of nodes with children, a quarter of a 60-node tree's, and the walk the one row that
    // it ends in: page-locked ones, too, are left where they are (60 rows of 128256 copied whole took 557 us).  Not where nearly all nodes
    // have children: the kernel takes 50 GB/s from the link and the copy 55.3, every row begun costs it about 0.08 us, and what it saves is
    // the copy's own 2 us of a greedy step and 12 us of a sampled one.  Calls in place and copied, us: chains of 60 x 128256 717 and 660
    // (greedy), four of 30 x 8000 208 and 184, one of 8 x 128256 158 and 169; two of 16 x 32000 178 and 164 greedy, 185 and 188 sampled.  The trees
    // are looked at here for that alone: if the stream has yet to bring them, what they hold now decides which way the logits go, and
    // nothing else.
    const float *far_logits = nullptr;
    if (fspad_scan_inner_fits(ctx->sm_count, batch * n_nodes, c.vocab)) far_logits = static_cast<const float *>(mapped_whole(target_logits, lg_bytes));
    if (misaligned(far_logits)) far_logits = nullptr;
    if (far_logits && on_host(parent)) {
        const double inner = rows_with_children(parent, n_nodes, batch), row_bytes = (double)c.vocab * sizeof(float);
        if (inner * (1.106 * row_bytes + 4700.0) >= (double)lg_bytes + (draft_probs ? 660e3 : 100e3)) far_logits = nullptr;
    }
    h2d(ctx->h_prefix, prefix_len, B * sizeof(int));
    h2d(ctx->h_parent, parent, B * N * sizeof(int));
    h2d(ctx->h_tk, tree_k, t_bytes);
    h2d(ctx->h_tv, tree_v, t_bytes);
    h2d(ctx->h_q, q, q_bytes);
    if (!ok) return give_up(FSPAD_ERR_CUDA);
    // the tree rows go into cache rows L_b .. of layer 0 (K at [0][0], V at [0][1]); the attention then takes them from there
    if (fspad_launch_tree_scatter(ctx, cache, ctx->h_tk, ctx->h_tv, ctx->h_prefix, n_nodes, batch, st) !=
        cudaSuccess)
        return give_up(FSPAD_ERR_CUDA);
    // fork: the attention and its result's way back run beside the copy of the logits
    if (cudaEventRecord(ctx->ev_fork, st) != cudaSuccess || cudaStreamWaitEvent(ctx->side, ctx->ev_fork, 0) != cudaSuccess)
        return give_up(FSPAD_ERR_CUDA);
    const size_t plane = (size_t)batch * c.n_kv_heads * (size_t)c.max_len * FSPAD_HEAD_DIM;
    const StepPlan plan = step_plan(ctx, n_nodes, batch, draft_probs != nullptr, false);
    const bool attn_ok = fspad_launch_tree_attn(ctx, ctx->h_q, cache, cache + plane, nullptr, nullptr, ctx->h_parent, ctx->h_prefix,
                                                n_nodes, batch, ctx->h_out, ctx->side, plan.attn_sms) == cudaSuccess;
    h2d(ctx->h_tokens, draft_tokens, B * N * sizeof(int));
    h2d(ctx->h_temp, temperature, B * sizeof(float));
    if (draft_probs) h2d(ctx->h_unif, uniforms, B * (N + 1) * sizeof(float));
    if (!far_logits) h2d(ctx->h_logits, target_logits, lg_bytes);
    if (draft_probs && !draft_in_place) {
        h2d(ctx->h_draft, draft_probs, lg_bytes);
        draft = ctx->h_draft;
    }
    ok = ok && attn_ok &&
         cudaMemcpyAsync(attn_out, ctx->h_out, q_bytes, cudaMemcpyDeviceToHost, ctx->side) == cudaSuccess;
    const bool joined = cudaEventRecord(ctx->ev_join, ctx->side) == cudaSuccess;
    FspadStatsGeom geom;
    if (far_logits || fspad_scan_inner(ctx->sm_count, batch * n_nodes, n_nodes, c.vocab, draft_probs != nullptr, false)) geom.parent = ctx->h_parent;
    if (far_logits) geom.stage = ctx->h_logits;
    const float *logits = far_logits ? far_logits : ctx->h_logits;
    ok = ok && fspad_launch_stats_partials(ctx, logits, ctx->h_temp, batch * n_nodes, n_nodes, c.vocab, &geom, st) == cudaSuccess;
    ok = ok && fspad_launch_accept_walk(ctx, logits, draft, ctx->h_tokens, ctx->h_parent, ctx->h_temp,
                                        draft_probs ? ctx->h_unif : nullptr, geom, n_nodes, batch, c.vocab, ctx->h_path, ctx->h_nacc,
                                        ctx->h_bonus, st, FspadWalkCompact(), draft_in_place) == cudaSuccess;
    // the compaction rewrites cache rows that the attention reads
    if (!joined || cudaStreamWaitEvent(st, ctx->ev_join, 0) != cudaSuccess || !ok) return give_up(FSPAD_ERR_CUDA);
    if (fspad_launch_kv_compact(ctx, cache, ctx->h_path, ctx->h_nacc, ctx->h_prefix, batch, ctx->h_newlen, st, false) != cudaSuccess)
        return give_up(FSPAD_ERR_CUDA);

    // the device path array has max_nodes entries per sequence, and so has the host one
    d2h(accepted_path, ctx->h_path, B * (size_t)c.max_nodes * sizeof(int));
    d2h(n_accepted, ctx->h_nacc, B * sizeof(int));
    d2h(bonus_token, ctx->h_bonus, B * sizeof(int));
    d2h(new_len, ctx->h_newlen, B * sizeof(int));
    if (!ok) return give_up(FSPAD_ERR_CUDA);
    rc = fspad_status(ctx, stream);                // (waits for the stream)
    return rc == FSPAD_ERR_CUDA ? give_up(rc) : rc;
}

}  // extern "C"
