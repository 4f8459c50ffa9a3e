// Internal declarations shared by the translation units of libfspad.so.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <utility>

#include "fspad.h"

#define FSPAD_MAX_NODES 64           /* nodes of a tree on the one-mask-word paths */
#define FSPAD_MAX_NODES_WIDE 256     /* nodes of a tree, any call of the verify step */
#define FSPAD_MAX_CANDIDATES 1024
#define FSPAD_MAX_FRONTIER 16      /* frontier nodes per sequence, and top-k per row, of a draft step */
#define FSPAD_HEAD_DIM 128
#define FSPAD_STATS_THREADS 256
#define FSPAD_LM_SLAB_ROWS 1024    /* rows of one launch of the LM-head product (more rows: several launches) */

// Scratch and bookkeeping owned by a context (all device pointers unless noted).
struct fspad_ctx {
    fspad_config cfg;
    int device;
    int sm_count;
    float scale;              // softmax scale actually used
    long long launches;       // host counter of kernels launched

    int *d_status;            // first device-detected error (0 = none)

    // split-KV attention partials
    int attn_max_splits;
    int attn_attr_done;       // dynamic shared-memory limit raised for the attention kernels
    // TMA descriptors of the K and V cache planes last seen (re-encoded when they change)
    alignas(64) unsigned char attn_tmap_k[128];
    alignas(64) unsigned char attn_tmap_v[128];
    alignas(64) unsigned char attn_tmap_k_half[128];
    const void *attn_tmap_kptr, *attn_tmap_vptr;
    size_t attn_tmap_rows;
    int attn_tmap_ok;
    float *part_o;            // [batch][Hkv][splits][M][d]
    float *part_ml;           // [batch][Hkv][splits][M][2]  (running max in log2 units, sum)
    int *attn_done;           // CTAs of the attention whose partials are written; zero between calls

    // per-node vocabulary scan
    int stats_slots;          // partial slots per row in st_part
    struct FspadStatsPart *st_part;   // [rows][stats_slots]
    float *row_max;           // [rows]
    double *row_sum;
    int *row_arg;
    int walk_cluster;         // largest cluster of the sampling walk (0 = not probed yet)
    int walk_fit;             // how many of that size the device holds at once

    // whole-step entry point: attention runs on `side`, forked from and joined into the caller's stream
    cudaStream_t side;
    cudaEvent_t ev_fork, ev_join;

    // LM head: per-(row, vocabulary tile) partials of one slab of rows, [min(max rows, slab)][tiles]
    struct FspadStatsPart *lm_parts;
    int lm_attr_done;
    int fs_attr_done;         // dynamic shared-memory limit raised for the Feature Sampler's product kernel

    void *dx_part;            // draft step: per-piece top-k lists [max_batch * 16 rows][pieces][16], 64-bit sort keys (0: none)
    int *dx_done;             // draft step: finished pieces of each sequence [max_batch]; zero between calls
    float *dx_front;          // draft step: a frontier put aside, values and candidates [2][max_batch][16]

    // device staging for the host entry point (h_ready: every buffer below is allocated)
    int h_ready;
    fspad_bf16 *h_q, *h_tk, *h_tv, *h_out;
    int *h_parent, *h_prefix, *h_tokens, *h_path, *h_nacc, *h_bonus, *h_newlen;
    float *h_logits, *h_draft, *h_temp, *h_unif;
};

// One CTA's contribution to a row of the vocabulary scan.
struct FspadStatsPart {
    float m;   // maximum over the CTA's part of the row
    float s;   // sum of exp2((x - m) * log2(e) / T) over that part
    int a;     // lowest index attaining m
    int pad;
};

// How the flat [rows x V] logits array is cut into equal per-CTA ranges.
struct FspadStatsGeom {
    int unit;          // floats per load unit: 4 (128-bit loads) or 1
    int shift;         // 1: V is no multiple of 4, a row's units count from the 16-byte boundary at or before its first token
    int upr;           // units per row (with shift: room for up to three positions in front of it)
    int n_cta;         // CTAs in the grid
    int slots;         // partial slots per row (capacity)
    long long chunk;   // units per CTA
    long long total;   // rows * upr
    int per_row;       // > 0: ranges are cut at the rows, this many per row (the last may be shorter); 0: they may cross rows
    int threads;       // threads per CTA of the scan: FSPAD_STATS_THREADS, or half of it for a small array
    // The trees [rows / rows_per_seq][rows_per_seq] the rows belong to: rows of nodes without children (other than a root) have
    // then no partials, and whoever walks into such a node looks at its row itself.  NULL: every row has them.  Set by the
    // caller of fspad_launch_stats_partials where the scan is to go by them, put back to NULL there if it cannot.
    const int *parent = nullptr;
    // With the trees: the logits lie in host memory, and the rows that the scan reads are left here, [rows][V] on the device.  NULL: they
    // are on the device.  Set by the caller, too.
    float *stage = nullptr;
};

// small_ctas: the scan may use CTAs of half the size when the array is small (the pieces, one of which the
// acceptance walk's bonus draw sweeps, halve with them; on a large array the smaller CTAs cost bandwidth:
// 5.93 against 6.20 TB/s on 960 rows of 128256)
// aligned: the array starts on a 16-byte boundary (otherwise it is read float by float)
static inline FspadStatsGeom fspad_stats_geom(int sm_count, int rows, int V, bool aligned, int slots, bool small_ctas = false)
{
    FspadStatsGeom g;
    g.unit = aligned ? 4 : 1;
    g.shift = aligned && V % 4 != 0;
    g.upr = g.shift ? (V + 6) / 4 : V / g.unit;
    g.slots = slots;
    g.total = (long long)rows * g.upr;
    g.threads = FSPAD_STATS_THREADS;
    // up to 32 units per thread of one wave at 1024 threads per SM
    if (small_ctas && g.total <= (long long)sm_count * 1024 * 32) g.threads = FSPAD_STATS_THREADS / 2;
    long long n = (long long)sm_count * (1024 / g.threads);   // 1024 threads per SM, one wave
    const long long by_size = (g.total + g.threads - 1) / g.threads;   // at least one unit per thread
    if (n > by_size) n = by_size;
    if (n < 1) n = 1;
    if (g.shift) {
        // Rows that start anywhere are always cut at the rows: into 16 pieces where every SM gets a CTA that way (see
        // below), else into what one wave holds; with more rows than CTAs in a wave, into the number of pieces (up to
        // 8) that leaves the last wave fullest.
        long long k = n / rows;
        if (k > 16 && (long long)rows * 16 >= sm_count) k = 16;
        if (k > slots - 2) k = slots - 2;
        if (k < 1) {
            double best = 0.0;
            for (int t = 1; t <= 8; ++t) {
                const long long waves = ((long long)rows * t + n - 1) / n;
                const double full = (double)rows * t / (double)(waves * n);
                if (full > best + 0.02) { best = full; k = t; }
            }
        }
        g.chunk = (g.upr + k - 1) / k;
        g.per_row = (int)((g.upr + g.chunk - 1) / g.chunk);
        g.n_cta = rows * g.per_row;
        return g;
    }
    g.chunk = (g.total + n - 1) / n;
    // A CTA whose range crosses a row boundary runs its reduction sequence twice and finishes about a
    // microsecond behind the others.  Where a row divides evenly into a whole number k of pieces such that
    // rows * k CTAs still fill three quarters of the wave, ranges are cut at the rows instead.
    if (rows >= 1 && n >= rows) {
        bool cut = false;
        // The acceptance walk keeps the masses of at most 16 pieces per row for its bonus draw (with more it
        // sweeps the whole row): with few rows, 16 pieces per row are preferred to a full wave as long as
        // every SM still gets a CTA.
        if (n / rows > 16 && (long long)rows * 16 >= sm_count) {
            for (long long k = 16; k >= 8 && !cut; --k)
                if (g.upr % k == 0) { g.chunk = g.upr / k; cut = true; }
        }
        for (long long k = n / rows; !cut && k >= 1 && (long long)rows * k * 4 >= n * 3; --k)
            if (g.upr % k == 0) { g.chunk = g.upr / k; cut = true; }
    }
    // a row may be shared by at most `slots` CTAs
    const long long min_chunk = (g.upr + (slots - 2) - 1) / (slots - 2);
    if (g.chunk < min_chunk) g.chunk = min_chunk;
    g.n_cta = (int)((g.total + g.chunk - 1) / g.chunk);
    g.per_row = g.upr % g.chunk == 0 ? (int)(g.upr / g.chunk) : 0;
    return g;
}

// Rows of the nodes that have children, of a batch of trees.
#define FSPAD_INNER_MAX_ROWS 8192      /* one bit each, a word to a thread of the scan's CTAs */
#define FSPAD_INNER_LIST 128           /* rows one CTA may be given pieces of */
// How the rows of the nodes with children are cut: into at most 16 pieces each, as many as the walk merges at once, with two units for
// each thread of a CTA at least.  How many rows there are is known to the kernel alone.  Where a CTA for every piece of every row is
// one wave, most of which leaves at once, the CTAs are the pieces; else the kernel numbers the rows first and may cut them into fewer
// (16 and 30 rows of 128256: the step 0.7 us shorter without; 60 rows, in two waves, 2 us longer).
static inline FspadStatsGeom fspad_stats_geom_inner(int sm_count, int rows, int V, int slots, const int *parent, float *stage)
{
    FspadStatsGeom g;
    g.unit = 4;
    g.shift = V % 4 != 0;
    g.upr = g.shift ? (V + 6) / 4 : V / 4;
    g.slots = slots;
    g.total = (long long)rows * g.upr;
    int k = g.upr / (2 * FSPAD_STATS_THREADS);
    k = k < 2 ? 2 : k > 16 ? 16 : k;
    g.chunk = (g.upr + k - 1) / k;
    g.per_row = k;
    const long long n = (long long)sm_count * (1024 / FSPAD_STATS_THREADS);
    g.threads = FSPAD_STATS_THREADS;
    g.n_cta = (int)((long long)rows * k <= n ? rows * k : n);
    g.parent = parent;
    g.stage = stage;
    return g;
}
// Whether the scan of these rows can go by the trees, and whether it does.  Up to nine rows (fewer than a sixteenth of the SMs) the scan
// of all rows cuts a row into more pieces than the walk merges at once, and the draw from more than 16 pieces reads the whole row
// again: 8 rows alone, all rows and by the trees, 22.5 and 16.0 us at 128256 tokens, 17.1 and 13.7 at 32000 (up to 8192 tokens there are no more than 16).
//   Otherwise the rows left out stand against what finding the others costs (1.3 to 1.6 us) and, of a greedy walk, its look at the row of its last
// node (2.4 us, which in a step passes beside the attention; `alone` says that nothing of the call does).  The gain grows with the array, and with
// the trees: of up to 11 nodes half and more have children, of 60 a fifth.  The lines, in thousands of logits, lie where trees of branching two
// to ten were no slower (acceptance, or step of 8 KV heads and 1 K to 2 K keys; us from a graph, all rows and by the trees):
//   sampled, a step   40 x 32000 twice 31.1 and 28.6, 24 x 50257 four times 33.4 and 31.4, 24 x 32000 twice 23.4 and 25.0; 8 x 128256 eight times 39.3 and 35.8
//   sampled, alone    40 x 32000 four times 31.4 and 29.7, 130 x 32000 21.9 and 24.7, 24 x 32000 eight times 26.7 and 26.7, 16 x 32000 eight times 21.3 and 21.9; 8 x 32000 16 times 26.6 and 29.3
//   greedy, a step    40 x 32000 twice 21.6 and 19.2, 24 x 32000 eight times 31.2 and 31.2; 16 x 50257 eight times 29.5 and 31.0, 8 x 50257 16 times 34.5 and 38.0
//   greedy, alone     40 x 32000 four times 11.0 and 10.3, 24 x 50257 eight times 13.0 and 11.6, 60 x 50257 twice 8.9 and 10.2; 16 x 32000 16 times 11.0 and 11.6
// Rows whose length is no multiple of four are always cut at the rows by the scan of all of them, which makes it the faster one of small
// arrays.  Where the CTAs are the pieces nothing is numbered: 24 x 128256, 32 x 128256 (16 nodes twice) in a sampled step 24.4 and 23.7, 28.2 and 24.8
// (alone 17.5 and 18.5, 22.6 and 22.1).
// What the kernel finds is not known here: a tree most of whose nodes have children (a chain) gains nothing from it.  Chains of 40 to 60
// nodes: acceptance alone 22.0 and 24.2 (60 x 128256 sampled), 12.3 and 12.3 (greedy), 17.5 and 20.5 at worst (40 x 50257 eight times, greedy);
// steps level to 7 % longer.
static inline bool fspad_scan_inner_fits(int sm_count, int rows, int V)
{
    return rows <= FSPAD_INNER_MAX_ROWS && (long long)rows * (V + 6ll) < 1ll << 31 &&
           rows / (sm_count * (1024 / FSPAD_STATS_THREADS)) + 2 <= FSPAD_INNER_LIST;
}
static inline bool fspad_scan_inner(int sm_count, int rows, int nodes, int V, bool may_sample, bool alone)
{
    if (!fspad_scan_inner_fits(sm_count, rows, V)) return false;
    if (rows * 16 < sm_count && V > 16 * 4 * (FSPAD_STATS_THREADS / 2)) return true;
    const bool odd = V % 4 != 0, one_wave = rows * 16 <= sm_count * (1024 / FSPAD_STATS_THREADS);
    int line;                                    // thousands of logits
    if (may_sample) line = alone ? nodes >= 24 ? 4400 : nodes >= 12 ? 6000 : 8000 : nodes >= 32 ? 2500 : nodes >= 12 ? 4000 : 8000;
    else if (alone) line = nodes >= 32 ? odd ? 9500 : 5000 : nodes >= 12 ? 9500 : 25000;
    else line = nodes >= 32 ? odd ? 4000 : 2500 : nodes >= 12 && !odd ? 6000 : 16000;
    const int few = may_sample && !alone ? 1500 : 4000;
    if (one_wave && (may_sample || !alone) && few < line) line = few;
    return (long long)rows * V >= 1000ll * line;
}

// How many of the first n units of four positions of row `row`, from position j0 of it on, can be loaded whole: the last one may reach
// into the next rows (its caller leaves out what is not the row's), but not past the end of the array [rows][V].
#ifdef __CUDACC__
__device__
#endif
static inline int fspad_whole_units(int rows, int row, int V, int j0, int n)
{
    const int behind = (rows - 1 - row) * V, whole = (V - j0 + (behind < 3 ? behind : 3)) >> 2;
    return n < whole ? n : whole;
}

#ifdef __CUDACC__
// ---- rows read 16 bytes at a time whatever their length ----
// Positions j .. j + 3 of a row whose valid positions are [0, hi); x + j is 16-byte aligned.  A group that reaches past either
// end is read element by element (nothing outside the row is touched), with `pad` for the rest.
static __device__ __noinline__ float4 fspad_edge4(const float *__restrict__ x, int j, int hi, float pad)
{
    float4 r = make_float4(pad, pad, pad, pad);
    if (j >= 0 && j < hi) r.x = x[j];
    if (j + 1 >= 0 && j + 1 < hi) r.y = x[j + 1];
    if (j + 2 >= 0 && j + 2 < hi) r.z = x[j + 2];
    if (j + 3 >= 0 && j + 3 < hi) r.w = x[j + 3];
    return r;
}
__device__ __forceinline__ float4 fspad_load4(const float *__restrict__ x, int j, int hi, float pad)
{
    if (j >= 0 && j + 4 <= hi) return __ldg(reinterpret_cast<const float4 *>(x + j));
    if (j + 4 <= 0 || j >= hi) return make_float4(pad, pad, pad, pad);
    return fspad_edge4(x, j, hi, pad);
}

// A row that an earlier kernel may still be writing when this one starts: read behind fspad_pdl_wait, and by plain loads.  The loads
// above go by the read-only path, which is for data that nobody writes during the reading kernel's life.  (A type of its own, so that
// such a row cannot come to them.)
struct FspadLateRow {
    const float *p;
    __device__ __forceinline__ FspadLateRow operator+(size_t n) const { return FspadLateRow{p + n}; }
    __device__ __forceinline__ float operator[](int j) const { return p[j]; }
};
static __device__ __noinline__ float4 fspad_late_edge4(FspadLateRow x, int j, int hi, float pad)
{
    float4 r = make_float4(pad, pad, pad, pad);
    if (j >= 0 && j < hi) r.x = x[j];
    if (j + 1 >= 0 && j + 1 < hi) r.y = x[j + 1];
    if (j + 2 >= 0 && j + 2 < hi) r.z = x[j + 2];
    if (j + 3 >= 0 && j + 3 < hi) r.w = x[j + 3];
    return r;
}
__device__ __forceinline__ float4 fspad_load4(FspadLateRow x, int j, int hi, float pad)
{
    if (j >= 0 && j + 4 <= hi) return *reinterpret_cast<const float4 *>(x.p + j);
    if (j + 4 <= 0 || j >= hi) return make_float4(pad, pad, pad, pad);
    return fspad_late_edge4(x, j, hi, pad);
}

// Merge the per-CTA partials of one row (warp-collective: all 32 lanes call it and all get
// the result): maximum, its lowest index, and the sum of exponentials rescaled to that
// maximum (k = log2(e)/T).  Every lane fetches up to two partial slots, so the loads of a
// row are in flight together instead of one after another.
__device__ __forceinline__ void fspad_stats_merge_warp(const FspadStatsPart *__restrict__ parts,
                                                       const FspadStatsGeom &g, int row, float k, int lane,
                                                       float &M, double &S, int &A)
{
    int cnt = g.per_row;                                    // <= g.slots <= 64
    if (cnt == 0) {
        const long long r0 = (long long)row * g.upr;
        cnt = (int)((r0 + g.upr - 1) / g.chunk) - (int)(r0 / g.chunk) + 1;
    }
    const FspadStatsPart *p = parts + (size_t)row * g.slots;
    float m0 = -INFINITY, m1 = -INFINITY, s0 = 0.f, s1 = 0.f;
    int a0 = 0x7fffffff, a1 = 0x7fffffff;
    if (lane < cnt) {
        const int4 v = __ldcg(reinterpret_cast<const int4 *>(p + lane));
        m0 = __int_as_float(v.x); s0 = __int_as_float(v.y); a0 = v.z;
    }
    if (lane + 32 < cnt) {
        const int4 v = __ldcg(reinterpret_cast<const int4 *>(p + lane + 32));
        m1 = __int_as_float(v.x); s1 = __int_as_float(v.y); a1 = v.z;
    }
    float m = m0;
    int a = a0;
    if (m1 > m || (m1 == m && a1 < a)) { m = m1; a = a1; }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, off);
        const int oa = __shfl_xor_sync(0xffffffffu, a, off);
        if (om > m || (om == m && oa < a)) { m = om; a = oa; }
    }
    double s = 0.0;
    if (m0 != -INFINITY) s += (double)s0 * (double)exp2f((m0 - m) * k);
    if (m1 != -INFINITY) s += (double)s1 * (double)exp2f((m1 - m) * k);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    M = m;
    S = s;
    A = (a == 0x7fffffff) ? 0 : a;
}

#endif

// ---- programmatic dependent launch -----------------------------------------------------
// Most kernels of the library are launched with the programmatic-serialization attribute and
// follow one rule: a kernel lets its successor start launching at once (fspad_pdl_trigger) and
// touches global memory only after the whole preceding kernel of the stream has completed and
// flushed (fspad_pdl_wait).  Launch latency and the memory-free part of a prologue (barrier
// set-up, tensor-memory allocation, table fills) then overlap the tail of the previous kernel,
// while results stay exactly those of plain stream order.
// The acceptance walk is the exception: it reads the caller's arrays (trees, logits, draft rows) before its wait.  It may,
// because the two kernels that can precede it, the vocabulary scan and the LM head's merge, let it start only after their own
// wait, when everything queued before them is complete, and themselves write nothing but what the walk reads after its wait and not by
// the read-only path: scan partials and, of logits in host memory, the rows that the scan brings to the device (FspadLateRow).  The attention of a step called as one is the other: launched behind the walk, it starts when every CTA of the
// walk has, reads what was complete before the scan started, and waits for the walk at its end.  The merge of its key ranges reads
// the partials as soon as a count of the attention's CTAs says that they are there, and waits for the attention at its end.  Kernels whose predecessor is not one kernel of the same stream (behind a fork, a join or a copy) may be
// launched without the attribute.
#ifdef __CUDACC__
__device__ __forceinline__ void fspad_pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void fspad_pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
static inline cudaError_t fspad_launch_opt(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                           cudaStream_t st, unsigned cluster_x, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    if (cluster_x > 0) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster_x; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
static inline cudaError_t fspad_launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                       cudaStream_t st, unsigned cluster_x, Args &&...args)
{
    return fspad_launch_opt(true, kernel, grid, block, smem, st, cluster_x, std::forward<Args>(args)...);
}
#endif

static inline cudaStream_t fspad_stream(void *s) { return reinterpret_cast<cudaStream_t>(s); }

// Record the first device-side error; later ones are dropped.
__device__ __forceinline__ void fspad_report(int *status, int err)
{
    atomicCAS(status, 0, err);
}

// launchers implemented in the kernel translation units (return cudaError_t)
cudaError_t fspad_launch_accept_stats(fspad_ctx *ctx, const float *logits, const float *temperature,
                                      int rows, int rows_per_seq, int V, float *row_max,
                                      double *row_sum, int *row_arg, cudaStream_t st);
// cache != NULL: the walk also compacts the accepted path's rows of `cache` (all layers of the context) and
// writes new_len; the caller then launches no compaction
struct FspadWalkCompact {
    fspad_bf16 *cache = nullptr;
    const int *prefix_len = nullptr;
    int *new_len = nullptr;
};
cudaError_t fspad_launch_accept_walk(fspad_ctx *ctx, const float *logits, const float *draft,
                                     const int *tokens, const int *parent, const float *temperature,
                                     const float *uniforms, const FspadStatsGeom &geom, int N, int B, int V,
                                     int *path, int *n_acc, int *bonus, cudaStream_t st, FspadWalkCompact kv = {},
                                     bool draft_far = false);   // draft_far: the draft rows lie in host memory
// pdl = false: launched as a plain dependent of what precedes it in the stream (griddepcontrol.wait is
// then a no-op; the guarantee its successor relies on holds either way)
cudaError_t fspad_launch_stats_partials(fspad_ctx *ctx, const float *logits, const float *temperature,
                                        int rows, int rows_per_seq, int V, FspadStatsGeom *geom,
                                        cudaStream_t st, bool pdl = true, int sms = 0);   // sms > 0: one wave on that many SMs
cudaError_t fspad_launch_tree_build(fspad_ctx *ctx, const int *cand_parent, const int *cand_token,
                                    const float *cand_logp, const int *root_token, int n_cand, int n_nodes,
                                    int B, int *parent_out, int *token_out, int *cand_out,
                                    unsigned long long *anc_out, int *n_out, cudaStream_t st);
int fspad_draft_expand_pieces(int V);
cudaError_t fspad_launch_draft_expand(fspad_ctx *ctx, const float *logprobs, const float *frontier_logp,
                                      const int *frontier_cand, int F, int k, int width, int base, int cap, int B,
                                      int *cand_parent, int *cand_token, float *cand_logp, int *next_cand,
                                      float *next_logp, cudaStream_t st);
cudaError_t fspad_launch_kv_compact(fspad_ctx *ctx, fspad_bf16 *cache, const int *path,
                                    const int *n_acc, const int *prefix_len, int B, int *new_len,
                                    cudaStream_t st, bool pdl = true);
// A cache kept as a pool of 128-row blocks: table[b * stride + i] is the block with rows 128 i .. 128 i + 127
// of sequence b (table == NULL: contiguous cache).
// early: the attention is launched beside the kernel before it in the stream, which has only been started when all that
// precedes the two of them, and so every input of the attention, is complete; the attention's end waits for that kernel's.
// alone: nothing else of the call runs beside the attention, which then leaves its row tiles to lone CTAs (see fspad_attn_pairs).
struct FspadPaged {
    const int *table;
    int stride, n_blocks;
    bool early = false, alone = false;
};
// sms: how many SMs the call may fill with CTAs (0 = all of them).  merge_pdl: the merge kernel is a programmatic
// dependent of the attention kernel (its CTAs become resident, waiting, as the attention's last CTAs finish).
cudaError_t fspad_launch_tree_attn(fspad_ctx *ctx, const fspad_bf16 *q, const fspad_bf16 *kc,
                                   const fspad_bf16 *vc, const fspad_bf16 *tk, const fspad_bf16 *tv,
                                   const int *parent, const int *prefix_len, int N, int B,
                                   fspad_bf16 *out, cudaStream_t st, int sms = 0, FspadPaged paged = FspadPaged{nullptr, 0, 0},
                                   bool merge_pdl = true);
cudaError_t fspad_launch_tree_scatter(fspad_ctx *ctx, fspad_bf16 *cache, const fspad_bf16 *tk,
                                      const fspad_bf16 *tv, const int *prefix_len, int N, int B,
                                      cudaStream_t st);
int fspad_attn_ranges(const fspad_ctx *ctx, int N, int B, int sms, int chunks, bool alone);   // key ranges per row of sequences of up to that many chunks
int fspad_attn_umma_splits(const fspad_ctx *ctx, int N, int B, int sms = 0);      // ... of a step's attention, by the context's max_len
bool fspad_attn_pairs(const fspad_ctx *ctx, int N, int B, int sms = 0);      // row tiles go in pairs of CTAs
int fspad_attn_mtiles(const fspad_ctx *ctx, int N, int B, int sms = 0);     // row tiles (CTAs) per kv head and key range
int fspad_lm_head_tiles(int V);
size_t fspad_feature_sampler_scratch_floats(int rows, int H, int I);
cudaError_t fspad_launch_feature_sampler(fspad_ctx *ctx, const fspad_bf16 *f, const fspad_bf16 *e, const fspad_bf16 *wup,
                                         const fspad_bf16 *wgate, const fspad_bf16 *wdown, int R, int H, int I,
                                         fspad_bf16 *inter, fspad_bf16 *eta, float *scratch, cudaStream_t st);
FspadStatsGeom fspad_lm_head_geom(int rows, int V, bool vec, int slots);
// LM head over R rows; with walk_geom the merged partials go to the context's scan scratch in that
// geometry (for the acceptance walk), otherwise to row_max / row_sum / row_arg
cudaError_t fspad_launch_lm_head(fspad_ctx *ctx, const fspad_bf16 *hidden, const fspad_bf16 *weight, int H, int R,
                                 int rows_per_seq, const float *temperature, float *logits, const FspadStatsGeom *walk_geom,
                                 float *row_max, double *row_sum, int *row_arg, cudaStream_t st);
int fspad_walk_ctas(fspad_ctx *ctx, int B, int V);   // CTAs of the sampling walk for B sequences
cudaError_t fspad_launch_wait_selftest(fspad_ctx *ctx, int polls, cudaStream_t st);
cudaError_t fspad_launch_walk_wait_selftest(fspad_ctx *ctx, int polls, cudaStream_t st);
cudaError_t fspad_launch_attn_umma_split(fspad_ctx *ctx, const fspad_bf16 *q, const fspad_bf16 *kc,
                                         const fspad_bf16 *vc, const fspad_bf16 *tk, const fspad_bf16 *tv,
                                         const int *parent, const int *prefix_len, int N, int B, int sms, int n_splits,
                                         float scale_log2, fspad_bf16 *out, cudaStream_t st, FspadPaged paged);
cudaError_t fspad_launch_kv_append(fspad_ctx *ctx, fspad_bf16 *cache, const fspad_bf16 *tree_kv, const int *path,
                                   const int *n_acc, const int *prefix_len, int N, int B, int *new_len, cudaStream_t st);
cudaError_t fspad_launch_kv_compact_paged(fspad_ctx *ctx, fspad_bf16 *pool, FspadPaged paged, const int *path,
                                          const int *n_acc, const int *prefix_len, int B, int *new_len, cudaStream_t st);
