// Target LM head with the per-node vocabulary scan as its epilogue.
//
// The acceptance stage compares the tree with the target's distribution at every
// tree node (paper, Section "Preliminaries": one target forward over the
// flattened tree, then strict comparison).  The last step of that forward is the
// product of the nodes' final hidden states with the vocabulary matrix; here its
// tiles are reduced to the scan's partial results (maximum, lowest index of the
// maximum, sum of exponentials) as they leave the tensor cores, so the logits
// need not make a round trip through HBM before they are scanned, and need not be
// written at all when every sequence is greedy.
//
//   logits[r][v] = sum_h hidden[r][h] * weight[v][h]      bf16 x bf16 -> fp32
//
// The vocabulary is the M side of the product and the rows are its N side: a pair of CTAs (one cluster, one pair of
// SMs) multiplies 256 vocabulary entries by up to 256 rows at a time with 256 x N x 16 tcgen05.mma.cta_group::2
// instructions, each CTA holding its own 128 vocabulary entries and half of the rows in shared memory.  That serves
// both ends of the range with one kernel:
//   - up to about 250 rows the product is bound by streaming the vocabulary matrix once (2 H V bytes): there is one
//     row tile as wide as the rows need (32, 64, ... 256), so what is not matrix takes little of the ring, and each
//     SM keeps up to ten 16 KB matrix stages in flight;
//   - above that it is a contraction (2 R V H operations).  The rows are cut into the fewest tiles of at most 256,
//     in units of 32 spread evenly (960 rows: 256, 256, 224, 224, nothing multiplied for padding), and the row tiles
//     of one stretch of the vocabulary are neighbouring work items, so HBM gives up the matrix once and L2 the rest.
//     Sharing the row operand between the two SMs is what keeps the tensor cores fed from shared memory: a single
//     CTA's 128 x 256 tile needs 190 bytes per clock (copies in, operands out) where a pair's needs 128.
// A thread of the epilogue holds one vocabulary entry of a row, so the logits leave as whole 128-byte lines whatever
// V is, and a row's statistics over a warp's 32 entries come from one redux, one ballot and a share of a transposing
// butterfly.
// Measured (H = 4096, V = 128256, logits written; before: single CTAs with the rows as the M side, one launch and one
// pass over the matrix per 128 rows): 960 rows 1736 -> 718 us (1.40 PFLOP/s, the power limit; cuBLAS's bare bf16 product
// 700), 480 rows 817 -> 430, 240 rows 416 -> 244, 60 rows 203 -> 201 (5.2 TB/s of matrix).  With the issue loop in one
// lane's branch instead of a whole warp's uniform one the 960-row call took 865 us: 717 cycles per stage against 502
// (the instructions themselves need 512 at the nominal rate); with four epilogue warps instead of eight 920 us.
// Two accumulators in tensor memory: the epilogue of one item runs under the product of the next.  Roles meet only on
// mbarriers; every wait is bounded.
#include <cuda.h>

#include "common.cuh"
#include "umma_common.cuh"

namespace lmh {

using namespace umma;

constexpr int BN = 128;                 // vocabulary entries per CTA and item (one partial result per row and tile)
constexpr int BKE = 64;                 // hidden elements per stage (128 bytes: the swizzle span)
constexpr int STAGE_W = BN * 128;       // bytes of one [128][64] bf16 box of the matrix
constexpr int kMaxTileRows = 256;       // rows of one accumulator
constexpr int kMaxStages = 10;
constexpr int kRingBytes = 200 * 1024;
constexpr int kSlabRows = FSPAD_LM_SLAB_ROWS;   // rows of one launch
constexpr int kEpiWarps = 8;            // two per tensor-memory lane quarter, taking every other 32 rows
constexpr int NT = 64 + 32 * kEpiWarps; // warp 0: copies; warp 1: tensor cores; the rest: epilogue
constexpr uint32_t TMEM_COLS = 512;     // two fp32 accumulators of 256 columns
constexpr float kLog2e = 1.4426950408889634f;

struct Args {
    int R, H, V, n_tiles, rows_per_seq, row0;   // row0: number of the slab's first row in the caller's arrays
    int row_tiles, units, extra;        // row tiles; 32-row units of each; the first `extra` tiles have one unit more
    int n_stages, x_bytes;              // ring stages; bytes of a stage's share of the rows
    const float *temperature;
    float *logits;                      // [R][V] or NULL
    FspadStatsPart *parts;              // [R][n_tiles]
    int *status;
};

struct Shared {
    unsigned long long bar[2 * kMaxStages + 5];
    uint32_t tmem;
    int fail;
    float kk[kSlabRows + 32];           // log2(e) / temperature of every row (the pad covers a last unit's missing rows)
    float pm[4][kMaxTileRows], ps[4][kMaxTileRows];     // one item's statistics by epilogue warp
    int pa[4][kMaxTileRows];
};
constexpr int SMEM_BYTES = kRingBytes + 1024;

// merge of two partial results (maximum, lowest index, sum rescaled to the common maximum)
__device__ __forceinline__ void merge_part(float &m, float &s, int &arg, float om, float os, int oa, float kk)
{
    if (om == -INFINITY) return;
    if (m == -INFINITY) { m = om; s = os; arg = oa; return; }
    const float mn = fmaxf(m, om);
    s = s * exp2f((m - mn) * kk) + os * exp2f((om - mn) * kk);
    if (om > m || (om == m && oa < arg)) arg = oa;
    m = mn;
}

__device__ __forceinline__ float warp_max(float v)      // every lane gets the maximum
{
    float r;
    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

__global__ void __launch_bounds__(NT, 1)
lm_head_stats_kernel(const Args a, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX0,
                     const __grid_constant__ CUtensorMap tmX1)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(16) Shared sh;

    fspad_pdl_wait();
    const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
    const uint32_t rank = cluster_rank();                           // CTA of the pair
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t stage = (uint32_t)(STAGE_W + a.x_bytes);         // [128 vocabulary entries | half of the rows][64]
    const int n_stages = a.n_stages;
    const uint32_t bar0 = smem_u32(&sh.bar[0]);
    auto full = [&](int s) { return bar0 + 8u * (uint32_t)s; };                     // the pair's stage s is filled (rank 0's counts)
    auto empty = [&](int s) { return bar0 + 8u * (uint32_t)(kMaxStages + s); };     // the pair's stage s has been multiplied (both)
    auto accf = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kMaxStages + b); };  // accumulator b is complete (both)
    auto acce = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kMaxStages + 2 + b); };   // ... has been read (rank 0's counts)
    const uint32_t drain = bar0 + 8u * (uint32_t)(2 * kMaxStages + 4);               // used only when a wait has run out
    const int n_k = (a.H + BKE - 1) / BKE;
    const int T = a.row_tiles;
    const int n_items = ((a.n_tiles + 1) / 2) * T;                  // (pair of vocabulary tiles, row tile), row tiles innermost
    const int pair = (int)blockIdx.x >> 1, n_pairs = (int)gridDim.x >> 1;
    const int my_items = pair < n_items ? (n_items - pair + n_pairs - 1) / n_pairs : 0;
    // item j of this pair -> this CTA's first vocabulary entry, first row of the tile and its 32-row units
    auto item = [&](int j, int &v0, int &r0, int &units) {
        const int i = pair + j * n_pairs, rt = i % T;
        v0 = (i / T) * (2 * BN) + (int)rank * BN;
        r0 = 32 * (rt * a.units + min(rt, a.extra));
        units = a.units + (rt < a.extra ? 1 : 0);
    };

    if (tid == 0) {
        for (int i = 0; i < 2 * kMaxStages + 5; ++i)
            mbar_init(bar0 + 8u * i, i >= 2 * kMaxStages + 2 && i < 2 * kMaxStages + 4 ? 2 * kEpiWarps : 1);
        sh.fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    for (int r = tid; r < kSlabRows + 32; r += NT) {
        float t = 1.0f;
        if (r < a.R && a.temperature) t = a.temperature[(a.row0 + r) / a.rows_per_seq];
        if (!(t > 0.0f)) t = 1.0f;
        sh.kk[r] = kLog2e / t;
    }
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     :: "r"(smem_u32(&sh.tmem)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                          // both CTAs' barriers are initialised and their tensor memory is allocated
    tc_fence_after();
    const uint32_t tmem = sh.tmem;
    bool failed = false;

    if (warp == 0) {
        // ================= copy warp: one thread runs the whole loop (and waits on its own) =================
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;                     // flips each time the ring wraps
            bool first = true;                   // the ring's first round waits for nothing
            for (int j = 0; j < my_items; ++j) {
                int v0, r0, units;
                item(j, v0, r0, units);
                const CUtensorMap *mX = units > a.units ? &tmX1 : &tmX0;
                const int half = 16 * units;     // this CTA's share of the tile's rows
                for (int k = 0; k < n_k; ++k) {
                    if (!first && !failed && !mbar_wait_thread(empty(s), ph ^ 1u)) failed = true;
                    if (!failed) {
                        const uint32_t dst = base + (uint32_t)s * stage;
                        if (rank == 0) mbar_expect_tx(full(s), 2u * (uint32_t)(STAGE_W + half * 128));
                        tma_load_2d_pair(dst, &tmW, k * BKE, v0, full(s));
                        tma_load_2d_pair(dst + STAGE_W, mX, k * BKE, r0 + (int)rank * half, full(s));
                    }
                    if (++s == n_stages) { s = 0; ph ^= 1u; first = false; }
                }
            }
            if (failed) sh.fail = 1;
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= tensor-core warp of rank 0: the whole warp runs the loop, one lane issues =================
        if (rank == 0) {
            const bool issuer = elect_one();
            const uint32_t hi = (uint32_t)(make_desc(0, 16) >> 32);
            const uint32_t w_lo = (uint32_t)make_desc(base, 16);
            int s = 0;
            uint32_t ph = 0;
            for (int j = 0; j < my_items; ++j) {
                int v0, r0, units;
                item(j, v0, r0, units);
                const uint32_t idesc = make_idesc_m256((uint32_t)units * 32u);
                const int buf = j & 1;
                // the accumulator is free once both CTAs' epilogues have read the item that used it two items ago
                if (j >= 2 && !failed && !mbar_wait(acce(buf), (uint32_t)((j - 2) >> 1) & 1u)) failed = true;
                tc_fence_after();
                for (int k = 0; k < n_k; ++k) {
                    if (!failed && !mbar_wait(full(s), ph)) failed = true;
                    if (!failed) {
                        tc_fence_after();
                        const uint32_t so = w_lo + (((uint32_t)s * stage) >> 4);
                        if (issuer) {
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks)      // 16 hidden elements = 32 bytes per instruction
                                mma_f16_pair(tmem + (uint32_t)buf * 256u, so + ks * 2, so + (STAGE_W >> 4) + ks * 2, hi, idesc,
                                             (k > 0) || (ks > 0));
                            mma_commit_pair(empty(s));
                            if (k == n_k - 1) mma_commit_pair(accf(buf));
                        }
                        __syncwarp();
                    }
                    if (++s == n_stages) { s = 0; ph ^= 1u; }
                }
            }
            if (failed) sh.fail = 1;
        }
    } else {
        // ================= epilogue warps: one vocabulary entry per thread, 32 rows at a time =================
        const int q = warp & 3;                          // tensor-memory lane quarter this warp may read
        const int et = tid - 64, part = et / 128;        // warps of one quarter share its rows: every other block of 32
        for (int j = 0; j < my_items; ++j) {
            int v0, r0, units;
            item(j, v0, r0, units);
            const int buf = j & 1;
            if (!failed && !mbar_wait(accf(buf), (uint32_t)(j >> 1) & 1u)) failed = true;
            tc_fence_after();
            const int c0 = v0 + q * 32, c = c0 + lane;   // this warp's first vocabulary entry, this lane's
#pragma unroll 1
            for (int blk = part; blk < units; blk += kEpiWarps / 4) {
                float v[32];
                tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)buf * 256u + (uint32_t)blk * 32u, v);
                const int rb = r0 + blk * 32;            // rows rb .. rb + 31 of the slab
                if (a.logits != nullptr && !failed && c < a.V) {
                    float *dst = a.logits + (size_t)rb * a.V + c;
                    const int nr = a.R - rb;
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (i < nr) dst[(size_t)i * a.V] = v[i];
                }
                if (c >= a.V) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = -INFINITY;
                }
                float my_m = -INFINITY;                  // lane i: maximum and its lowest index for row rb + i
                int my_a = 0;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const float m = warp_max(v[i]);
                    const unsigned at = __ballot_sync(0xffffffffu, v[i] == m);
                    if (lane == i) { my_m = m; my_a = max(__ffs((int)at) - 1, 0); }
                    const float ref = m == -INFINITY ? 0.f : m;
                    v[i] = ex2f((v[i] - ref) * sh.kk[rb + i]);
                }
                // 32 sums over 32 lanes: each step halves the columns a lane carries; lane i ends up with row rb + i
#pragma unroll
                for (int h = 16; h >= 1; h >>= 1) {
                    const bool up = (lane & h) != 0;
#pragma unroll
                    for (int i = 0; i < h; ++i) {
                        const float keep = up ? v[i + h] : v[i], give = up ? v[i] : v[i + h];
                        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, h);
                    }
                }
                const int col = blk * 32 + lane;
                sh.pm[q][col] = my_m;
                sh.ps[q][col] = v[0];
                sh.pa[q][col] = c0 + my_a;
            }
            // the accumulator may be overwritten: every lane's loads have completed (tmem_ld32 waits)
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_rank0(acce(buf));
            asm volatile("bar.sync 1, %0;\n" ::"n"(32 * kEpiWarps) : "memory");        // the warps' statistics are in shared memory
            const int tile = v0 / BN;
            if (!failed && tile < a.n_tiles) {
                for (int col = et; col < units * 32; col += 32 * kEpiWarps) {
                    const int row = r0 + col;
                    if (row >= a.R) break;
                    float m = sh.pm[0][col], s = sh.ps[0][col];
                    int arg = sh.pa[0][col];
#pragma unroll
                    for (int w = 1; w < 4; ++w) merge_part(m, s, arg, sh.pm[w][col], sh.ps[w][col], sh.pa[w][col], sh.kk[row]);
                    FspadStatsPart out;
                    out.m = m; out.s = m == -INFINITY ? 0.f : s; out.a = m == -INFINITY ? v0 : arg; out.pad = 0;
                    a.parts[(size_t)row * a.n_tiles + tile] = out;
                }
            }
            asm volatile("bar.sync 1, %0;\n" ::"n"(32 * kEpiWarps) : "memory");        // read before the next item writes
        }
        if (failed) sh.fail = 1;
    }
    fspad_pdl_trigger();
    tc_fence_before();
    __syncthreads();
    if (sh.fail != 0) {
        // a wait ran out: whatever was started asynchronously gets a bounded time to land before the
        // shared and tensor memory go back to the SMs (the pair's copies are all counted by rank 0's barriers)
        if (tid == 0) fspad_report(a.status, FSPAD_ERR_TIMEOUT);
        if (rank == 0 && warp == 0) {
            const long long total = (long long)my_items * n_k;
            for (int s = 0; s < n_stages; ++s) {
                const long long fills = (total - s + n_stages - 1) / n_stages;     // upper bound of the fills started in stage s
                if (fills > 0) (void)mbar_wait(full(s), (uint32_t)(fills - 1) & 1u, 20000);
            }
        } else if (rank == 0 && warp == 1) {
            if (lane == 0) mma_commit_pair(drain);
            (void)mbar_wait(drain, 0u, 20000);
        }
        __syncthreads();
    }
    // neither CTA leaves (or gives up its tensor memory) while the other may still reach it
    cluster_sync_all();
    if (warp != 1) return;
    tc_fence_after();
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(TMEM_COLS) : "memory");
}

// Tile partials -> one partial per output slot.  Slot (row, p) covers the tiles [t0, t1) that the
// caller's geometry gives it; one warp per slot.  With `rows_out` the result goes out as row
// statistics (one slot per row), otherwise as FspadStatsPart into out_parts[row * slots + p].
__global__ void __launch_bounds__(128)
lm_head_merge_kernel(const FspadStatsPart *__restrict__ tile_parts, int R, int n_tiles, int rows_per_seq,
                     const float *__restrict__ temperature, int row0, FspadStatsGeom g, int tile_units,
                     FspadStatsPart *__restrict__ out_parts, float *__restrict__ row_max, double *__restrict__ row_sum,
                     int *__restrict__ row_arg)
{
    // Wait first, then let the successor start: the acceptance walk reads logits in its prologue, and they are complete
    // only when the product kernel is.
    fspad_pdl_wait();
    fspad_pdl_trigger();
    const int lane = threadIdx.x & 31;
    const long long wi = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    const bool as_rows = out_parts == nullptr;
    const int per_row = as_rows ? 1 : g.per_row;
    if (wi >= (long long)R * per_row) return;
    const int r = (int)(wi / per_row), p = (int)(wi % per_row);     // r: row inside this slab
    const int grow = row0 + r;                                       // row in the caller's numbering
    int t0 = 0, t1 = n_tiles;
    if (!as_rows) {
        const int tiles = (int)(g.chunk / tile_units);               // pieces are whole tiles, the last may be shorter
        t0 = p * tiles;
        t1 = min(n_tiles, t0 + tiles);
    }
    float T = temperature ? temperature[grow / rows_per_seq] : 1.0f;
    if (!(T > 0.0f)) T = 1.0f;
    const float kk = lmh::kLog2e / T;
    float m = -INFINITY, s = 0.f;
    int arg = 0x7fffffff;
    // A lane's partials are requested eight at a time, before any of them is merged: the merge carries a
    // dependency from one partial to the next, and with one request per step a row of a thousand tiles was
    // thirty-two trips to L2 one after the other (about 19 us of a 190 us call).
    constexpr int kAhead = 8;
    for (int tb = t0 + lane; tb < t1; tb += 32 * kAhead) {
        int4 v[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int t = tb + 32 * u;
            v[u] = make_int4(__float_as_int(-INFINITY), 0, 0x7fffffff, 0);
            if (t < t1) v[u] = __ldcg(reinterpret_cast<const int4 *>(tile_parts + (size_t)r * n_tiles + t));
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            if (tb + 32 * u < t1) merge_part(m, s, arg, __int_as_float(v[u].x), __int_as_float(v[u].y), v[u].z, kk);
    }
    double sd = 0.0;
    {
        float mm = m;
        int aa = arg;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float om = __shfl_xor_sync(0xffffffffu, mm, off);
            const int oa = __shfl_xor_sync(0xffffffffu, aa, off);
            if (om > mm || (om == mm && oa < aa)) { mm = om; aa = oa; }
        }
        sd = (m == -INFINITY) ? 0.0 : (double)s * (double)exp2f((m - mm) * kk);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sd += __shfl_xor_sync(0xffffffffu, sd, off);
        m = mm;
        arg = aa;
    }
    if (lane == 0) {
        if (as_rows) {
            row_max[grow] = m;
            row_sum[grow] = sd;
            row_arg[grow] = (arg == 0x7fffffff) ? 0 : arg;
        } else {
            FspadStatsPart out;
            out.m = m; out.s = (float)sd; out.a = arg; out.pad = 0;
            out_parts[(size_t)grow * g.slots + p] = out;
        }
    }
}

}  // namespace lmh

int fspad_lm_head_tiles(int V) { return (V + lmh::BN - 1) / lmh::BN; }

// Geometry under which the walk reads the merged partials: pieces of whole tiles, at most 14 per row (the walk keeps the
// masses of 16), cut at the rows; the last piece of a row may be shorter.
FspadStatsGeom fspad_lm_head_geom(int rows, int V, bool vec, int slots)
{
    FspadStatsGeom g;
    g.unit = vec ? 4 : 1;
    g.shift = 0;
    g.upr = V / g.unit;
    g.slots = slots;
    g.total = (long long)rows * g.upr;
    g.threads = FSPAD_STATS_THREADS;            // no scan kernel runs on this geometry; the walk reads the pieces only
    const int n_tiles = fspad_lm_head_tiles(V), tiles = (n_tiles + 13) / 14;
    g.chunk = (long long)tiles * (lmh::BN / g.unit);
    g.per_row = (n_tiles + tiles - 1) / tiles;
    g.n_cta = rows * g.per_row;
    return g;
}

// rows 0 .. R-1 of hidden ([R][H]) against weight ([V][H]); slabs of kSlabRows rows, one launch each
cudaError_t fspad_launch_lm_head(fspad_ctx *ctx, const fspad_bf16 *hidden, const fspad_bf16 *weight, int H, int R,
                                 int rows_per_seq, const float *temperature, float *logits, const FspadStatsGeom *walk_geom,
                                 float *row_max, double *row_sum, int *row_arg, cudaStream_t st)
{
    const int V = ctx->cfg.vocab;
    const int n_tiles = fspad_lm_head_tiles(V);
    if (!ctx->lm_attr_done) {
        cudaError_t e = cudaFuncSetAttribute(lmh::lm_head_stats_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             lmh::SMEM_BYTES);
        if (e != cudaSuccess) return e;
        ctx->lm_attr_done = 1;
    }
    CUtensorMap mW;
    if (!fspad_make_tmap_bf16_2d(&mW, weight, (size_t)H, (size_t)V, lmh::BN, true)) return cudaErrorInvalidValue;
    for (int r0 = 0; r0 < R; r0 += lmh::kSlabRows) {
        const int rs = (R - r0 < lmh::kSlabRows) ? R - r0 : lmh::kSlabRows;
        const int units = (rs + 31) / 32;
        lmh::Args a;
        a.row_tiles = (units + lmh::kMaxTileRows / 32 - 1) / (lmh::kMaxTileRows / 32);
        a.units = units / a.row_tiles; a.extra = units % a.row_tiles;
        const int widest = a.units + (a.extra ? 1 : 0);
        a.x_bytes = widest * 16 * 128;
        a.n_stages = lmh::kRingBytes / (lmh::STAGE_W + a.x_bytes);
        if (a.n_stages > lmh::kMaxStages) a.n_stages = lmh::kMaxStages;
        // a CTA's share of a row tile is 16 rows per unit: one map per tile width
        CUtensorMap mX0, mX1;
        if (!fspad_make_tmap_bf16_2d(&mX0, hidden + (size_t)r0 * H, (size_t)H, (size_t)rs, 16u * (unsigned)a.units) ||
            !fspad_make_tmap_bf16_2d(&mX1, hidden + (size_t)r0 * H, (size_t)H, (size_t)rs, 16u * (unsigned)widest))
            return cudaErrorInvalidValue;
        a.R = rs; a.H = H; a.V = V; a.n_tiles = n_tiles; a.rows_per_seq = rows_per_seq; a.row0 = r0;
        a.temperature = temperature;
        a.logits = logits ? logits + (size_t)r0 * V : nullptr;
        a.parts = ctx->lm_parts;
        a.status = ctx->d_status;
        const int items = (n_tiles + 1) / 2 * a.row_tiles, pairs = ctx->sm_count / 2 > 0 ? ctx->sm_count / 2 : 1;
        const int grid = 2 * (pairs < items ? pairs : items);
        ctx->launches++;
        cudaError_t e = fspad_launch_opt(r0 == 0, lmh::lm_head_stats_kernel, dim3(grid), dim3(lmh::NT), lmh::SMEM_BYTES, st, 2,
                                         a, mW, mX0, mX1);
        if (e != cudaSuccess) return e;
        ctx->launches++;
        const bool as_rows = walk_geom == nullptr;
        FspadStatsGeom g = as_rows ? FspadStatsGeom() : *walk_geom;
        const long long warps = (long long)rs * (as_rows ? 1 : g.per_row);
        e = fspad_launch(lmh::lm_head_merge_kernel, dim3((unsigned)((warps + 3) / 4)), dim3(128), 0, st, 0,
                         (const FspadStatsPart *)ctx->lm_parts, rs, n_tiles, rows_per_seq, temperature, r0, g,
                         as_rows ? 1 : lmh::BN / g.unit, as_rows ? (FspadStatsPart *)nullptr : ctx->st_part, row_max, row_sum,
                         row_arg);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
