// Tree-masked verify attention on the 5th-generation tensor cores (paper,
// Section "Preliminaries": the target processes the flattened token tree under
// the attention mask built from the tree).
//
// Split-KV flash-decode with tcgen05: all query rows that share a kv head (tree
// node x GQA group member) are cut into row tiles of 128, one CTA each; where the
// row tiles alone fill the SMs, two neighbouring ones go to a pair of CTAs as one
// tile of 256 rows (cta_group::2).  Keys are consumed in chunks of 128.  Per chunk:
// S = Q K^T is one chain of eight tcgen05.mma (128 or 256 x 128 x 16, bf16 -> fp32)
// into tensor memory; two softmax threads per query row, 64 keys each, read its
// scores back with tcgen05.ld, apply the ancestor mask (only on chunks that reach
// past the cached prefix) and the softmax in registers, and write P as packed bf16
// pairs back into tensor memory, over the scores; O += P V is a second chain of
// eight tcgen05.mma whose A operand is read from tensor memory and whose B operand
// is V in its [key][d] layout (MN-major).  O stays in tensor memory across chunks.
// The work is split over three kinds of warps that meet only on mbarriers (see the
// kernel's comment); K/V chunks go through a ring of 128-byte-swizzled tiles (three
// whole chunks in a lone CTA, half of each of five in a pair's): one chunk of the prefix, then from the last one
// down, filled by TMA, as Q is; only the chunks with rows of an explicit tree array or
// zero padding, which come early, are gathered with 16-byte asynchronous copies, and
// Q where a group of query heads does not divide the tile.  Where a row's keys are
// split over several CTAs the partials are merged by the combine kernel; with one
// range per row the kernel writes the result itself.
//
// What bounds it.  A chunk takes a CTA 2000 cycles: the softmax threads' own chain (wait,
// scores from tensor memory, maximum, 64 exponentials, P back, arrival: 1500 to 1600 busy, of which
// 1024 are the special-function units' when both groups are at it), beside 1050 of the tensor cores.  Around the
// loop stood 9600 cycles to the first scores (18500 in a pair), 5500 and 4700 of the tail's gather by the copy warp and 4000 (7000)
// behind the last product, before Q came by TMA, the gather went ahead of the loop and the rows left as whole lines.  One B200, us a
// call, that kernel and this one: 52 heads and 4 K keys 34.2 -> 29.9, 8 heads of 8 and 8 K 32.6 -> 28.6, 16 sequences of 2.2 K
// 70.3 -> 56.8, four paged sequences of 130 nodes and 1.3 K keys 74.2 -> 39.1.
//
// Every wait on an mbarrier is bounded; on expiry the CTA records
// FSPAD_ERR_TIMEOUT, skips the remaining tensor-core work, frees its tensor
// memory and returns.
#include <cuda.h>

#include "common.cuh"
#include "umma_common.cuh"

namespace umma {

constexpr int D = FSPAD_HEAD_DIM;      // 128
constexpr int BM = 128;                // query rows per CTA
constexpr int BK = 128;                // keys per chunk
constexpr int NT = 320;                // threads per CTA: two per query row + a copy warp + a tensor-core warp
constexpr int HALF = 128 * 128;        // bytes of one [128 rows][64 bf16] half tile
constexpr int TILE = 2 * HALF;         // bytes of one [128][128] bf16 tile
// K / V chunks in flight: a lone CTA holds whole ones, a pair's CTA half of each
__host__ __device__ constexpr int ring_slots(bool pair) { return pair ? 5 : 3; }
constexpr int smem_bytes(bool pair) { return TILE + 2 * ring_slots(pair) * (pair ? HALF : TILE) + 1024; }   // Q, K ring, V ring + alignment slack
constexpr uint32_t TMEM_COLS = 512;    // S/P of group 0, of group 1: columns 0..255; O of group 0, of group 1: 256..511
constexpr float kLazyLog2 = 8.f;        // a row's reference maximum may lag its true maximum by this much (log2)
struct Args {
    const fspad_bf16 *q, *kc, *vc, *tk, *tv;
    const int *parent, *prefix_len;
    int N, Hq, Hkv, G, M, max_len, n_splits, mtiles, use_tma, q_tma;
    int early;                          // launched beside its predecessors in the stream: they have read everything this kernel needs to be complete
    int longest_first;                  // the launch needs several waves of CTAs: blockIdx.z counts the sequences from the longest down
    // paged cache: the planes are pools of 128-row blocks [n_blocks][Hkv][128][d] and block_table[b][i] names
    // the block that holds rows 128 i .. 128 i + 127 of sequence b (NULL: contiguous planes)
    const int *block_table;
    int table_stride, n_blocks;
    float scale_log2;
    float *part_o, *part_ml;
    fspad_bf16 *out;                    // one key range per row: the result itself, and no partials (NULL otherwise)
    int *done;                          // counts the CTAs whose partials are written, for a merge that does not wait for this kernel's end (or NULL)
    int *status;
};

// byte offset of 16-byte chunk c (0..15) of row r inside a [128][128] bf16 tile stored as two
// 128-byte-swizzled halves (columns 0..63 | 64..127), each [128 rows][128 bytes]
__device__ __forceinline__ uint32_t tile_off(int r, int c)
{
    return (uint32_t)((c >> 3) * HALF + r * 128 + (((c & 7) ^ (r & 7)) << 4));
}


// Roles.  Warps 0-7 are the softmax warps, in two groups of four (128 threads, one query row per
// thread, a warp reaching the tensor-memory lane quarter given by its index modulo 4).  Group g
// owns keys 64 g .. 64 g + 63 of every chunk: its half of each score buffer, its own running
// reference maximum, sum and O accumulator, merged with the other group's by log-sum-exp when the
// loop ends; ahead of the loop they gather what TMA cannot describe.  Warp 8 is the copy warp: it issues every TMA copy.  Warp 9 is the tensor-core warp: all its lanes run the issue loop and
// one elected lane issues every tcgen05.mma (in a pair, rank 0's for both); the warp owns the tensor memory.
// Tensor memory: columns [128 p, 128 p + 128) hold the fp32 scores S of the chunks of parity p, the
// 64 columns at 128 p + 64 g being group g's, and then, written over the first 32 of those, P_g as
// packed bf16 pairs, which the second product reads directly as its A operand; columns
// [256 + 128 g, 384 + 128 g) hold O_g.
// With two score buffers the scores of chunk c + 1 are complete long before the groups have
// finished chunk c, and O_g += P V runs under the group's next softmax: a group never waits for
// the tensor cores unless it has to rescale O.
// The sides meet only on mbarriers, never on a CTA-wide barrier inside the loop:
//   kfull/vfull(b)  K / V ring slot b filled (TMA bytes, or one arrival)     tensor-core warp waits
//   kfree/vfree(b)  both S (both P V) of the chunk in slot b complete        copy warp waits
//   sfull(p)        S of a chunk of parity p complete (tcgen05.commit)       both groups wait
//   pfull(g, p)     P_g written and O_g rescaled by the 4 warps of group g    tensor-core warp waits
//   odone(g, p)     O_g += P_g V of a chunk of parity p complete             group g waits (rescale, end)
// A new phase of a barrier can only begin after every side that waits on it has seen the previous
// one (a parity wait must never fall two phases behind).
// Tensor-core order: S(0) S(1) | PV_0(0) PV_1(0) S(2) | PV_0(1) PV_1(1) S(3) | ...
// PAIR: two CTAs of a cluster (two SMs) take two neighbouring row tiles of the same keys as one 256-row tile
// (cta_group::2): each keeps its own rows' Q, scores, P and O, and holds keys 64 r .. 64 r + 63 of every K chunk and
// columns 64 r .. 64 r + 63 of every V chunk (r: its rank), which the tensor cores of both read.  Rank 0's thread issues
// for both; K / V and P barriers that it waits on are its own (rank 1 arrives remotely), the others exist in both CTAs.
// (Neither filling the ring nor the products bound the loop: without either it takes as long.)
template <bool PAIR>
__global__ void __launch_bounds__(NT, 1)
tree_attn_umma_kernel(const Args a, const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV)
{
    constexpr int NS = ring_slots(PAIR);                     // ring slots
    constexpr int SLOT = PAIR ? HALF : TILE;                 // bytes of this CTA's share of a K or V chunk
    constexpr int KROWS = PAIR ? BK / 2 : BK;                // keys of its share of a K chunk
    constexpr int KSUB = KROWS * 128;                        // bytes of one 64-column half of that share
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long s_bar[4 * NS + 16];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    __shared__ __align__(8) short s_par[FSPAD_MAX_NODES_WIDE];      // parents (only where this CTA's keys reach into the tree)

    if (!a.early) fspad_pdl_wait();
    const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
    const bool producer = warp >= 8;         // warp 8 copies, warp 9 drives the tensor cores
    const int row = tid & (BM - 1), grp = (tid >> 7) & 1;
    const int split = PAIR ? blockIdx.y : blockIdx.x, tile_g = PAIR ? blockIdx.x : blockIdx.y;
    const int g = tile_g / a.mtiles, mt = tile_g % a.mtiles;
    const int rank = PAIR ? mt & 1 : 0;           // a.mtiles is even then, so a pair has one kv head
    const int N = a.N, G = a.G, M = a.M;
    const uint32_t bar0 = smem_u32(&s_bar[0]);
    // The thread that issues the first TMA copies also initialises the barriers, so those copies
    // leave as soon as the prefix length is known, ahead of the CTA's first barrier (a pair's: as soon as both CTAs'
    // barriers are initialised).
    if (tid == 256) {
#pragma unroll
        for (int i = 0; i < 4 * NS + 16; ++i) {
            int count = 1;
            if (i >= 4 * NS + 4 && i < 4 * NS + 8) count = PAIR ? 8 : 4;                     // softmax warps of a group
            if (i >= 4 * NS + 14) count = PAIR ? 16 : 8;                         // all of them
            if (i == 4 * NS + 13 && PAIR) count = a.q_tma ? 2 : 1;               // Q, and rank 1's tensor memory
            mbar_init(bar0 + 8u * i, count);
        }
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 8) {
        __syncwarp();
        asm volatile("bar.arrive 2, 320;\n" ::: "memory");                       // (waited for by the other warps in the prologue)
    }
    // Launched while its predecessors still run (see Args::early), the grid must not be complete before they are: one CTA sees to it.
    const bool last_cta = a.early && blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1 && blockIdx.z == gridDim.z - 1;
    int b = blockIdx.z, L;
    if (a.longest_first) {
        // CTAs are dispatched in index order as SMs come free, so with more CTAs than SMs the sequences
        // handled last decide the tail: they should be the short ones.  Every warp ranks the sequences by
        // length (ties by index, so the ranks are a permutation) and takes the one whose rank is blockIdx.z; without a barrier
        // (through shared memory the first wave knew its length after 3800 cycles).
        const int nb = (int)gridDim.z;            // at most 128
        int len[4], place[4] = {0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < 4; ++i) len[i] = lane + 32 * i < nb ? a.prefix_len[lane + 32 * i] : 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll 4
            for (int u = 32 * j; u < min(nb, 32 * j + 32); ++u) {
                const int Lu = __shfl_sync(0xffffffffu, len[j], u & 31);
#pragma unroll
                for (int i = 0; i < 4; ++i) place[i] += (Lu > len[i] || (Lu == len[i] && u < lane + 32 * i)) ? 1 : 0;
            }
        L = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned hit = __ballot_sync(0xffffffffu, lane + 32 * i < nb && place[i] == (int)blockIdx.z);
            const int at = __shfl_sync(0xffffffffu, len[i], hit ? __ffs((int)hit) - 1 : 0);
            if (hit) { b = __ffs((int)hit) - 1 + 32 * i; L = at; }
        }
    } else {
        L = a.prefix_len[b];
    }
    const int par_of = tid < N ? a.parent[(size_t)b * N + tid] : -1;      // (under way with the prefix length)
    if (PAIR) {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    }

    if (L < 0 || L + N > a.max_len) {
        if (tid == 0) fspad_report(a.status, FSPAD_ERR_RANGE);
        L = max(0, min(L, a.max_len - N));
    }
    const int Ltot = L + N;
    const int n_chunks = (Ltot + BK - 1) / BK;
    const int per = (n_chunks + a.n_splits - 1) / a.n_splits;
    const int c0 = split * per, c1 = min(n_chunks, c0 + per);
    const int n_ch = c1 - c0;

    const int gr = mt * BM + row;                 // this thread's row among the kv head's M rows
    const bool row_ok = gr < M && !producer;
    const size_t prow = ((size_t)b * a.Hkv + g) * a.n_splits + split;

    if (n_ch <= 0) {                              // nothing to do for this split: empty partial (never in a pair: one range per row)
        if (row_ok && grp == 0) { float *ml = a.part_ml + (prow * M + gr) * 2; ml[0] = -INFINITY; ml[1] = 0.f; }
        if (a.done != nullptr) {
            __syncthreads();
            if (tid == 0) { __threadfence(); atomicAdd(a.done, 1); fspad_pdl_trigger(); }
        }
        if (last_cta) fspad_pdl_wait();
        return;
    }

    // 1024-byte aligned tiles: Q | K[NS] | V[NS]
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sQ = base, sK = base + TILE, sV = base + TILE + NS * SLOT;
    auto kfull = [&](int buf) { return bar0 + 8u * (uint32_t)buf; };
    auto vfull = [&](int buf) { return bar0 + 8u * (uint32_t)(NS + buf); };
    auto kfree = [&](int buf) { return bar0 + 8u * (uint32_t)(2 * NS + buf); };
    auto vfree = [&](int buf) { return bar0 + 8u * (uint32_t)(3 * NS + buf); };
    auto sfull = [&](int par) { return bar0 + 8u * (uint32_t)(4 * NS + par); };
    auto pfull = [&](int grp2, int par) { return bar0 + 8u * (uint32_t)(4 * NS + 4 + 2 * grp2 + par); };
    auto odone = [&](int grp2, int par) { return bar0 + 8u * (uint32_t)(4 * NS + 8 + 2 * grp2 + par); };
    const uint32_t drain = bar0 + 8u * (uint32_t)(4 * NS + 12);   // used only when a wait has run out
    const uint32_t qfull = bar0 + 8u * (uint32_t)(4 * NS + 13);   // Q by TMA
    const uint32_t gkfull = bar0 + 8u * (uint32_t)(4 * NS + 14), gvfull = gkfull + 8u;   // what the softmax warps gather: Q and K, V
    const bool tma_ok = a.use_tma != 0, q_tma = a.q_tma != 0;
    // arrivals on the barriers of the side that issues
    auto arrive0 = [&](uint32_t bar) { if (PAIR) mbar_arrive_rank0(bar); else mbar_arrive(bar); };
    auto arrive_p = [&](uint32_t bar) { if (PAIR && rank != 0) mbar_arrive_rank0_light(bar); else mbar_arrive_light(bar); };

    const bool paged = a.block_table != nullptr;
    const int *blocks = paged ? a.block_table + (size_t)b * a.table_stride : nullptr;
    const int plane_row0 = (b * a.Hkv + g) * a.max_len;   // contiguous planes: first row of this kv head
    // row of the plane matrix [rows][128] with which chunk `ch` of this sequence and kv head begins (paged: a chunk is one
    // block; an entry out of range is reported and replaced)
    auto chunk_row = [&](int ch) -> int {
        if (!paged) return plane_row0 + ch * BK;
        int blk = __ldg(blocks + ch);
        if (blk < 0 || blk >= a.n_blocks) { fspad_report(a.status, FSPAD_ERR_RANGE); blk = 0; }
        return (blk * a.Hkv + g) * BK;
    };
    const fspad_bf16 *tkb = a.tk ? a.tk + ((size_t)b * a.Hkv + g) * (size_t)N * D : nullptr;
    const fspad_bf16 *tvb = a.tv ? a.tv + ((size_t)b * a.Hkv + g) * (size_t)N * D : nullptr;
    // The chunks are taken from the last one down, so that those TMA cannot describe come early: the ones with rows of an
    // explicit tree array, and the one that ends in zero padding (at most three of them: 256 nodes).  The softmax warps, idle until
    // the first scores are there, gather them side by side with the copies of the others.  (Gathered where they stood, at
    // the end of the range and by the copy warp alone, they held everything up: 2.5 us for each operand.)
    // Before them goes one chunk of the prefix alone, where the range has one and the ring room: a row's reference maximum then comes
    // from whole groups of keys and not from the row's few ancestors.  (With the tree's chunks first either the reference lags behind
    // the prefix's scores, and the largest weight, an exact one otherwise, is rounded: three sequences of 110 keys 2.17e-3 off 64 bits against
    // 2.09e-3; or it follows, with a pass over O behind the product: us, pass / this: 16 sequences of 1 K keys, the attention alone 40.2 / 38.8, 32 heads
    // and 570 keys 14.0 / 13.8, 32 heads and 1.5 K 18.2 / 17.8; the other way round 52 heads and 4 K in a step 38.6 / 39.0.)
    const int n_mask = max(0, c1 - max(c0, L / BK));                  // chunks of the range that reach past the prefix
    const bool lead = n_mask > 0 && n_mask < n_ch && n_mask < ring_slots(false);       // (the same on pairs, and with it the bits)
    auto chunk_at = [&](int c) { return c1 - 1 - (!lead || c > n_mask ? c : c == 0 ? n_mask : c - 1); };      // c-th chunk to be taken
    const int key_tma = tkb ? L : Ltot;           // rows in front of this key lie in the cache
    auto is_tma = [&](int ch) { return tma_ok && (ch + 1) * BK <= key_tma; };
    const int g0 = lead && tma_ok ? 1 : 0;        // chunks g0 .. g0 + n_gather - 1 of the first ring filling are gathered
    int n_gather = 0;
    while (g0 + n_gather < NS && g0 + n_gather < n_ch && !is_tma(chunk_at(g0 + n_gather))) ++n_gather;

    // Gather chunk `ch` into ring slot `buf` with 16-byte asynchronous copies by threads t0, t0 + nt, ... (nt a multiple of 16):
    // 16-byte piece c of every row that falls to a thread is the same, so all its addresses follow from one.
    auto gather = [&](int ch, int buf, bool is_v, int t0, int nt) {
        const uint32_t dst = (is_v ? sV : sK) + buf * SLOT;
        const fspad_bf16 *tb = is_v ? tvb : tkb;
        const fspad_bf16 *cb = (is_v ? a.vc : a.kc) + (size_t)chunk_row(ch) * D;
        const int sh = PAIR && is_v ? 3 : 4;      // a pair's V share: half the columns; its K share: half the keys
        const int cl = t0 & ((1 << sh) - 1), c = PAIR && is_v ? cl + 8 * rank : cl;
        const int k_lo = PAIR && !is_v ? KROWS * rank : 0;
        const uint32_t half = (uint32_t)(cl >> 3) * (PAIR ? KSUB : HALF);
#pragma unroll 4
        for (int r = t0 >> sh; r < (PAIR && !is_v ? KROWS : BK); r += nt >> sh) {
            const int kr = r + k_lo, key = ch * BK + kr;
            const bool ok = key < Ltot;
            // prefix rows, and tree rows that live in the cache, come from the planes; explicit tree rows from their array
            const fspad_bf16 *src = cb;
            if (ok) src = (key < L || tb == nullptr) ? cb + (size_t)kr * D : tb + (size_t)(key - L) * D;
            cp_async16(dst + half + (uint32_t)(r * 128 + (((cl & 7) ^ (r & 7)) << 4)), src + c * 8, ok);
        }
    };
    // One lane: the TMA copies of a chunk that begins with row y of the planes.  A pair's bytes are all expected by rank 0, whose
    // barrier counts them (an arrival there by rank 1 took it 400 cycles); rank 1's may land before they are expected,
    // never before the phase they belong to, because a slot is only refilled when rank 0 has waited for what it held.
    auto tma_fill = [&](int y, int buf, bool is_v) {
        const uint32_t dst = (is_v ? sV : sK) + buf * SLOT;
        const uint32_t bar = is_v ? vfull(buf) : kfull(buf);
        const CUtensorMap *map = is_v ? &tmV : &tmK;
        if constexpr (PAIR) {
            if (rank == 0) mbar_expect_tx(bar, 2 * SLOT);
            if (is_v) {
                tma_load_2d_pair(dst, map, 64 * rank, y, bar);                    // 128 keys x 64 columns
            } else {
                tma_load_2d_pair(dst, map, 0, y + KROWS * rank, bar);             // 64 keys x 64 columns, twice
                tma_load_2d_pair(dst + KSUB, map, 64, y + KROWS * rank, bar);
            }
        } else {
            mbar_expect_tx(bar, TILE);
            tma_load_2d(dst, map, 0, y, bar);
            tma_load_2d(dst + HALF, map, 64, y, bar);
        }
    };

    // ---- prologue: the tensor memory, then every warp goes its own way; what each needs from the others comes by mbarrier ----
    if (warp == 9) {
        __syncwarp();
        if constexpr (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n"
                         :: "r"(smem_u32(&s_tmem)), "r"(TMEM_COLS) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                         :: "r"(smem_u32(&s_tmem)), "r"(TMEM_COLS) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
        }
    }
    auto peer_ready = [&]() {                     // both CTAs' barriers are initialised
        if (PAIR) {
            __syncwarp();
            asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
        }
    };
    const bool in_tree = c1 * BK > L;             // this range's keys reach into the tree
    int blk_row = 0;                              // copy warp: first plane row of the (32 i + lane)-th chunk to be taken
    auto first_fills = [&](int u0, int u1) {      // copy warp: ring slots u0 .. u1 - 1, for the first time
        for (int u = u0; u < u1 && u < n_ch; ++u) {
            const int y = __shfl_sync(0xffffffffu, blk_row, u);
            if (lane == 0) {
                if (u < g0 || u >= g0 + n_gather) { tma_fill(y, u, false); tma_fill(y, u, true); }
                else if (rank == 0) { mbar_arrive(kfull(u)); mbar_arrive(vfull(u)); }       // (gkfull and gvfull tell when they are there)
            }
            __syncwarp();
        }
    };
    // The rings of all SMs are 24 to 28 MB, 4 us of HBM, and what is asked for together arrives together: the first scores would wait
    // for all of it.  So the rest of the ring is asked for when the first scores are there.
    constexpr int kFirst = PAIR ? 3 : 2;
    if (warp == 8) {
        if (lane < n_ch) blk_row = chunk_row(chunk_at(lane));
        peer_ready();
        if (lane == 0 && q_tma) {
            const int nd = b * N + mt * (BM / G);
            if constexpr (PAIR) {
                if (rank == 0) mbar_expect_tx(qfull, 2 * TILE);
                tma_load_3d_pair(sQ, &tmQ, 0, g * G, nd, qfull);
                tma_load_3d_pair(sQ + HALF, &tmQ, 64, g * G, nd, qfull);
            } else {
                mbar_expect_tx(qfull, TILE);
                tma_load_3d(sQ, &tmQ, 0, g * G, nd, qfull);
                tma_load_3d(sQ + HALF, &tmQ, 64, g * G, nd, qfull);
            }
        }
        first_fills(0, kFirst);
    } else if (warp < 8) {
        // What TMA cannot describe: Q where a group of query heads does not divide the tile, and n_gather of the first chunks.
        if (!q_tma) {
            const int c = tid & 15;
            int r = tid >> 4;                     // 16 rows a step
            int nd = (mt * BM + r) / G, hh = (mt * BM + r) % G;
            const int dn = 16 / G, dh = 16 % G;
            for (; r < BM; r += 16) {
                const bool ok = mt * BM + r < M;
                const fspad_bf16 *src = a.q + (ok ? (((size_t)b * N + nd) * a.Hq + g * G + hh) * D + c * 8 : 0);
                cp_async16(sQ + tile_off(r, c), src, ok);
                nd += dn; hh += dh;
                if (hh >= G) { hh -= G; ++nd; }
            }
        }
        for (int u = g0; u < g0 + n_gather; ++u) gather(chunk_at(u), u, false, tid, 256);
        cp_async_commit();
        for (int u = g0; u < g0 + n_gather; ++u) gather(chunk_at(u), u, true, tid, 256);
        cp_async_commit();
        peer_ready();
    } else {
        peer_ready();
    }
    if (PAIR && warp == 9 && lane == 0 && rank != 0) arrive0(qfull);             // rank 1's tensor memory is there
    if (in_tree && tid < N) s_par[tid] = par_of < -1 ? (short)-2 : (short)min(par_of, 32767);
    // barriers initialised, tensor memory there, parents staged: the copy warp, which has use for none of it, has arrived with
    // the barriers' initialisation (with it here, the nine other warps waited 2000 cycles for its copies to be issued)
    if (warp != 8) {
        tc_fence_before();
        asm volatile("bar.sync 2, 320;\n" ::: "memory");
        tc_fence_after();
    }
    const uint32_t tmem = warp != 8 ? s_tmem : 0u;
    const uint32_t idesc_s = PAIR ? make_idesc_m256(128) : make_idesc(false, 128);
    const uint32_t idesc_o = PAIR ? make_idesc_m256(128) | (1u << 16) : make_idesc(true, 128);      // B (= V) MN-major
    const uint32_t tO = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 256u + (uint32_t)grp * 128u;   // this group's O row
    bool failed = false;
    int filled_k = min(n_ch, NS), filled_v = filled_k;   // copy warp: chunks whose K (V) fill has been started

    if (warp == 8) {
        // ================= copy warp: fills and refills the K / V buffers =================
        if (n_ch > kFirst && !mbar_wait(kfree(0), 0u)) failed = true;
        if (!failed) first_fills(kFirst, NS);
        auto fill = [&](int c, int y, int buf, bool is_v) {
            if (is_tma(chunk_at(c))) {
                if (lane == 0) tma_fill(y, buf, is_v);
            } else {
                gather(chunk_at(c), buf, is_v, lane, 32);
                cp_async_commit();
                cp_async_wait<0>();
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(is_v ? vfull(buf) : kfull(buf));      // (a lone CTA: pairs have their maps)
            }
            __syncwarp();
        };
        int buf = 0;                             // i modulo NS
        uint32_t ph = 0;                         // flips each time the ring wraps
        for (int i = 0; i + NS < n_ch; ++i) {
            const int c = i + NS;
            if ((c & 31) == 0 && c + lane < n_ch) blk_row = chunk_row(chunk_at(c + lane));
            const int y = __shfl_sync(0xffffffffu, blk_row, c & 31);
            // the K buffer of chunk i is free once S(i) has completed, its V buffer once O += P(i) V(i) has
            if (!failed && !mbar_wait(kfree(buf), ph)) failed = true;
            if (!failed) { fill(c, y, buf, false); ++filled_k; }
            if (!failed && !mbar_wait(vfree(buf), ph)) failed = true;
            if (!failed) { fill(c, y, buf, true); ++filled_v; }
            if (++buf == NS) { buf = 0; ph ^= 1u; }
        }
        if (failed) s_fail = 1;
    } else if (warp == 9) {
        // ================= tensor-core warp: the whole warp runs the loop, one lane issues every tcgen05.mma =================
        // (one lane's branch kept every operand in ordinary registers: 17.4 against 19.0 us per call at 4 heads per KV head
        // and 2 K keys, 35.8 against 37.8 at 8 and 8 K, 99.3 against 101.4 on the ragged batch of 16)
        if (rank == 0) {
            const bool issuer = elect_one();
            auto commit = [&](uint32_t bar) { if (PAIR) mma_commit_pair(bar); else mma_commit(bar); };
            // low words of the shared-memory descriptors (start address and leading byte offset);
            // the high word (8-row group stride, version, swizzle mode) is the same for all
            const uint32_t hi = (uint32_t)(make_desc(0, 16) >> 32);
            const uint32_t q_lo = (uint32_t)make_desc(sQ, 16), k_lo = (uint32_t)make_desc(sK, 16);
            const uint32_t v_lo = (uint32_t)make_desc(sV, HALF);
            int kbuf = 0, vbuf = 0;              // ring slots of the next chunk to score / to multiply by V
            uint32_t kph = 0, vph = 0;           // and their phases (flip each time the ring wraps)
            // S(c) = Q K(c)^T into score buffer c & 1 (columns 0..63 of it belong to group 0, 64..127 to
            // group 1); K(c) sits in ring slot kbuf, which the second commit releases
            auto issue_s = [&](int c) {
                if (!failed && !mbar_wait(kfull(kbuf), kph)) failed = true;
                if (!failed && issuer) {
                    // no tcgen05 fence here: the K chunk comes through the barrier's own acquire, and the
                    // score buffer's last readers and writers (softmax of chunk c - 2) were ordered before this
                    // thread's instructions by the fence behind its pfull wait of that chunk
                    const uint32_t kb = k_lo + (uint32_t)kbuf * (SLOT >> 4);
                    const uint32_t d = tmem + (uint32_t)(c & 1) * 128u;
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) { // K = 16 per instruction over d = 128
                        const uint32_t qoff = ((ks >> 2) * HALF + (ks & 3) * 32) >> 4, koff = ((ks >> 2) * KSUB + (ks & 3) * 32) >> 4;
                        if constexpr (PAIR) mma_f16_pair(d, q_lo + qoff, kb + koff, hi, idesc_s, ks > 0);
                        else mma_f16_ss(d, q_lo + qoff, kb + koff, hi, idesc_s, ks > 0);
                    }
                    commit(sfull(c & 1));
                    commit(kfree(kbuf));
                }
                __syncwarp();
                if (++kbuf == NS) { kbuf = 0; kph ^= 1u; }
            };
            if ((PAIR || q_tma) && !mbar_wait(qfull, 0u)) failed = true;
            if (((n_gather > 0 && g0 == 0) || !q_tma) && !failed && !mbar_wait(gkfull, 0u)) failed = true;
            issue_s(0);
            if (n_gather > 0 && !failed && !mbar_wait(gkfull, 0u)) failed = true;
            if (n_ch > 1) issue_s(1);
            for (int c = 0; c < n_ch; ++c) {
                const int p = c & 1;
                const uint32_t ph = (uint32_t)(c >> 1) & 1u;
                const uint32_t vb = v_lo + (uint32_t)vbuf * (SLOT >> 4);
                if (n_gather > 0 && c == g0 && !failed && !mbar_wait(gvfull, 0u)) failed = true;
#pragma unroll
                for (int g2 = 0; g2 < 2; ++g2) {
                    // O[g2] += P_g2(c) V(c)[64 g2 .. 64 g2 + 63]: P from the four warps of group g2 (in tensor
                    // memory, over the scores it was computed from) and the V chunk
                    if (!failed && !mbar_wait(pfull(g2, p), ph)) failed = true;
                    if (g2 == 0 && !failed && !mbar_wait(vfull(vbuf), vph)) failed = true;
                    if (!failed && issuer) {
                        tc_fence_after();
                        const uint32_t a_t = tmem + (uint32_t)p * 128u + (uint32_t)g2 * 64u;
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) { // K = 16 keys per instruction = 8 columns of packed bf16 pairs
                            // V as an MN-major operand: d is contiguous, the two 64-wide halves are HALF bytes apart
                            // (a pair's CTA holds one of those halves)
                            const uint32_t od = tmem + 256u + (uint32_t)g2 * 128u, at = a_t + (uint32_t)ks * 8u;
                            const uint32_t vk = vb + (uint32_t)((g2 * 64 + ks * 16) * 128 >> 4);
                            if constexpr (PAIR) mma_f16_ts_pair(od, at, vk, hi, idesc_o, (c > 0) || (ks > 0));
                            else mma_f16_ts(od, at, vk, hi, idesc_o, (c > 0) || (ks > 0));
                        }
                        commit(odone(g2, p));
                        if (g2 == 1) commit(vfree(vbuf));
                    }
                    __syncwarp();
                }
                // tensor-core work completes in issue order, so the scores of chunk c + 2 may replace P(c)
                if (c + 2 < n_ch) issue_s(c + 2);
                if (++vbuf == NS) { vbuf = 0; vph ^= 1u; }
            }
            if (failed) s_fail = 1;
        }
        __syncwarp();
    } else {
        // ================= softmax warps =================
        const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
        if (n_gather > 0 || !q_tma) {
            cp_async_wait<1>();
            fence_async_smem();
            __syncwarp();
            if (lane == 0) arrive0(gkfull);
            cp_async_wait<0>();
            fence_async_smem();
            __syncwarp();
            if (lane == 0) arrive0(gvfull);
        }
        const float scale = a.scale_log2;
        const bool live = mt * BM + (warp & 3) * 32 < M;   // the last row tile may end before this warp's rows
        float m_run = -INFINITY, l_run = 0.f;
        int cur = in_tree && row_ok ? gr / G : -1;         // this row's node, then its ancestors: how far the chunks so far have taken them

        for (int c = 0; c < n_ch; ++c) {
            const int ch = chunk_at(c), p = c & 1;
            const uint32_t tS = tmem + lanes + (uint32_t)p * 128u + (uint32_t)grp * 64u;   // scores, then P
            const bool masked = (ch + 1) * BK > L;   // only chunks that reach past the cached prefix
            // Validity of this group's 64 keys for this row: prefix keys are valid, tree key L + t is valid iff t is the row's node
            // or one of its ancestors (which also rules out the zero padding).  Parents come before their children and the
            // tree's chunks from the last one down, so every chunk takes the walk to the root on from where the one before it left off;
            // no mask is kept, whatever the tree's size.
            unsigned long long valid = ~0ull;
            if (masked) {
                const int t0 = ch * BK + grp * 64 - L, t_chunk = ch * BK - L;        // tree index of the group's, the chunk's first key
                valid = t0 >= 0 ? 0ull : t0 <= -64 ? ~0ull : (1ull << -t0) - 1ull;
                while (cur >= 0 && cur >= t_chunk) {
                    const unsigned o = (unsigned)(cur - t0);
                    if (o < 64u) valid |= 1ull << o;
                    const int p = s_par[cur];
                    if (cur == 0 ? p != -1 : (p < 0 || p >= cur)) fspad_report(a.status, FSPAD_ERR_BAD_TREE);
                    cur = p < cur ? p : -1;
                }
            }
            if (!failed && !mbar_wait(sfull(p), (uint32_t)(c >> 1) & 1u)) failed = true;
            if (!live) {
                // (no row of this warp exists: its scores are not looked at, and what its lanes' P holds stays in their
                // own rows of O, which nobody stores)
                __syncwarp();
                if (lane == 0) arrive_p(pfull(grp, p));
                continue;
            }
            tc_fence_after();
            // ---- this row's 64 scores of the group, in registers after one trip to tensor memory, with the
            // tree mask applied where it matters; the row maximum as four independent chains ----
            float v[64];
            {
                uint32_t r0[32], r1[32];
                __syncwarp();
                tmem_ld32_issue(tS, r0);
                tmem_ld32_issue(tS + 32u, r1);
                tmem_ld_wait(r0);
                tmem_ld_pin(r1);
#pragma unroll
                for (int j = 0; j < 32; ++j) { v[j] = __uint_as_float(r0[j]); v[32 + j] = __uint_as_float(r1[j]); }
            }
            if (masked) {
#pragma unroll
                for (int j = 0; j < 64; ++j)
                    if (!(((uint32_t)(valid >> (j & 32)) >> (j & 31)) & 1u)) v[j] = -INFINITY;
            }
            float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int j = 0; j < 64; ++j) mx4[j & 3] = fmaxf(mx4[j & 3], v[j]);
            const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
            // The reference value m of a row (P = exp2(s * scale - m), O and the sum are relative to it)
            // only has to bound the scores loosely: it follows the row maximum when some row of the warp
            // would otherwise see a P above 2^kLazyLog2, and stays put - no pass over O - when not.
            // (The decision is taken per warp because the tensor-memory accesses are warp-collective;
            // a comparison with -inf - -inf = NaN is false and so counts as a move.  Lanes whose row does not exist have no say: by
            // TMA they hold the next sequence's queries, and what that one asks must not decide how this one's P is rounded.)
            // Where the tree's chunks do come first (no chunk of the prefix alone, or three of the tree's), the reference follows every larger
            // score up to the first chunk behind them.
            const float m_cand = fmaxf(m_run, mx * scale), lag = !lead && (ch + 2) * BK > L ? 0.f : kLazyLog2;
            const bool move = !__all_sync(0xffffffffu, !row_ok || m_cand - m_run <= lag);
            const float m_new = move ? m_cand : m_run;
            const float m_safe = (m_new == -INFINITY) ? 0.f : m_new;
            const float alpha = move ? ex2f(m_run - m_safe) : 1.f;
            // ---- rescale this row of O[grp], once the group's product of the previous chunk is complete ----
            if (c >= 1 && move) {
                if (!failed && !mbar_wait(odone(grp, (c - 1) & 1), (uint32_t)((c - 1) >> 1) & 1u)) failed = true;
                tc_fence_after();
#pragma unroll
                for (int blk = 0; blk < 4; ++blk) {
                    float o[32];
                    tmem_ld32(tO + (uint32_t)blk * 32u, o);
#pragma unroll
                    for (int j = 0; j < 32; ++j) o[j] *= alpha;
                    tmem_st32(tO + (uint32_t)blk * 32u, o);
                }
            }
            // ---- P = exp2(s * scale - m) as bf16 pairs, written over the group's score columns (every score
            // is in registers by now); the row sum as four pairs of chains; multiply-adds and sums two to an instruction
            // (33.6 against 34.1 us on 52 heads and 4 K keys, 75.9 against 77.2 on the ragged batch; taking the exponentials
            // against the old reference while the maximum is being found cost registers: 2 us more on every shape; asking for
            // half of the next chunk's scores between the two halves of this one's exponentials: 112 against 96 us on 16
            // sequences of 4 K keys) ----
            float rs;
            {
                const uint64_t scale2 = f32x2(scale, scale), neg = f32x2(-m_safe, -m_safe);
                uint64_t acc[4];
#pragma unroll
                for (int blk = 0; blk < 2; ++blk) {
                    uint32_t w[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        float x0, x1;
                        f32x2_split(f32x2_fma(f32x2(v[blk * 32 + 2 * e], v[blk * 32 + 2 * e + 1]), scale2, neg), x0, x1);
                        const float p0 = ex2f(x0), p1 = ex2f(x1);
                        const uint64_t pp = f32x2(p0, p1);
                        acc[e & 3] = blk == 0 && e < 4 ? pp : f32x2_add(acc[e & 3], pp);
                        w[e] = pack_bf16(p0, p1);
                    }
                    tmem_st16(tS + (uint32_t)blk * 16u, w);
                }
                float lo, hi;
                f32x2_split(f32x2_add(f32x2_add(acc[0], acc[1]), f32x2_add(acc[2], acc[3])), lo, hi);
                rs = lo + hi;
            }
            l_run = l_run * alpha + rs;
            m_run = m_new;
            asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_p(pfull(grp, p));
        }
        // ---- each group waits for its own last product (tensor-core work completes in order, so the
        // one before it is complete too); the CTA-wide barrier below then orders both accumulators
        // before the merge ----
        if (!failed && !mbar_wait(odone(grp, (n_ch - 1) & 1), (uint32_t)((n_ch - 1) >> 1) & 1u)) failed = true;
        tc_fence_after();
        if (failed) s_fail = 1;
        // the Q tile is dead (every S was issued before that product and completes before it): it
        // carries the groups' (max, sum) exchange
        float2 *s_ml = reinterpret_cast<float2 *>(smem_raw + (base - smem_u32(smem_raw)));
        s_ml[grp * BM + row] = make_float2(m_run, l_run);
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        // ---- publish the row: the two groups' (max, sum, O row) merged by log-sum-exp ----
        // Thread (row, grp) owns output columns grp*64 .. grp*64+63.  Every lane of every softmax warp
        // takes part in the tensor-memory loads (they are warp-collective); only the stores to global
        // memory depend on whether the row exists.
        const bool any_fail = s_fail != 0;
        if (any_fail && tid == 0) fspad_report(a.status, FSPAD_ERR_TIMEOUT);
        const float2 ml0 = s_ml[row], ml1 = s_ml[BM + row];
        const float m_all = fmaxf(ml0.x, ml1.x);
        const float m_fin = (m_all == -INFINITY) ? 0.f : m_all;
        float f0 = ex2f(ml0.x - m_fin), f1 = ex2f(ml1.x - m_fin);           // exp2(-inf) = 0 for a fully masked half
        const float l_all = ml0.y * f0 + ml1.y * f1;
        const bool final = a.out != nullptr;
        if (final) {
            const float inv = l_all > 0.f ? 1.f / l_all : 0.f;
            f0 *= inv;
            f1 *= inv;
        }
        // The merged rows are staged in shared memory (the K ring is idle by now), so that they leave as whole rows, 16 bytes a
        // lane.  (Stores straight from the registers are row-strided pieces, each a transaction of its own: 3 us per CTA; a bulk
        // copy per row: 1.1 us until the last of the 128 has been read; rows one after another with their addresses: 1.2 us.)
        constexpr int FROW = D * 4 + 16, HROW = D * 2 + 16;      // bytes of a staged row; the pad keeps 16-byte stores conflict-free
        const uint32_t stage = base + TILE, stg = stage + (uint32_t)(row * (final ? HROW : FROW));
        int *s_row = reinterpret_cast<int *>(s_par);             // where each row goes (-1: nowhere); nobody looks at the parents any more
        static_assert(sizeof(s_par) >= BM * sizeof(int), "one place per row");
        if (grp == 0) s_row[row] = !row_ok || any_fail ? -1 : final ? (b * N + gr / G) * a.Hq + g * G + gr % G : gr;
        const uint32_t tO0 = tmem + lanes + 256u + (uint32_t)grp * 64u, tO1 = tO0 + 128u;
#pragma unroll
        for (int q2 = 0; q2 < 2; ++q2) {
            uint32_t o[32], o1[32];
            __syncwarp();
            tmem_ld32_issue(tO0 + q2 * 32, o);
            tmem_ld32_issue(tO1 + q2 * 32, o1);
            tmem_ld_wait(o);
            tmem_ld_pin(o1);
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = __float_as_uint(fmaf(__uint_as_float(o1[j]), f1, __uint_as_float(o[j]) * f0));
            if (final) {
#pragma unroll
                for (int j = 0; j < 32; j += 8)
                    st_shared16(stg + (uint32_t)(grp * 128 + q2 * 64 + j * 2),
                                pack_bf16(__uint_as_float(o[j]), __uint_as_float(o[j + 1])), pack_bf16(__uint_as_float(o[j + 2]), __uint_as_float(o[j + 3])),
                                pack_bf16(__uint_as_float(o[j + 4]), __uint_as_float(o[j + 5])), pack_bf16(__uint_as_float(o[j + 6]), __uint_as_float(o[j + 7])));
            } else {
#pragma unroll
                for (int j = 0; j < 32; j += 4) st_shared16(stg + (uint32_t)(grp * 256 + q2 * 128 + j * 4), o[j], o[j + 1], o[j + 2], o[j + 3]);
            }
        }
        if (!final && row_ok && grp == 0 && !any_fail) {
            float *ml = a.part_ml + (prow * M + gr) * 2;
            ml[0] = m_all;
            ml[1] = l_all;
        }
        asm volatile("bar.sync 1, 256;\n" ::: "memory");   // the eight softmax warps
        if (final) {
#pragma unroll
            for (int i = 0; i < BM / 16; ++i) {                  // a warp takes 16 rows, two at a time
                const int r = warp * 16 + 2 * i + (lane >> 4), to = s_row[r];
                if (to >= 0) reinterpret_cast<uint4 *>(a.out + (size_t)to * D)[lane & 15] = ld_shared16(stage + (uint32_t)(r * HROW + (lane & 15) * 16));
            }
        } else {
#pragma unroll
            for (int i = 0; i < BM / 8; ++i) {
                const int r = warp * 16 + i, to = s_row[r];
                if (to >= 0) reinterpret_cast<uint4 *>(a.part_o + (prow * M + to) * D)[lane] = ld_shared16(stage + (uint32_t)(r * FROW + lane * 16));
            }
        }
        // partial written: the merge kernel may start launching, and where it does not wait for this kernel's end, not before the
        // count says that the partial is there (behind the barrier the fence stands for all eight warps' stores)
        if (a.done != nullptr) {
            asm volatile("bar.sync 1, 256;\n" ::: "memory");
            if (tid == 0) { __threadfence(); atomicAdd(a.done, 1); fspad_pdl_trigger(); }
        } else {
            fspad_pdl_trigger();
        }
        tc_fence_before();
        __syncthreads();
        if (PAIR) cluster_sync_all();             // neither CTA leaves while the other may still reach it
        if (last_cta) fspad_pdl_wait();
        return;
    }
    // copy and tensor-core warps: meet the softmax warps at their two CTA-wide barriers; the warp
    // that allocated the tensor memory then frees it
    tc_fence_before();
    __syncthreads();
    if (s_fail != 0) {
        // A wait ran out somewhere in this CTA.  Before the shared and tensor memory go back to
        // the SM, whatever was started asynchronously is given a bounded time to land: the copy warp
        // waits for the last fill it started in every ring slot, the tensor-core warp for everything
        // its thread has issued (one more commit on a barrier of its own).
        if (warp == 8) {
            if ((PAIR || q_tma) && rank == 0) (void)mbar_wait(qfull, 0u);
            for (int sl = 0; sl < NS && rank == 0; ++sl) {    // (a pair's fills are all counted by rank 0's barriers)
                const int nk = (filled_k - sl + NS - 1) / NS, nv = (filled_v - sl + NS - 1) / NS;   // fills of slot sl
                if (nk > 0) (void)mbar_wait(kfull(sl), (uint32_t)(nk - 1) & 1u);
                if (nv > 0) (void)mbar_wait(vfull(sl), (uint32_t)(nv - 1) & 1u);
            }
        } else if (rank == 0) {
            if constexpr (PAIR) { if (lane == 0) mma_commit_pair(drain); }
            else { if (lane == 0) mma_commit(drain); }
            (void)mbar_wait(drain, 0u);
        }
    }
    __syncthreads();
    if (PAIR) cluster_sync_all();
    if (warp != 9) return;
    tc_fence_after();
    __syncwarp();
    if constexpr (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(TMEM_COLS) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(TMEM_COLS) : "memory");
}

// Self-test of the bounded wait: one warp waits, with a small cap, on a barrier that nothing ever
// arrives on; the wait must run out, the kernel records FSPAD_ERR_TIMEOUT and returns normally.
__global__ void __launch_bounds__(32)
wait_timeout_selftest_kernel(int *status, uint32_t cap)
{
    __shared__ __align__(8) unsigned long long bar;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncwarp();
    const bool ok = mbar_wait(smem_u32(&bar), 0u, cap);
    if (!ok && threadIdx.x == 0) fspad_report(status, FSPAD_ERR_TIMEOUT);
}

}  // namespace umma

cudaError_t fspad_launch_wait_selftest(fspad_ctx *ctx, int polls, cudaStream_t st)
{
    ctx->launches++;
    return fspad_launch_opt(false, umma::wait_timeout_selftest_kernel, dim3(1), dim3(32), 0, st, 0, ctx->d_status,
                            (uint32_t)polls);
}

// Key ranges per row: one CTA per SM, never a partial second wave; and one where the call's sequences are so short that walking all of their
// chunks takes no longer than the merge of the ranges (2.5 us and a launch, a chunk 1.05).  A greedy step of 26 nodes and 32 heads, us with
// ranges and without: 3 chunks 14.4 and 12.8, 4 chunks 14.3 and 12.6, 5 chunks 14.6 and 14.1, 6 chunks 15.5 and 15.2, 8 chunks 15.6 and 17.0.
// A wide tree on few CTAs is cut all the same: its up to three gathered chunks are a third of the loop and would all be one CTA's (8 heads on 2,
// 250 nodes and 380 keys, the attention alone: 14.6 us in ranges, 18.7 in one; 32 heads on 8, 64 CTAs: 20.7 and 18.7).
// So is a call of the attention alone on few CTAs at five chunks: without a step around it, whose order goes by the ranges, the merge costs less
// than the fifth chunk (us from a graph, ranges and one: 8 heads on one 11.9 and 12.9, 4 heads of 26 nodes 12.1 and 13.5, 32 on 8 13.1 and 13.4; with 32
// CTAs, 64 heads on 8, 13.4 and 13.1).
// chunks: how many a sequence may have, by the context's max_len or by the block table of a paged call.  The scratch is sized for
// as many ranges as the context's own sequences have chunks.
constexpr int kOneRange = 5;
int fspad_attn_ranges(const fspad_ctx *ctx, int N, int B, int sms, int chunks, bool alone)
{
    if (sms <= 0 || sms > ctx->sm_count) sms = ctx->sm_count;
    const long long base = (long long)B * ctx->cfg.n_kv_heads * fspad_attn_mtiles(ctx, N, B, sms);
    long long s = sms / base;
    const int held = (ctx->cfg.max_len + umma::BK - 1) / umma::BK;
    const bool few = (N > FSPAD_MAX_NODES && base * 4 < sms) || (alone && chunks == kOneRange && base * 8 < sms);
    if (chunks <= kOneRange && !few) return 1;
    if (s > chunks) s = chunks;
    if (s > held) s = held;
    if (s > 64) s = 64;
    if (s < 1) s = 1;
    return (int)s;
}

// Row tiles of a kv head.  In a step's attention, which shares the SMs with the scan and the walk, tiles that fill the SMs by
// themselves (a batch: one key range per row, long loops) go in pairs where there are two or more, the last pair possibly with an empty half.
// us a step, pairs against lone CTAs, called one by one / from a graph: 16 ragged sequences 193 / 189 against 186 / 198, five of 4 K
// keys 139 / 105 against 144 / 110, twelve of 100 to 400 130 / 128 against 130 / 133; nine at 32000 tokens 86 / 86 against 80 / 80.
// A call that has the SMs for itself (FspadPaged::alone) takes lone CTAs: of 160 shapes (33 to 250 nodes, 1 to 8 heads a group, 5 to 16
// sequences, 150 to 4096 keys) they were slower at a few of nine sequences or more and 4 K keys, by up to 3 %, and faster at all others:
// 58.5 -> 42.9 us on eight sequences of 4 K (whose chunks take pairs in step with one another 1.4 us, lone CTAs 1.0), 69 -> 62 on 16
// ragged ones, 41.4 -> 30.9 on four of 130 nodes.
// Where the keys are split as well, the loops are short and the pair's hand-shakes cost more than
// it saves: 23.6 against 19.5 us with two chunks a CTA, 40 against 38 us with 17.
bool fspad_attn_pairs(const fspad_ctx *ctx, int N, int B, int sms)
{
    if (sms <= 0 || sms > ctx->sm_count) sms = ctx->sm_count;
    const int mtiles = (N * (ctx->cfg.n_q_heads / ctx->cfg.n_kv_heads) + umma::BM - 1) / umma::BM;
    return mtiles > 1 && 2ll * B * ctx->cfg.n_kv_heads * mtiles > sms;          // (no room for two ranges)
}
int fspad_attn_mtiles(const fspad_ctx *ctx, int N, int B, int sms)
{
    const int mtiles = (N * (ctx->cfg.n_q_heads / ctx->cfg.n_kv_heads) + umma::BM - 1) / umma::BM;
    return fspad_attn_pairs(ctx, N, B, sms) ? (mtiles + 1) & ~1 : mtiles;
}

int fspad_attn_umma_splits(const fspad_ctx *ctx, int N, int B, int sms)
{
    return fspad_attn_ranges(ctx, N, B, sms, (ctx->cfg.max_len + umma::BK - 1) / umma::BK, false);
}

// ---- TMA descriptors of the K and V cache planes ----------------------------------------
// Each plane is viewed as one row-major matrix [batch * Hkv * max_len][128] bf16; a box is
// 64 columns (128 bytes, the swizzle span) by 128 rows and lands as one half tile.
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        (void)cudaGetLastError();
    }
    return fn;
}

bool fspad_make_tmap_bf16_2d(CUtensorMap *map, const fspad_bf16 *base, size_t cols, size_t rows, unsigned box_rows,
                             bool wide_l2_fetch)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn || rows == 0 || rows > 0x7fffffffull || cols == 0 || (cols * sizeof(fspad_bf16)) % 16 != 0) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * sizeof(fspad_bf16)};
    const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<fspad_bf16 *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              wide_l2_fetch ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The query rows [nodes of all sequences][Hq][128] as boxes of 64 columns, the G heads of a kv head and the 128 / G nodes of a
// row tile, which land as one half tile in the rows' order (G divides 128; nodes past a sequence's last one belong to rows that
// nobody looks at).
static bool make_q_map(CUtensorMap *map, const fspad_bf16 *q, size_t nodes, int Hq, int G)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn || umma::BM % G != 0 || nodes > 0x7fffffffull) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)umma::D, (cuuint64_t)Hq, (cuuint64_t)nodes};
    const cuuint64_t strides[2] = {umma::D * sizeof(fspad_bf16), (cuuint64_t)Hq * umma::D * sizeof(fspad_bf16)};
    const cuuint32_t box[3] = {64u, (cuuint32_t)G, (cuuint32_t)(umma::BM / G)};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<fspad_bf16 *>(q), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static bool make_plane_map(CUtensorMap *map, const fspad_bf16 *plane, size_t rows)
{
    return fspad_make_tmap_bf16_2d(map, plane, (size_t)umma::D, rows, (unsigned)umma::BK);
}

cudaError_t fspad_launch_attn_umma_split(fspad_ctx *ctx, const fspad_bf16 *q, const fspad_bf16 *kc,
                                         const fspad_bf16 *vc, const fspad_bf16 *tk, const fspad_bf16 *tv,
                                         const int *parent, const int *prefix_len, int N, int B, int sms, int n_splits,
                                         float scale_log2, fspad_bf16 *out, cudaStream_t st, FspadPaged paged)
{
    const fspad_config &c = ctx->cfg;
    umma::Args a;
    a.q = q; a.kc = kc; a.vc = vc; a.tk = tk; a.tv = tv; a.parent = parent; a.prefix_len = prefix_len;
    a.N = N; a.Hq = c.n_q_heads; a.Hkv = c.n_kv_heads; a.G = c.n_q_heads / c.n_kv_heads;
    a.M = N * a.G; a.max_len = paged.table ? paged.stride * umma::BK : c.max_len; a.n_splits = n_splits;
    a.block_table = paged.table; a.table_stride = paged.stride; a.n_blocks = paged.n_blocks;
    const bool in_pairs = !paged.alone && fspad_attn_pairs(ctx, N, B, sms);
    a.mtiles = in_pairs ? fspad_attn_mtiles(ctx, N, B, sms) : (a.M + umma::BM - 1) / umma::BM;
    // (every warp ranks all sequences itself, up to four loads a lane and a shuffle a sequence: kept to batches where that is small change)
    a.longest_first = (B > 1 && B <= 128 && (long long)B * c.n_kv_heads * a.mtiles * n_splits > ctx->sm_count) ? 1 : 0;
    a.scale_log2 = scale_log2;
    a.part_o = ctx->part_o; a.part_ml = ctx->part_ml; a.out = n_splits == 1 ? out : nullptr; a.status = ctx->d_status;
    if (!ctx->attn_attr_done) {
        const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
        cudaError_t e = cudaFuncSetAttribute(umma::tree_attn_umma_kernel<false>, at, umma::smem_bytes(false));
        if (e == cudaSuccess) e = cudaFuncSetAttribute(umma::tree_attn_umma_kernel<true>, at, umma::smem_bytes(true));
        if (e != cudaSuccess) return e;
        ctx->attn_attr_done = 1;
    }
    // descriptors are re-encoded only when a plane pointer or the batch changes
    static_assert(sizeof(CUtensorMap) <= sizeof(ctx->attn_tmap_k), "tensor map storage");
    CUtensorMap *mk = reinterpret_cast<CUtensorMap *>(ctx->attn_tmap_k);
    CUtensorMap *mv = reinterpret_cast<CUtensorMap *>(ctx->attn_tmap_v);
    CUtensorMap *mk_half = reinterpret_cast<CUtensorMap *>(ctx->attn_tmap_k_half);     // boxes of 64 keys: a pair's CTA loads half a K chunk
    // rows of the plane matrix: every sequence's cache, or the whole pool of blocks
    const size_t rows = paged.table ? (size_t)paged.n_blocks * c.n_kv_heads * umma::BK : (size_t)B * c.n_kv_heads * c.max_len;
    if (ctx->attn_tmap_kptr != kc || ctx->attn_tmap_vptr != vc || ctx->attn_tmap_rows != rows) {
        ctx->attn_tmap_ok = make_plane_map(mk, kc, rows) && make_plane_map(mv, vc, rows) &&
                            fspad_make_tmap_bf16_2d(mk_half, kc, (size_t)umma::D, rows, (unsigned)umma::BK / 2);
        ctx->attn_tmap_kptr = kc; ctx->attn_tmap_vptr = vc; ctx->attn_tmap_rows = rows;
    }
    a.use_tma = ctx->attn_tmap_ok ? 1 : 0;
    const bool pair = a.use_tma && in_pairs;      // (without maps the tiles go to lone CTAs, one of them perhaps empty)
    a.early = paged.early ? 1 : 0;
    a.done = paged.early && n_splits > 1 ? ctx->attn_done : nullptr;
    CUtensorMap mq = {};
    a.q_tma = make_q_map(&mq, q, (size_t)B * N, c.n_q_heads, a.G) ? 1 : 0;
    const dim3 grid = pair ? dim3(c.n_kv_heads * a.mtiles, n_splits, B) : dim3(n_splits, c.n_kv_heads * a.mtiles, B);
    ctx->launches++;
    auto kernel = pair ? umma::tree_attn_umma_kernel<true> : umma::tree_attn_umma_kernel<false>;
    return fspad_launch_opt(paged.early, kernel, grid, dim3(umma::NT), umma::smem_bytes(pair), st, pair ? 2u : 0u, a, mq, pair ? *mk_half : *mk, *mv);
}
