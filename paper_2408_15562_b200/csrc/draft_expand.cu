// Dynamic token tree, one draft step (paper, Section "Preliminaries", last
// paragraph: the output of each draft step is truncated to its top-k and every
// token carries the joint probability of its path).
//
// One kernel per call, grid (pieces of a row, rows):
//   1. every CTA streams its piece: the half-warp maxima of the first 4096 tokens give a lower
//      bound of the piece's k-th largest value, the tokens that reach it are listed in
//      shared memory, a warp cuts the list by a bound of the same kind and ranks what is left by counting; the one HBM pass over
//      the rows;
//   2. the CTA that finishes a sequence's last piece (told by a counter per sequence that it then puts back to zero; nobody
//      waits for anybody) takes one warp to a row and ranks the pieces' lists the same way; the first k
//      become candidates base + f k + r with the frontier node as parent and the joint
//      log-probability frontier_logp + value, one single-precision addition;
//   3. it ranks the F k new joint values; the first `width` are the next frontier.
// Comparisons and one addition only, so every decision is the oracle's bit for bit.
//
// What bounds it: HBM with many rows, otherwise a chain of latencies.  As three kernels (one CTA per 4096 tokens, then a
// 1024-entry sorting network per row, then one per sequence) a level of ten rows took 15 us at V = 32000 and 40 us with
// 16 sequences at V = 128256 (82 MB); with lists ranked by all threads, every member against every other, 8.1 and 23; now 7.2 and 20
// (11 sequences, 16 of 151936 tokens a row, where lists of 265 keys now and then outgrew what was ranked and were cut bit by bit: 45 -> 31).  What
// is left behind the stream is mostly a chain of code that each CTA runs once: code inlined twice, or fetched early by a call
// that does nothing, made a level 0.5 us longer, and so did lists handed on unranked.  Pieces are at most 16 per row, so that the lists merged for a row stay short.
// (Prefetching rounds further ahead into L2 or asking for the second round before the bound is known made it slower: it is not HBM's
// latency that the rounds wait for.)
#include "common.cuh"
#include "sort_key.cuh"

namespace {

constexpr int kThreads = 512;                          // one warp for each of a sequence's up to 16 rows
constexpr int kPerThread = 8;                         // tokens per thread and round
constexpr int kRound = kThreads * kPerThread;          // 4096 tokens
constexpr int kKeep = 512;                             // longest list left by a round where lists are cut between rounds
constexpr int kShort = 128;                            // longest list that is ranked by counting
constexpr int kMaxPieces = 16;

struct DraftArgs {
    const float *logprobs, *frontier_logp;
    const int *frontier_cand;
    int V, F, k, width, base, cap, pieces, len;        // len: tokens of a piece (a multiple of 32)
    unsigned long long *part;                          // [rows][pieces][k] keys, 0 where a piece has fewer tokens
    int *seq_done;                                     // pieces of a sequence's rows that have finished
    int *cand_parent, *cand_token;
    float *cand_logp;
    int *next_cand;
    float *next_logp;
};

struct DraftShared {
    unsigned long long list[kKeep + kRound];           // keys of the tokens that reach the bound
    unsigned long long top[FSPAD_MAX_FRONTIER];
    float hmax[kThreads / 16];
    alignas(16) uint32_t scratch[kThreads / 32][32];
    float joint[FSPAD_MAX_FRONTIER * FSPAD_MAX_FRONTIER];
    float bound;
    int cnt, n, hits, last;
    uint32_t lowest;
};

// The list cut to its k largest keys (a long list: ascending or constant values).  The k-th largest key is found bit by bit, a count
// of the list to a bit (0.6 us).  Tokens are below V: a key's low word has the bits above those of V - 1 set, whatever the token.  equal:
// the list was cut by a bound before, so what makes it long are keys of one value as a rule, its lowest, and the values' bits need no search.
// Constant rows, ten of 32000 tokens, 64 bits searched behind nothing / 64 behind a warp's bound / this: 42, 55 and 32 us.
__device__ __noinline__ void cut_list(DraftShared &s, int k, int V, bool equal, int tid)
{
    const int n = s.cnt, token_bits = 32 - __clz((V - 1) | 1);
    unsigned long long t = 0ull;
    int bit = 63;
    if (equal) {
        if (tid == 0) { s.lowest = 0xffffffffu; s.hits = 0; }
        __syncthreads();
        uint32_t low = 0xffffffffu;
        for (int i = tid; i < n; i += kThreads) low = min(low, (uint32_t)(s.list[i] >> 32));
        atomicMin(&s.lowest, low);
        __syncthreads();
        low = s.lowest;
        int above = 0;
        for (int i = tid; i < n; i += kThreads) above += (uint32_t)(s.list[i] >> 32) > low ? 1 : 0;
        if (above) atomicAdd(&s.hits, above);
        __syncthreads();
        if (s.hits < k) {
            t = (unsigned long long)low << 32;
            bit = 31;
        }
        __syncthreads();
    }
    for (; bit >= 0; --bit) {
        const unsigned long long with = t | (1ull << bit);
        if (bit < 32 && bit >= token_bits) {
            t = with;
            continue;
        }
        int c = 0;
        for (int i = tid; i < n; i += kThreads) c += s.list[i] >= with ? 1 : 0;
        if (tid == 0) s.hits = 0;
        __syncthreads();
        if (c) atomicAdd(&s.hits, c);
        __syncthreads();
        if (s.hits >= k) t = with;
        __syncthreads();
    }
    if (tid == 0) s.n = 0;
    __syncthreads();
    for (int i = tid; i < n; i += kThreads)
        if (s.list[i] >= t) s.top[atomicAdd(&s.n, 1)] = s.list[i];       // keys differ: exactly k of them
    __syncthreads();
    if (tid < k) s.list[tid] = s.top[tid];
    if (tid == 0) { s.cnt = k; s.bound = fspad_key_value(t); }
    __syncthreads();
}

// place of key `me` among the n keys of the list
__device__ __forceinline__ int rank_of(const unsigned long long *list, int n, unsigned long long me)
{
    int rank = 0;
#pragma unroll 4
    for (int o = 0; o < n; ++o) rank += list[o] > me ? 1 : 0;
    return rank;
}

// One warp, the n keys of `list` (0: no key): those that can be among its k <= 32 largest are moved to its front, and their number
// is returned.  The k-th largest of the lanes' maxima is a bound that k keys reach; few others do (150 keys, k = 10: about 13 are left), and
// ranking those takes a tenth of what ranking all of them against one another took (3 us of a level of 16 sequences).
__device__ __noinline__ int shorten(unsigned long long *list, int n, int k, uint32_t *scratch, int lane)
{
    uint32_t top = 0u;                                 // (the high words, the values, are enough for a bound)
    for (int i = lane; i < n; i += 32) top = max(top, (uint32_t)(list[i] >> 32));
    scratch[lane] = top;
    __syncwarp();
    int rank = 0;
#pragma unroll 2
    for (int o = 0; o < 32; o += 4) {
        const uint4 t = *reinterpret_cast<const uint4 *>(scratch + o);
        rank += (t.x > top || (t.x == top && o < lane)) + (t.y > top || (t.y == top && o + 1 < lane)) +
                (t.z > top || (t.z == top && o + 2 < lane)) + (t.w > top || (t.w == top && o + 3 < lane));
    }
    const unsigned who = __ballot_sync(0xffffffffu, rank == k - 1);
    const uint32_t bound = max(__shfl_sync(0xffffffffu, top, __ffs((int)who) - 1), 1u);      // (a key's value is never 0)
    int m = 0;
#pragma unroll 1
    for (int i = 0; i < n; i += 32) {
        const unsigned long long key = i + lane < n ? list[i + lane] : 0ull;
        const bool stays = (uint32_t)(key >> 32) >= bound;
        const unsigned all = __ballot_sync(0xffffffffu, stays);
        if (stays) list[m + __popc(all & ((1u << lane) - 1u))] = key;      // (behind every key already read, or that one itself)
        m += __popc(all);
    }
    __syncwarp();
    return m;
}

// PER_SM: CTAs an SM holds.  Four leave a thread 32 registers, which is a few too few; with three a level's chain is shorter (ten rows:
// 8.9 -> 8.1 us at 32000 tokens, 12.7 -> 11.1 at 151936).
template <int PER_SM>
__global__ void __launch_bounds__(kThreads, PER_SM)
draft_expand_kernel(const DraftArgs a)
{
    __shared__ DraftShared s;
    fspad_pdl_trigger();
    fspad_pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31;
    const int piece = blockIdx.x, row = blockIdx.y, V = a.V, k = a.k;
    const float *x = a.logprobs + (size_t)row * V;
    // Positions count from the 16-byte boundary at or before the row's first token: loads are aligned whatever V is.
    const int ph = (int)((reinterpret_cast<uintptr_t>(x) >> 2) & 3);
    const int lo = piece * a.len - ph, hi = min(V, lo + a.len);      // positions before token 0 and past `hi` are empty
    const float *__restrict__ xp = x;
    if (tid == 0) s.cnt = 0;
    float4 cur[kPerThread / 4], nxt[kPerThread / 4];
    auto fetch = [&](int e0, float4 (&v)[kPerThread / 4]) {
#pragma unroll
        for (int i = 0; i < kPerThread / 4; ++i) {
            const int j = e0 + 4 * (i * kThreads + tid);             // (groups that reach past an end of the row are looked at apart)
            v[i] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if (j >= 0 && j + 4 <= hi) v[i] = __ldg(reinterpret_cast<const float4 *>(xp + j));
        }
    };
    // the tokens of one round that reach the bound go to the list (where there is room: the count goes on in any case)
    auto push = [&](int e0) {
        const float bound = s.bound;
#pragma unroll
        for (int i = 0; i < kPerThread / 4; ++i) {
            const int tok = e0 + 4 * (i * kThreads + tid);
            const float v4[4] = {cur[i].x, cur[i].y, cur[i].z, cur[i].w};
            if (fmaxf(fmaxf(v4[0], v4[1]), fmaxf(v4[2], v4[3])) >= bound && tok >= 0 && tok + 4 <= hi) {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (v4[c] >= bound) {
                        const int at = atomicAdd(&s.cnt, 1);
                        if (at < kKeep + kRound) s.list[at] = fspad_sort_key(v4[c], (uint32_t)(tok + c));
                    }
            }
        }
    };
    fetch(lo, cur);
    {
        // The k-th largest of the 32 half-warp maxima is a lower bound of the piece's k-th largest value, because k
        // tokens at least that large exist (a half-warp without any token reports -inf, which can only
        // lower the bound and so lengthen the list, never lose a token).
        float bv = -INFINITY;
#pragma unroll
        for (int i = 0; i < kPerThread / 4; ++i) bv = fmaxf(fmaxf(bv, fmaxf(cur[i].x, cur[i].y)), fmaxf(cur[i].z, cur[i].w));
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) bv = fmaxf(bv, __shfl_xor_sync(0xffffffffu, bv, off));
        if ((lane & 15) == 0) s.hmax[tid >> 4] = bv;
        __syncthreads();
        if (tid < kThreads / 16) {
            const float me = s.hmax[tid];
            int rank = 0;
#pragma unroll
            for (int o = 0; o < kThreads / 16; ++o) {
                const float ot = s.hmax[o];
                rank += (ot > me || (ot == me && o < tid)) ? 1 : 0;
            }
            if (rank == k - 1) s.bound = me;                     // k <= 16: exactly one thread
        }
        __syncthreads();
    }
    // the up to three tokens at either end of the row that no aligned group of four covers
    auto push_ends = [&]() {
        if (tid >= 6) return;
        const int tok = tid < 3 ? lo + 1 + tid : hi - 1 - (tid - 3);
        const bool end = tid < 3 ? lo < 0 && tok >= 0 && tok < min(lo + 4, hi) : tok >= max(lo, 0) && tok >= hi - ((hi - lo) & 3) && (lo >= 0 || tok >= lo + 4);
        if (end && x[tok] >= s.bound) {
            const int at = atomicAdd(&s.cnt, 1);
            if (at < kKeep + kRound) s.list[at] = fspad_sort_key(x[tok], (uint32_t)tok);
        }
    };
    push_ends();
    for (int e0 = lo; e0 < hi; e0 += kRound) {
        if (e0 + kRound < hi) fetch(e0 + kRound, nxt);
        push(e0);
#pragma unroll
        for (int i = 0; i < kPerThread / 4; ++i) cur[i] = nxt[i];
    }
    __syncthreads();
    if (s.cnt > kKeep + kRound) {                                // (uniform) ascending or constant values: once more, the list cut between rounds
        __syncthreads();
        if (tid == 0) s.cnt = 0;
        __syncthreads();
        push_ends();
        for (int e0 = lo; e0 < hi; e0 += kRound) {
            fetch(e0, cur);
            __syncthreads();
            push(e0);
            __syncthreads();
            if (s.cnt > kKeep) cut_list(s, k, V, false, tid);
        }
    } else if (s.cnt > kShort) {                                 // cut it here only if a warp would be long about it: many equal values
        const int n = s.cnt;
        __syncthreads();
        if (tid < 32) {
            const int m = shorten(s.list, n, k, s.scratch[0], lane);
            if (lane == 0) s.cnt = m;
        }
        __syncthreads();
        if (s.cnt > kShort) cut_list(s, k, V, true, tid);
    }
    __syncthreads();
    // ---- the piece's list, and whether it is the sequence's last: one warp ----
    const int b = row / a.F;
    if (tid < 32) {
        const int n = s.cnt > 32 ? shorten(s.list, s.cnt, k, s.scratch[0], lane) : s.cnt;
        unsigned long long *out = a.part + ((size_t)row * a.pieces + piece) * k;
        for (int i = lane; i < n; i += 32) {
            const unsigned long long me = s.list[i];
            const int rank = rank_of(s.list, n, me);
            if (rank < k) __stcg(out + rank, me);
        }
        for (int r = n + lane; r < k; r += 32) __stcg(out + r, 0ull);          // empty slots
        __syncwarp();
        if (lane == 0) {
            int done;                                // (release: behind the warp's barrier it stands for the whole list)
            asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(done) : "l"(a.seq_done + b) : "memory");
            s.last = done == a.F * a.pieces - 1;
            if (s.last) a.seq_done[b] = 0;
        }
    }
    __syncthreads();
    if (s.last == 0) return;
    // ---- the last piece of the sequence: the pieces' lists of a row -> candidates, one warp to a row ----
    const int n2 = a.pieces * k;                                     // at most 256: eight entries per lane
    unsigned long long *list = s.list + (tid >> 5) * (kMaxPieces * FSPAD_MAX_FRONTIER);
    for (int f = tid >> 5; f < a.F; f += kThreads / 32) {
        const unsigned long long *in = a.part + (size_t)(b * a.F + f) * n2;
        const float above = a.frontier_logp[b * a.F + f];
        const int parent = a.frontier_cand[b * a.F + f];
        unsigned long long e[kMaxPieces * FSPAD_MAX_FRONTIER / 32];
#pragma unroll
        for (int u = 0; u < kMaxPieces * FSPAD_MAX_FRONTIER / 32; ++u) e[u] = lane + 32 * u < n2 ? __ldcg(in + lane + 32 * u) : 0ull;
        // The lists are in descending order: at least k entries are as large as the smallest of the pieces' j-th, j = k / pieces
        // rounded up.  What is below that needs no ranking.
        unsigned long long jth = ~0ull;
        if (lane < a.pieces) jth = __ldcg(in + lane * k + (k + a.pieces - 1) / a.pieces - 1);
        const uint32_t bound = max(__reduce_min_sync(0xffffffffu, (uint32_t)(jth >> 32)), 1u);
        int n = 0;
#pragma unroll
        for (int u = 0; u < kMaxPieces * FSPAD_MAX_FRONTIER / 32; ++u) {
            if (32 * u >= n2) break;
            const bool in_list = (uint32_t)(e[u] >> 32) >= bound;
            const unsigned m = __ballot_sync(0xffffffffu, in_list);
            if (in_list) list[n + __popc(m & ((1u << lane) - 1u))] = e[u];
            n += __popc(m);
        }
        if (lane < k) s.joint[f * k + lane] = -INFINITY;
        __syncwarp();
        if (n > 32) n = shorten(list, n, k, s.scratch[tid >> 5], lane);      // (many short lists: the bound is a low one)
        for (int i = lane; i < n; i += 32) {
            const unsigned long long me = list[i];
            const int rank = rank_of(list, n, me);
            if (rank < k) {
                const size_t c = (size_t)b * a.cap + a.base + f * k + rank;
                const float v = __fadd_rn(above, fspad_key_value(me));    // one fp32 addition
                a.cand_parent[c] = parent;
                a.cand_token[c] = (int)fspad_key_index(me);
                a.cand_logp[c] = v;
                s.joint[f * k + rank] = v;
            }
        }
        __syncwarp();
    }
    __syncthreads();
    // The new joint values -> next frontier: one warp where there are few places, else every value's rank by all threads (32 lanes' maxima
    // are no bound for 32 places: ten rows of 32000 tokens, width 32, 8.2 us by all threads and 9.6 by a warp; width 10 7.9 and 6.9).
    const int n_new = a.F * k;                                       // at most 256
    if (tid < n_new) s.list[tid] = fspad_sort_key(s.joint[tid], (uint32_t)tid);
    __syncthreads();
    const bool few = a.width <= FSPAD_MAX_FRONTIER;
    if (few && tid >= 32) return;
    const int n = few ? shorten(s.list, n_new, a.width, s.scratch[0], lane) : n_new;
    for (int i = tid; i < n; i += few ? 32 : kThreads) {
        const unsigned long long me = s.list[i];
        const int rank = rank_of(s.list, n, me);
        if (rank < a.width) {
            const int at = (int)fspad_key_index(me);
            a.next_cand[(size_t)b * a.width + rank] = a.base + at;
            a.next_logp[(size_t)b * a.width + rank] = s.joint[at];
        }
    }
}

}  // namespace

// pieces of 4096 tokens: the limit on vocabulary times k is stated in them
int fspad_draft_expand_pieces(int V) { return (V + kRound - 1) / kRound; }

cudaError_t fspad_launch_draft_expand(fspad_ctx *ctx, const float *logprobs, const float *frontier_logp,
                                      const int *frontier_cand, int F, int k, int width, int base, int cap, int B,
                                      int *cand_parent, int *cand_token, float *cand_logp, int *next_cand,
                                      float *next_logp, cudaStream_t st)
{
    if (B == 0) return cudaSuccess;
    // A sequence's next frontier is written while other sequences may not have read theirs yet.  Where the caller's next_* lie over
    // frontier_* in any other way than list over list of the same length, the current ones are first put aside.
    const size_t in_bytes = (size_t)B * F * sizeof(float), out_bytes = (size_t)B * width * sizeof(float);
    auto overlap = [&](const void *in, const void *out) {
        const uintptr_t i = reinterpret_cast<uintptr_t>(in), o = reinterpret_cast<uintptr_t>(out);
        return i < o + out_bytes && o < i + in_bytes;
    };
    const bool same_place = F == width && frontier_cand == next_cand && frontier_logp == next_logp;
    const bool aside = !same_place && (overlap(frontier_cand, next_cand) || overlap(frontier_cand, next_logp) ||
                                       overlap(frontier_logp, next_cand) || overlap(frontier_logp, next_logp));
    if (aside) {
        float *keep_logp = ctx->dx_front;
        int *keep_cand = reinterpret_cast<int *>(ctx->dx_front + (size_t)ctx->cfg.max_batch * FSPAD_MAX_FRONTIER);
        cudaError_t e = cudaMemcpyAsync(keep_logp, frontier_logp, in_bytes, cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(keep_cand, frontier_cand, in_bytes, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return e;
        frontier_logp = keep_logp;
        frontier_cand = keep_cand;
    }
    static_assert(kMaxPieces * FSPAD_MAX_FRONTIER <= kThreads && FSPAD_MAX_FRONTIER * FSPAD_MAX_FRONTIER <= kThreads,
                  "the merged lists have at most one entry per thread");
    DraftArgs a;
    a.V = ctx->cfg.vocab;
    const int rows = B * F;
    // One wave of CTAs at most.  Pieces of two rounds, or of one where the rows are too few to give every SM a CTA (a piece's ranking
    // and hand-over cost what two rounds do: four sequences of ten rows at 50257 tokens 16.3 -> 10 us a level); where a CTA per SM
    // leaves a row eight pieces or more, no more than that, because the SMs with two would set the pace.
    const int sms = ctx->sm_count;
    const int most = fspad_draft_expand_pieces(a.V);                 // a round of 4096 tokens (and what `part` is sized for)
    const int fill = sms / rows < most ? sms / rows : most, two = (most + 1) / 2;
    auto pieces_of = [&](int per_sm) {
        int n = (int)((long long)sms * per_sm / rows);
        const int want = two > fill ? two : fill;
        if (n > want) n = want;
        if (n > kMaxPieces) n = kMaxPieces;
        if ((long long)rows * n > sms && sms / rows >= 8) n = sms / rows;
        return n < 1 ? 1 : n;
    };
    // Three CTAs per SM, or four where whole pieces would leave three's wave a fifth empty and four's does not: 160 rows of 128256
    // tokens are 320 CTAs (72 %) against 480, 26 against 23 us a level; 80 rows 400 (90 %) against 560, 15.4 against 16.0.
    const int three = pieces_of(3), four = pieces_of(4);
    const bool use_four = four > three && (long long)rows * three * 5 < 4ll * 3 * sms;
    const int pieces = use_four ? four : three;
    const int quantum = 32;                                          // a line; pieces of equal length, or the last one sets a bound of its own from few tokens
    a.len = (((a.V + 3 + pieces - 1) / pieces) + quantum - 1) / quantum * quantum;    // (up to three empty positions in front)
    a.pieces = (a.V + 3 + a.len - 1) / a.len;
    a.logprobs = logprobs; a.frontier_logp = frontier_logp; a.frontier_cand = frontier_cand;
    a.F = F; a.k = k; a.width = width; a.base = base; a.cap = cap;
    a.part = static_cast<unsigned long long *>(ctx->dx_part);
    a.seq_done = ctx->dx_done;
    a.cand_parent = cand_parent; a.cand_token = cand_token; a.cand_logp = cand_logp;
    a.next_cand = next_cand; a.next_logp = next_logp;
    ctx->launches++;
    return fspad_launch_opt(!aside, use_four ? draft_expand_kernel<4> : draft_expand_kernel<3>, dim3(a.pieces, rows), dim3(kThreads), 0, st, 0, a);
}
