// Lossless tree acceptance, second stage: the walk from the root.
//
// Greedy (T = 0): strict comparison of each child's draft token with the
// target's argmax at its parent (paper, Section "Preliminaries": differing
// tokens and their descendants are discarded).  Sampling (T > 0, Section
// "Experiments": T = 1 with unrelaxed acceptance): recursive rejection
// sampling over the children of the current node with residual-distribution
// resampling over the whole vocabulary.
//
// One thread-block cluster serves one sequence.  The walk itself is a short
// serial chain of scalar decisions taken in fp64; whenever a decision needs a
// whole-vocabulary quantity (an exact softmax denominator, the mass of a
// residual distribution, the inverse CDF of the bonus draw) the cluster sweeps
// the node's rows, every CTA reducing its contiguous slice of the vocabulary
// and the CTAs exchanging partial sums through distributed shared memory.
// Only rows on the realised path are ever read.  The first sweep at a node
// evaluates exp((x - max)/T) in fp64 once per token and parks the values (and
// the draft row) in shared memory, from where each thread takes its share into
// registers for the sweeps that follow at that node.
//
// The residual after k rejections at a node is kept in closed form instead of
// as a vector: for a token j that has not been rejected,
//     u_j = max(p_j - c * q_j, 0),   p_j = softmax(logits/T)_j,  q_j = draft_j
// with one scalar c that grows with every rejection; a rejected token keeps the
// value it had when it was rejected.  The current target distribution is u / U
// (U = sum of u) and the current draft distribution is q restricted to the
// tokens not yet rejected, divided by its sum D.  A rejection of token x turns
// c into c + U / D, which is exactly p <- norm(max(p - q, 0)), q <- norm(q
// without x) written without materialising either vector.
//
// Where the scan has gone by the trees it has left out the rows of nodes without
// children.  A walk comes to one of them at its end at most: it then draws from the row, or
// takes its argmax, itself.
//
// The per-row maximum and argmax come exact from the vocabulary scan; its sum
// of exponentials is fp32-accurate and is trusted only when a decision clears
// a 1e-4 relative margin, otherwise (and before any residual) the exact sum is
// swept here.
//
// What bounds it is latency: a chain of sweeps, exchanges and scalar decisions on
// 16 SMs, and the fetching of its own instructions, which each launch does anew (at
// 149 KB of code a third of the warps' active time went into waiting for them; rare
// paths are therefore single, non-inlined copies, loops are not unrolled unless
// they are the hot ones).  Measured on a 128256-token row: a rejection after a
// node's first 5.3 -> 2.0 us (sweep 2.0 -> 0.8, exchange 2.4 -> 0.7, decision 0.9 ->
// 0.5), the walk of a 60-node sampling step with eight rejections 53 -> 29 us.  (Masses
// in double throughout, exact conversions of q and differences taken before scaling,
// which came after these stamps, cost a step 0.3 to 0.7 us.)
#include <climits>

#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kMaxCluster = 16;
constexpr int kSmallerCluster = 10;        // where a batch needs more clusters than fit at once
constexpr int kGreedyCluster = 8;          // all sequences greedy, rows of nodes without children not scanned
constexpr int kWalkThreads = 512;          // 128 registers each: a thread keeps 16 tokens of the node's rows in them
constexpr int kWarps = kWalkThreads / 32;
constexpr int kTile = 16;                  // tokens of a thread's chunk that later residual sweeps take from registers
constexpr int kSmemBudget = 200 * 1024;   // dynamic shared memory for the per-node cache
constexpr int kSmemBudgetWide = 168 * 1024;   // the same for the instance with room for 256 nodes (its other parts are larger)
constexpr double kAmbiguous = 1e-4;
constexpr double kScanRel = 1e-6;          // bound taken for the relative error of the scan's sum of exponentials
constexpr double kFusedTol = 1e-9;         // relative error the fused first-rejection sweep may leave in the residual mass
constexpr double k16OverLn2 = 23.083120654223414;   // steps of the exponential's table per unit of its argument
constexpr int kExpRange = 0x40cf8f17;      // high word of 700 * 16 / ln 2
constexpr float kLog2eF = 1.4426950408889634f;
constexpr int kPieceSlots = 16;            // pieces of a row whose scan sums are kept for the bonus draw
constexpr int kPieceBytes = kPieceSlots * sizeof(double);      // of one row; ahead of the per-node cache in dynamic shared memory
constexpr int kExpTable = 16;              // entries of the exponential's table: one per pair of shared-memory banks
enum { REQ_DONE = 0, REQ_EXP = 1, REQ_FUSED = 2, REQ_RESID = 3 };

// 2^(i/16), i = 0..15, correctly rounded
__constant__ double kExp2Tbl[16] = {
    1.0, 1.0442737824274138, 1.0905077326652577, 1.1387886347566916, 1.189207115002721, 1.241857812073484,
    1.2968395546510096, 1.3542555469368927, 1.4142135623730951, 1.4768261459394993, 1.5422108254079407,
    1.6104903319492543, 1.681792830507429, 1.7562521603732995, 1.8340080864093424, 1.9152065613971474,
};

struct WalkArgs {
    const float *logits, *draft, *temperature, *uniforms;
    const float *given;                 // the caller's logits: other than `logits` where they lie in host memory and the scan has brought
                                        // the rows that it reads to the device
    const int *tokens, *parent;
    const FspadStatsPart *parts;
    FspadStatsGeom geom;
    int N, V, path_stride, cache_ok;
    int draft_far;                      // the draft rows lie in host memory: not asked for ahead of need
    int B, sampled_first;               // sequences; clusters take the sampling ones first
    int *path, *n_acc, *bonus, *status;
    // optional: the cluster that has walked a sequence also moves its accepted K/V rows up (NULL: not asked for)
    uint4 *kv_cache;                    // [layers][2][B][Hkv][max_len][d] bf16 as 16-byte chunks
    const int *kv_prefix;
    int *kv_new_len;
    int kv_layers, kv_B, kv_H, kv_max_len;
};

// The walk's state at the current node; thread 0's own, in shared memory while the CTA sweeps.  Weights and masses of
// the target's side are kept times the softmax denominator S.
struct WalkState {
    double S, C, U, D, invD, F;     // denominator, coefficient of the draft row, residual mass, draft mass and its
                                    // inverse, sum of the weights that rejected tokens keep
    double Cp;                      // coefficient of the rejection under way
    double base;                    // draft mass of the tokens that no child carries (after the first rejection)
    int cur, nrem, len, ch, ridx;   // ch: child under test (0: none left); ridx: its token's place in the list of rejected ones, or -1
    int exact, parked;              // S is exact; e and q of the node's rows are parked (first rejection done)
};
// What the test of a child needs.
struct Child {
    int ch, next, tok, dup;         // next: the sibling after it (0: none)
    double ex, qx, rq;              // exponential and draft probability of its token, uniform times the latter
};

// MAXN: capacity in tree nodes of this instance of the kernel (64 or FSPAD_MAX_NODES_WIDE)
// INNER: the scan has gone by the trees and left out the rows of nodes without children
template <int MAXN, bool INNER> struct TreeShared {
    int parent[MAXN];
    int tok[MAXN];
    int path[MAXN];
    int rowA[MAXN];                 // argmax of every row
    int next[MAXN];                 // greedy: the child that carries it, MAXN if none
    int len;
    int kv_L;                       // prefix length (where the walk compacts the cache)
};
template <int MAXN> struct TreeShared<MAXN, true> : TreeShared<MAXN, false> {
    unsigned char known[MAXN];      // the scan has been over the node's row
    int last;                       // greedy: the node the walk ended at, if its row is still to be looked at, else -1
    unsigned long long best;        // ... the row's maximum and where it is (see argmax_key)
};
// The logits' rows as the walk sweeps them: those that the scan has gone over by the trees it may have brought to the device itself.
template <bool INNER> struct LogitsRow { typedef const float *__restrict__ T; };
template <> struct LogitsRow<true> { typedef FspadLateRow T; };
// (The functions that are not inlined are instantiated by it, too, so that what one kind of walk calls has no say in the other's registers.)
template <int MAXN, bool INNER> struct SharedT {
    typedef typename LogitsRow<INNER>::T Row;
    TreeShared<MAXN, INNER> t;
    alignas(128) double exp_tbl[kExpTable];      // 2^(i/16)
    // what thread 0 asks for and about which node (written by thread 0, read by all after a barrier)
    double S, C;                    // sum of exponentials in use, coefficient of the draft row
    double S_exact;                 // what the first rejection's sweep found
    WalkState state;
    int req, cur, xnew, parked;
    int nrem, sel;
    int rem_tok[MAXN];              // tokens rejected at the current node and the weights they keep
    double rem_frozen[MAXN];
    // gathered once, in parallel, before the walk: the scan result of every row and, for
    // every node, its draft probability in its parent's row and its uniform
    float rowM[MAXN];
    double rowS[MAXN];
    float cq[MAXN], cu[MAXN];
    double cex[MAXN];               // exp((logit - row max)/T) of each node's token in its parent's row
    double later_q[MAXN];           // draft mass of the tokens that only siblings after node c carry (children of nodes with a rejection)
    int first_child[MAXN], next_sib[MAXN];   // 0: none
    unsigned char dup[MAXN];        // an earlier sibling carries the same token
    float ubonus;
    int bonus_ok;                   // the last residual sweep already holds the bonus draw's per-thread sums
    int fail;
    // reductions: warp totals, totals received from every CTA of the cluster (by exchange parity), their barriers
    double warp_v[5][kWarps], warp_off[kWarps], warp_total;
    double slot[2][5][kMaxCluster];
    unsigned long long bar[2];
    int verdict;                    // bonus draw from one piece of the row: 1 = settled, 2 = the whole row must be swept
    // piece_cnt[row]: pieces of the row whose masses are kept (in dynamic shared memory); 0 when it has more than kPieceSlots
    // (the draw then sweeps the whole row)
    int piece_cnt[MAXN];
};

// ---- where the scan's partial results of a row are ----
// first CTA and number of CTAs that share row `row` (rows not cut evenly)
__device__ __noinline__ int flat_first(const FspadStatsGeom &g, int row, int *cnt)
{
    const long long r0 = (long long)row * g.upr;
    if (g.total <= 0xffffffffll) {
        const unsigned ch = (unsigned)g.chunk, f = (unsigned)r0 / ch;
        *cnt = (int)(((unsigned)r0 + (unsigned)g.upr - 1u) / ch - f) + 1;
        return (int)f;
    }
    const long long first = r0 / g.chunk, last = (r0 + g.upr - 1) / g.chunk;
    *cnt = (int)(last - first) + 1;
    return (int)first;
}
__device__ __forceinline__ int row_pieces(const FspadStatsGeom &g, int row)
{
    if (g.per_row > 0) return g.per_row;
    int cnt;
    flat_first(g, row, &cnt);
    return cnt;
}
// tokens [lo, hi) of piece `pick` of row `row`
__device__ __noinline__ void piece_bounds(const FspadStatsGeom &g, int row, int pick, int V, int *lo, int *hi)
{
    long long u_lo = pick * g.chunk, u_hi = u_lo + g.chunk;
    if (g.per_row == 0) {
        int cnt;
        const long long first = flat_first(g, row, &cnt), row_lo = (long long)row * g.upr;
        u_lo = max(0ll, (first + pick) * g.chunk - row_lo);
        u_hi = (first + pick + 1) * g.chunk - row_lo;
    }
    const int before = g.shift ? (int)(((size_t)row * V) & 3) : 0;         // positions in front of the row's first token
    *lo = max(0, (int)u_lo * g.unit - before);
    *hi = (int)min((long long)V, u_hi * g.unit - before);
}

// The scan's partials of one row, merged by eight lanes (slots lane, lane + 8 at once; any further ones in a loop).
// The whole warp calls it; `valid` is false for lanes without a row.  piece_w (may be NULL): mass of each piece relative
// to the row's maximum.
__device__ __forceinline__ void merge_row(const FspadStatsPart *__restrict__ parts, const FspadStatsGeom &g, int row, bool valid,
                                          float k, int l8, float &M, double &S, int &A, double *piece_w, int *piece_cnt)
{
    const int cnt = valid ? row_pieces(g, row) : 0;
    const FspadStatsPart *p = parts + (size_t)(valid ? row : 0) * g.slots;
    float m0 = -INFINITY, s0 = 0.f, m1 = -INFINITY, s1 = 0.f;
    int a0 = 0x7fffffff, a1 = 0x7fffffff;
    if (l8 < cnt) {
        const int4 v = __ldcg(reinterpret_cast<const int4 *>(p + l8));
        m0 = __int_as_float(v.x); s0 = __int_as_float(v.y); a0 = v.z;
    }
    if (l8 + 8 < cnt) {
        const int4 v = __ldcg(reinterpret_cast<const int4 *>(p + l8 + 8));
        m1 = __int_as_float(v.x); s1 = __int_as_float(v.y); a1 = v.z;
    }
    float m = m0;
    int a = a0;
    if (m1 > m || (m1 == m && a1 < a)) { m = m1; a = a1; }
#pragma unroll 1
    for (int sl = l8 + 16; sl < cnt; sl += 8) {
        const int4 v = __ldcg(reinterpret_cast<const int4 *>(p + sl));
        if (__int_as_float(v.x) > m || (__int_as_float(v.x) == m && v.z < a)) { m = __int_as_float(v.x); a = v.z; }
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, off);
        const int oa = __shfl_xor_sync(0xffffffffu, a, off);
        if (om > m || (om == m && oa < a)) { m = om; a = oa; }
    }
    const double w0 = (m0 != -INFINITY) ? (double)s0 * (double)exp2f((m0 - m) * k) : 0.0;
    const double w1 = (m1 != -INFINITY) ? (double)s1 * (double)exp2f((m1 - m) * k) : 0.0;
    if (piece_w != nullptr && valid) {
        piece_w[l8] = w0;
        piece_w[l8 + 8] = w1;
        if (l8 == 0) *piece_cnt = (cnt <= kPieceSlots) ? cnt : 0;
    }
    double s = w0 + w1;
#pragma unroll 1
    for (int sl = l8 + 16; sl < cnt; sl += 8) {
        const int4 v = __ldcg(reinterpret_cast<const int4 *>(p + sl));
        if (__int_as_float(v.x) != -INFINITY) s += (double)__int_as_float(v.y) * (double)exp2f((__int_as_float(v.x) - m) * k);
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    M = m;
    S = s;
    A = (a == 0x7fffffff) ? 0 : a;
}

// exp((x - m) / T) for x <= m in double precision, by table and polynomial (the scheme of Tang's 1989 paper): with
// t = (x - m) 16 / (T ln 2) = 16 n + i + f, |f| <= 1/2, the value is 2^n 2^(i/16) exp(f ln2/16).  The exponential
// of the remainder is its Taylor series to the fifth order with the sixth economised into the lower ones (error below
// 5e-15).  Sixteen entries lie in sixteen pairs of banks, so that a warp's look-ups never collide (with 256 entries and a
// cubic each cost six shared-memory cycles).  The caller hands over s = 16 / (T ln 2) and m; the difference x - m is taken
// first (of two floats it is exact or nearly so), because the rounding of a product m s has no bound at low temperatures:
// at T = 1e-12 and m = 20 it is 2 % of a step, at 1e-16 hundreds of steps.  The rounding to
// the nearest integer is done by adding and subtracting 1.5 * 2^52 (the integer then sits in the low word of the sum):
// conversions run at a quarter of the fp64 rate (16 against 63 per clock and SM).  Values below e^-700 are taken as zero.
struct ExpArg {
    double s, m;
};
__device__ __forceinline__ ExpArg exp_arg(float m, double invT) { return ExpArg{invT * k16OverLn2, (double)m}; }
__device__ __forceinline__ double exp_neg(float x, const ExpArg &g, const double *tbl)
{
    const double magic = 6755399441055744.0;              // 1.5 * 2^52
    const double t = ((double)x - g.m) * g.s;
    const double tm = t + magic;
    const double f = t - (tm - magic);
    const int k = __double2loint(tm);
    double p = fma(f, 1.2715871950558131e-09, 1.4676444618653448e-07);
    p = fma(p, f, 1.3550807779497457e-05);
    p = fma(p, f, 0.0009383847924862099);
    p = fma(p, f, 0.04332169878499658);
    p = fma(p, f, 1.0000000000000044);
    const double y = tbl[k & (kExpTable - 1)] * p;
    const double e = __hiloint2double(__double2hiint(y) + ((k >> 4) << 20), __double2loint(y));
    // |t| < 16158.2 = 700 * 16 / ln 2, told by the high word alone (to one part in a million): false for -inf and NaN, too
    return (__double2hiint(t) & 0x7fffffff) < kExpRange ? e : 0.0;
}

// w where it is not negative, else zero, without a branch (tokens of a warp are of both kinds)
__device__ __forceinline__ double positive(double w)
{
    const int keep = ~(__double2hiint(w) >> 31);
    return __hiloint2double(__double2hiint(w) & keep, __double2loint(w) & keep);
}

// All weights are kept times the softmax denominator S: w = max(e - C q, 0) with e = exp((x - m)/T) and C = c S.
__device__ __forceinline__ double weight(double e, double q, double C)
{
    const double w = fma(-C, q, e);
    return w > 0.0 ? w : 0.0;
}

// ---- how a row is shared out ----
// Every CTA of the cluster takes a contiguous stretch, every thread of it per_thr positions, a multiple of four.  The
// boundaries are multiples of 16 bytes from the array's start, whatever V is (both arrays start on one): positions before
// the row's first token (at most three, of the first thread) and past its last one are empty.
struct Chunk {
    int lo, hi;                     // first position (may be -1 .. -3), end of the tokens
};
__device__ __forceinline__ Chunk chunk_of(size_t row_start, int V, int per_cta, int per_thr, int rank, int tid)
{
    const int ph = (int)(row_start & 3);
    const int end = (rank + 1) * per_cta;
    const int u = min(end, rank * per_cta + tid * per_thr);
    return Chunk{u - ph, min(V, min(end, u + per_thr) - ph)};
}
enum { MODE_EXP = 0, MODE_RESID = 1, MODE_CDF = 2 };

// The sweeps that are not on the usual path, over this thread's chunk, from the arrays in global memory or, with
// `parked`, from the e_j and q_j the first rejection's sweep left in shared memory (one copy, not inlined).
//   MODE_EXP  : sum of e_j
//   MODE_RESID: sum of the weights at coefficient C over the tokens neither rejected before nor equal to xnew
//               (rows that do not fit into shared memory)
//   MODE_CDF  : sum of the weights the bonus token is drawn from (a rejected token's is the one it keeps)
// With `found` the running sum starts at run and *found receives the first token where it exceeds target (else the
// last positive-weight token).
template <class Shared>
__device__ __noinline__ double sweep_row(int mode, const Shared &sh, typename Shared::Row x, const float *__restrict__ q,
                                         const double *__restrict__ se, const float *__restrict__ sq, int stride, Chunk ck,
                                         bool parked, const ExpArg &arg, double C, int xnew, double run, double target, int *found)
{
    const int nrem = mode == MODE_EXP ? 0 : sh.nrem;
    bool special = mode == MODE_RESID && xnew >= ck.lo && xnew < ck.hi;
#pragma unroll 1
    for (int r = 0; r < nrem; ++r) special |= (sh.rem_tok[r] >= ck.lo && sh.rem_tok[r] < ck.hi);
    double a = 0.0;
    int last_pos = -1, hit = -1;
#pragma unroll 1
    for (int j = ck.lo; j < ck.hi; j += 4) {
        double ev[4], qv[4] = {0.0, 0.0, 0.0, 0.0};
        if (parked) {
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                ev[t] = se[(j - ck.lo + t) * stride];
                qv[t] = (double)sq[(j - ck.lo + t) * stride];
            }
        } else {
            const float4 xs = fspad_load4(x, j, ck.hi, -INFINITY);
            ev[0] = exp_neg(xs.x, arg, sh.exp_tbl); ev[1] = exp_neg(xs.y, arg, sh.exp_tbl);
            ev[2] = exp_neg(xs.z, arg, sh.exp_tbl); ev[3] = exp_neg(xs.w, arg, sh.exp_tbl);
            if (C != 0.0) {
                const float4 qs = fspad_load4(q, j, ck.hi, 0.f);
                qv[0] = (double)qs.x; qv[1] = (double)qs.y; qv[2] = (double)qs.z; qv[3] = (double)qs.w;
            }
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            double w = weight(ev[t], qv[t], C);
            if (special) {
#pragma unroll 1
                for (int r = 0; r < nrem; ++r)
                    if (sh.rem_tok[r] == j + t) w = mode == MODE_CDF ? sh.rem_frozen[r] : 0.0;
                if (mode == MODE_RESID && j + t == xnew) w = 0.0;
            }
            a += w;
            run += w;
            if (w > 0.0) last_pos = j + t;
            if (hit < 0 && w > 0.0 && run > target) hit = j + t;
        }
    }
    if (found != nullptr) *found = (hit >= 0) ? hit : last_pos;
    return a;
}

// The residual sweep over the values parked in shared memory (rows of more than kTile tokens a thread): sum of
// max(e_j - C q_j, 0) over this thread's chunk without the tokens rejected so far, whose parked values are zero (as are
// the empty positions).
__device__ __noinline__ double parked_sweep(double *__restrict__ se, float *__restrict__ sq, int stride, Chunk ck, int per_thr,
                                            double C, int xnew)
{
    if (xnew >= ck.lo && xnew < ck.hi) {
        se[(xnew - ck.lo) * stride] = 0.0;
        sq[(xnew - ck.lo) * stride] = 0.f;
    }
    double a[2] = {0.0, 0.0};
#pragma unroll 1
    for (int k = 0; k < per_thr; k += 4) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            a[t & 1] += positive(fma(-C, (double)sq[(k + t) * stride], se[(k + t) * stride]));
        }
    }
    return a[0] + a[1];
}

// The same from registers: a conversion, a multiply-add, a look at the sign in the high word and an addition per token, no
// shared-memory traffic.  q is converted by the instruction, which is exact for zeros, denormals and a negative zero alike: the
// coefficient it is multiplied by has no bound (a rejection adds U / D, and D, the draft mass left, may be a denormal itself),
// so no draft probability is too small to matter.  At 16 per clock and SM the conversions take 512 cycles of a sweep of 16
// tokens a thread, most of them beside the sums; widening zeros and normal numbers by integer operations, with another way
// for threads that hold anything else, took longer (60-node step at 2 K keys: 42.2 against 40.2 us with many rejections,
// 34.7 against 34.3 with few; 39.9 and 33.6 with integer operations that are exact for normal numbers only).
__device__ __forceinline__ double residual_of_tile(const double (&er)[kTile], const float (&qr)[kTile], int per_thr, double C)
{
    double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int b = 0; b < kTile; b += 4) {
        if (b < per_thr) {
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                a[t] += positive(fma(-C, (double)qr[b + t], er[b + t]));
            }
        }
    }
    return (a[0] + a[1]) + (a[2] + a[3]);
}

// The first rejection at a node, in one sweep.  The exact denominator S is not known yet and the residual is taken at
// C = S: with P = { j : e_j - S' q_j > 0 } taken at the scan's S',
//   sum_j max(e_j - S q_j, 0) = sum_P (e_j - S' q_j) - (S - S') sum_P q_j        for every S that leaves P unchanged.
// The sweep returns (j = xnew, the token being rejected, counts in the first and, parked, is zero from here on)
//   v[0] = sum e_j (= S)                    v[1] = sum_P (e_j - S' q_j), xnew left out
//   v[2] = sum of q_j over the tokens that no child of the node carries (the draft mass left by any rejections here is
//          this plus what the siblings still to be tested carry)
//   v[3] = sum_P q_j                        v[4] = sum of e_j over the tokens whose sign a relative error kScanRel of S'
//                                                  could flip;
// a flipped token changes the result by at most kScanRel times its e_j, so kScanRel times that sum bounds the error and the
// caller sweeps again at the exact S when that is not negligible.
// e_j and q_j are parked in shared memory, zeros in the empty positions.  The loop is kept short (four tokens, the next
// four in flight): it runs two or three times per launch, and eight unrolled tokens spent longer on their first pass
// through the instruction cache (3 us) than on the work.
template <class Shared>
__device__ __forceinline__ void fused_reject_sweep(const Shared &sh, typename Shared::Row x, const float *__restrict__ q,
                                                   double *__restrict__ se, float *__restrict__ sq, int stride, Chunk ck,
                                                   int per_thr, bool park, const ExpArg &arg, double S, int xnew, int node,
                                                   int n_nodes, double (&v)[5])
{
    // Which of this thread's first 64 positions hold a child's token: the warp's lanes look at the nodes side by side, and
    // only for the few tokens that fall into the warp's stretch is the owner told.
    unsigned long long kids = 0ull;
    bool far = false;                            // (a position from 64 on: the token is compared with the children one by one)
    {
        const int lane = threadIdx.x & 31;
        const int w_lo = __shfl_sync(0xffffffffu, ck.lo, 0), w_hi = __shfl_sync(0xffffffffu, ck.hi, 31);
#pragma unroll 1
        for (int n0 = 0; n0 < n_nodes; n0 += 32) {
            const int c = n0 + lane;
            const int t = (c < n_nodes && sh.t.parent[c] == node) ? sh.t.tok[c] : -8;
#pragma unroll 1
            for (unsigned m = __ballot_sync(0xffffffffu, t >= w_lo && t < w_hi && t >= 0); m; m &= m - 1) {
                const int ct = __shfl_sync(0xffffffffu, t, __ffs((int)m) - 1);
                if (ct >= ck.lo && ct < ck.hi) {
                    if (ct - ck.lo < 64) kids |= 1ull << (ct - ck.lo);
                    else far = true;
                }
            }
        }
    }
    v[0] = v[1] = v[2] = v[3] = v[4] = 0.0;
    float4 x4 = fspad_load4(x, ck.lo, ck.hi, -INFINITY), q4 = fspad_load4(q, ck.lo, ck.hi, 0.f);
#pragma unroll 1
    for (int k = 0; k < per_thr; k += 4) {
        float4 xn = x4, qn = q4;
        if (k + 4 < per_thr) {
            xn = fspad_load4(x, ck.lo + k + 4, ck.hi, -INFINITY);
            qn = fspad_load4(q, ck.lo + k + 4, ck.hi, 0.f);
        }
        double ev[4] = {exp_neg(x4.x, arg, sh.exp_tbl), exp_neg(x4.y, arg, sh.exp_tbl), exp_neg(x4.z, arg, sh.exp_tbl),
                        exp_neg(x4.w, arg, sh.exp_tbl)};
        float qv[4] = {q4.x, q4.y, q4.z, q4.w};
        v[0] += (ev[0] + ev[1]) + (ev[2] + ev[3]);
        double qd = ((double)qv[0] + (double)qv[1]) + ((double)qv[2] + (double)qv[3]);   // what counts towards the draft mass
        if (k < 64 ? ((unsigned)(kids >> k) & 15u) != 0u : far) {
            qd = 0.0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int id = ck.lo + k + t;
                bool kid = k < 64 && ((kids >> (k + t)) & 1ull) != 0ull;
                if (k >= 64)
#pragma unroll 1
                    for (int c = 1; c < n_nodes; ++c) kid |= sh.t.parent[c] == node && sh.t.tok[c] == id;
                if (!kid) qd += (double)qv[t];
                if (id == xnew) { ev[t] = 0.0; qv[t] = 0.f; }
            }
        }
        v[2] += qd;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const double e = ev[t];
            if (park) {
                se[(k + t) * stride] = e;
                sq[(k + t) * stride] = qv[t];
            }
            const double q64 = (double)qv[t], w = fma(-S, q64, e);
            v[1] += positive(w);
            v[3] += __double2hiint(w) >= 0 ? q64 : 0.0;
            // |w| <= kScanRel * e needs the binary exponent of w at least 19 below that of e: an
            // integer comparison sorts out all but a handful of tokens
            if ((__double2hiint(w) & 0x7ff00000) <= (__double2hiint(e) & 0x7ff00000) - (19 << 20))
                if (e > 0.0 && fabs(w) <= kScanRel * e) v[4] += e;
        }
        x4 = xn;
        q4 = qn;
    }
}

// ---- sums over the cluster ----
// A CTA's totals go to every CTA of the cluster as asynchronous remote stores that count their bytes on the receiver's
// barrier; only warp 0 waits.  (With remote stores, a cluster-wide barrier of all threads and two more CTA barriers an
// exchange took 2.4 us.)  The wait is bounded like every other.
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void send_double(uint32_t dst, uint32_t bar, int peer, double v)
{
    asm volatile("{\n\t.reg .b32 d, b;\n\tmapa.shared::cluster.u32 d, %0, %2;\n\tmapa.shared::cluster.u32 b, %1, %2;\n\t"
                 "st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [d], %3, [b];\n\t}\n"
                 :: "r"(dst), "r"(bar), "r"(peer), "l"(__double_as_longlong(v)) : "memory");
}
__device__ __forceinline__ void expect_bytes(uint32_t bar, int bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
constexpr uint32_t kPolls = 2000000;                 // about 50 ms
__device__ __forceinline__ bool wait_cluster(uint32_t bar, uint32_t parity, uint32_t polls = kPolls)
{
#pragma unroll 1
    for (uint32_t i = 0; i < polls; ++i) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

// The same wait by every thread of the CTA.  What a thread has seen is its own: one may give up just before the last bytes
// land and the next may not, and barriers of the CTA in what follows would then be reached by some only.  So nobody goes on
// before all have waited, and all go on (true) or none does.
template <class Shared>
__device__ __forceinline__ bool wait_cluster_all(Shared &sh, uint32_t bar, uint32_t parity, uint32_t polls = kPolls)
{
    if (!wait_cluster(bar, parity, polls)) sh.fail = 1;
    __syncthreads();
    return sh.fail == 0;
}

// block-wide scan of one value per thread (index order): this thread's exclusive and inclusive prefix and the CTA total
template <class Shared>
__device__ __noinline__ double block_scan(Shared &sh, double v, double *excl_out, double *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double t2 = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += t2;
    }
    const double prev_incl = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 31) sh.warp_v[0][wid] = incl;
    __syncthreads();
    if (wid == 0) {
        // exclusive scan of the warp totals; the last inclusive value is the CTA total
        double sc = (lane < kWarps) ? sh.warp_v[0][lane] : 0.0;
#pragma unroll
        for (int off = 1; off < kWarps; off <<= 1) {
            const double t2 = __shfl_up_sync(0xffffffffu, sc, off);
            if (lane >= off) sc += t2;
        }
        const double excl = __shfl_up_sync(0xffffffffu, sc, 1);
        if (lane < kWarps) sh.warp_off[lane] = (lane == 0) ? 0.0 : excl;
        if (lane == kWarps - 1) sh.warp_total = sc;
    }
    __syncthreads();
    const double woff = sh.warp_off[wid];
    *excl_out = (lane == 0) ? woff : woff + prev_incl;
    *total = sh.warp_total;
    return woff + incl;
}

// The bonus draw from a row that the scan has left out: inverse CDF of its softmax.  Every CTA takes its own slice's maximum for the
// row's; the slices' masses are brought to the largest of them when all have come, in one exchange.  The row is read once and kept in
// shared memory (`park`, NULL where it does not fit).  `last`: the thread has the last tokens of its CTA.  false: a wait ran out.
template <class Shared>
__device__ __forceinline__ bool draw_from_row(Shared &sh, const float *__restrict__ x, float *__restrict__ park, Chunk ck, int per_thr,
                                              bool last, int rank, int C, int par, uint32_t phase, double invT, int V, int *bonus)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    float m = -INFINITY;
#pragma unroll 1
    for (int j = ck.lo; j < ck.hi; j += 16) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = fspad_load4(x, j + 4 * u, ck.hi, -INFINITY);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            m = fmaxf(m, fmaxf(fmaxf(v[u].x, v[u].y), fmaxf(v[u].z, v[u].w)));
            const int k = j - ck.lo + 4 * u;
            if (park != nullptr && k < per_thr) {
                park[k * kWalkThreads] = v[u].x;
                park[(k + 1) * kWalkThreads] = v[u].y;
                park[(k + 2) * kWalkThreads] = v[u].z;
                park[(k + 3) * kWalkThreads] = v[u].w;
            }
        }
    }
    const int n = max(ck.hi - ck.lo, 0);
    auto token = [&](int k) { return park != nullptr ? park[k * kWalkThreads] : ck.lo + k < 0 ? -INFINITY : x[ck.lo + k]; };
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if (lane == 0) sh.warp_v[1][wid] = (double)m;
    __syncthreads();
    m = (float)sh.warp_v[1][lane % kWarps];
#pragma unroll
    for (int off = kWarps / 2; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    const ExpArg arg = exp_arg(m, invT);
    double mine = 0.0;
#pragma unroll 4
    for (int k = 0; k < n; ++k) mine += exp_neg(token(k), arg, sh.exp_tbl);
    double E, total;
    const double P = block_scan(sh, mine, &E, &total);
    const uint32_t bar = smem_addr(&sh.bar[par]);
    if (tid == 0) expect_bytes(bar, C * 16);
    if (tid < C) {
        send_double(smem_addr(&sh.slot[par][0][rank]), bar, tid, total);
        send_double(smem_addr(&sh.slot[par][1][rank]), bar, tid, (double)m);
    }
    if (!wait_cluster_all(sh, bar, phase)) return false;
    const float own = lane < C ? (float)sh.slot[par][1][lane & (kMaxCluster - 1)] : -INFINITY;
    float top = own;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
    const double scale = exp_neg(own, exp_arg(top, invT), sh.exp_tbl);       // (lane r: CTA r's)
    double cum = lane < C ? sh.slot[par][0][lane & (kMaxCluster - 1)] * scale : 0.0;
#pragma unroll
    for (int off = 1; off < kMaxCluster; off <<= 1) {
        const double t = __shfl_up_sync(0xffffffffu, cum, off);
        if (lane >= off) cum += t;
    }
    const double target = (double)sh.ubonus * __shfl_sync(0xffffffffu, cum, C - 1);
    const double before = __shfl_sync(0xffffffffu, cum, rank > 0 ? rank - 1 : 0);
    const int owner = __ffs((int)__ballot_sync(0xffffffffu, lane < C && cum > target)) - 1;
    if (owner == rank) {
        const double local = (target - (rank > 0 ? before : 0.0)) / __shfl_sync(0xffffffffu, scale, rank);
        if (tid == 0) sh.sel = 0x7fffffff;
        __syncthreads();
        if (P > local) atomicMin(&sh.sel, tid);
        __syncthreads();
        // (the rounding of the two levels can leave no thread above the target: the last tokens of the CTA then take the draw)
        if (tid == sh.sel || (sh.sel == 0x7fffffff && last && ck.lo < ck.hi)) {
            double run = E;
            int found = max(ck.lo, 0);                        // the first token above the target, else the last of positive weight
#pragma unroll 1
            for (int k = 0; k < n; ++k) {
                const double w = exp_neg(token(k), arg, sh.exp_tbl);
                run += w;
                if (w > 0.0) found = ck.lo + k;
                if (w > 0.0 && run > local) break;
            }
            *bonus = found;
        }
    }
    if (owner < 0 && rank == 0 && tid == 0) *bonus = 0;       // no positive weight anywhere
    return true;
}

// Compaction of the accepted path by the CTAs that walked it (every CTA of the cluster holds the same path in
// its shared memory): row L + path[j] -> row L + j of every (layer, K/V, head) slice of the sequence, one warp
// per slice, eight rows in flight, every load of a batch before any of its stores (path[j] >= j and the path
// is increasing, so moves in index order never overwrite a row that is still to be read).  The same moves as
// the stand-alone compaction kernel makes; doing them here saves the step one dependent launch.
template <typename Tree>
__device__ __noinline__ void compact_accepted(const WalkArgs &args, const Tree &sh, int b, int rank, int C, int tid, int nthr)
{
    const int lane = tid & 31, n_warps = nthr >> 5;
    int n = sh.len;
    const int L = sh.kv_L;
    if (L < 0 || n < 1 || L + sh.path[n - 1] >= args.kv_max_len) {
        if (rank == 0 && tid == 0) fspad_report(args.status, FSPAD_ERR_RANGE);
        n = 0;
    }
    if (rank == 0 && tid == 0 && args.kv_new_len) args.kv_new_len[b] = max(L, 0) + n;
    const int per_seq = args.kv_layers * 2 * args.kv_H;
    const int chunk = lane & 15, half = lane >> 4;
#pragma unroll 1
    for (int s = (tid >> 5) * C + rank; s < per_seq; s += C * n_warps) {
        const int lk = s / args.kv_H, h = s % args.kv_H;
        uint4 *base = args.kv_cache + ((((size_t)lk * args.kv_B + b) * args.kv_H + h) * args.kv_max_len + L) * 16;
#pragma unroll 1
        for (int j0 = 0; j0 < n; j0 += 8) {
            uint4 v[4];
            int dst[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + 2 * u + half;
                dst[u] = -1;
                if (j < n) {
                    const int src = sh.path[j];
                    if (src != j) {
                        v[u] = base[(size_t)src * 16 + chunk];
                        dst[u] = j;
                    }
                }
            }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (dst[u] >= 0) base[(size_t)dst[u] * 16 + chunk] = v[u];
        }
    }
}

// Node c of the tree (its thread's), checked: the parent is a lower node, the token lies in the vocabulary.
__device__ __forceinline__ void check_node(int c, int V, int &p, int &t, int *status)
{
    if (c == 0 ? p != -1 : (p < 0 || p >= c)) {
        fspad_report(status, FSPAD_ERR_BAD_TREE);
        p = 0;
    }
    if (c == 0) p = -1;
    if (t < 0 || t >= V) {
        fspad_report(status, FSPAD_ERR_RANGE);
        t = 0;
    }
}

// The row of a node without children, which the scan by the trees has left out.  Maximum and lowest index in one word: the larger
// word is the larger value or, of equal ones (the two zeros are), the lower index.
__device__ __forceinline__ unsigned long long argmax_key(float m, int a)
{
    const unsigned u = __float_as_uint(m + 0.0f);
    return ((unsigned long long)(u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u)) << 32) | (0xffffffffu - (unsigned)a);
}
// The largest key of row positions [lo, hi), of which lo (it may lie before the row's first) is on a 16-byte boundary, into t.best (set to
// 0 before; the caller's barrier comes after).  Eight loads in flight a thread: on one CTA a 128256-token row is bound by what one SM
// can have under way.
template <typename Tree>
__device__ __noinline__ void argmax_row(Tree &t, const float *__restrict__ x, int lo, int hi, int tid, int nthr)
{
    constexpr int kLoads = 8;
    float m = -INFINITY;
    int a = 0x7fffffff;
#pragma unroll 1
    for (int j0 = lo + 4 * tid; j0 < hi; j0 += 4 * kLoads * nthr) {
        float4 v[kLoads];
#pragma unroll
        for (int u = 0; u < kLoads; ++u) {
            const int j = j0 + 4 * u * nthr;
            v[u] = fspad_load4(x, j, hi, -INFINITY);
        }
#pragma unroll
        for (int u = 0; u < kLoads; ++u) {
            const int j = j0 + 4 * u * nthr;
            if (v[u].x > m) { m = v[u].x; a = j; }
            if (v[u].y > m) { m = v[u].y; a = j + 1; }
            if (v[u].z > m) { m = v[u].z; a = j + 2; }
            if (v[u].w > m) { m = v[u].w; a = j + 3; }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, off);
        const int oa = __shfl_xor_sync(0xffffffffu, a, off);
        if (om > m || (om == m && oa < a)) { m = om; a = oa; }
    }
    if ((tid & 31) == 0) atomicMax(&t.best, argmax_key(m, a));
}
__device__ __forceinline__ int argmax_of(unsigned long long key)
{
    const unsigned a = 0xffffffffu - (unsigned)key;
    return a == 0x7fffffffu ? 0 : (int)a;        // (nothing above -inf anywhere)
}

// Greedy walk of one sequence by one CTA: strict comparison of the draft tokens with the target's argmax.  Every node looks
// at its parent's argmax side by side; what is left for one thread is to follow the chain of matches.
template <bool INNER, int MAXN>
__device__ __forceinline__ void greedy_walk(TreeShared<MAXN, INNER> &t, const WalkArgs &args, int b, int N, int tid, int nthr, bool writer)
{
    if (tid < MAXN) t.next[tid] = MAXN;
    __syncthreads();
    if (tid >= 1 && tid < N && t.tok[tid] == t.rowA[t.parent[tid]]) atomicMin(&t.next[t.parent[tid]], tid);   // lowest node index
    __syncthreads();
    if (tid == 0) {                               // every CTA of a cluster: same data, same path
        int cur = 0, len = 1;
        t.path[0] = 0;
#pragma unroll 1
        for (int nx = t.next[0]; nx < MAXN; nx = t.next[nx]) {
            t.path[len++] = nx;
            cur = nx;
        }
        t.len = len;
        bool known = true;
        if constexpr (INNER) {
            known = t.known[cur] != 0;
            t.last = known ? -1 : cur;
            t.best = 0ull;
        }
        if (writer) {
            args.n_acc[b] = len;
            if (known) args.bonus[b] = t.rowA[cur];
        }
    }
    __syncthreads();
    if (writer) {
        int *out_path = args.path + (size_t)b * args.path_stride;
#pragma unroll 1
        for (int i = tid; i < args.path_stride; i += nthr) out_path[i] = (i < t.len) ? t.path[i] : -1;
    }
}

// All sequences greedy: one CTA per sequence, nothing of the sampling walk's apparatus.  INNER: the scan has gone by the trees, and
// a cluster of CTAs shares the row of a node without children that the walk ends in.
template <int MAXN, bool INNER>
__global__ void __launch_bounds__(kWalkThreads)
accept_greedy_kernel(const __grid_constant__ WalkArgs args)
{
    __shared__ TreeShared<MAXN, INNER> t;
    __shared__ unsigned long long peer_best[kGreedyCluster];
    cg::cluster_group cluster = cg::this_cluster();
    const int C = INNER ? (int)cluster.num_blocks() : 1, rank = INNER ? (int)cluster.block_rank() : 0;
    const int b = blockIdx.x / C, tid = threadIdx.x, nthr = blockDim.x, N = args.N;
    fspad_pdl_trigger();
    if constexpr (INNER) {
        if (tid < MAXN) t.known[tid] = tid == 0;
        __syncthreads();
    }
    // (read before the scan has finished: see the sampling kernel)
    const float Tf = args.temperature[b];
    int p = -1, tk = 0;
    if (tid < N) {
        p = args.parent[(size_t)b * N + tid];
        tk = args.tokens[(size_t)b * N + tid];
        check_node(tid, args.V, p, tk, args.status);
        t.parent[tid] = p;
        t.tok[tid] = tk;
        if constexpr (INNER)
            if (tid > 0) t.known[p] = 1;
    }
    if constexpr (INNER) {
        __syncthreads();
        cluster.barrier_arrive();
    }
    if (tid == 0 && args.kv_cache != nullptr) t.kv_L = args.kv_prefix[b];
    if (tid == 0 && !(Tf >= 0.0f)) fspad_report(args.status, FSPAD_ERR_RANGE);
    if (tid == 0 && Tf > 0.0f) fspad_report(args.status, FSPAD_ERR_NULL);      // a sampling sequence without draft rows
    fspad_pdl_wait();
    const int l8 = tid & 7;
#pragma unroll 1
    for (int r0 = 0; r0 < N; r0 += nthr >> 3) {      // whole warps iterate together
        const int row = r0 + (tid >> 3);
        float M; double S; int A;
        bool scanned = row < N;
        if constexpr (INNER) scanned = scanned && t.known[row];
        merge_row(args.parts, args.geom, b * N + row, scanned, 0.f, l8, M, S, A, nullptr, nullptr);
        if (l8 == 0 && row < N) t.rowA[row] = A;
    }
    __syncthreads();
    if constexpr (INNER) cluster.barrier_wait();     // (every CTA of the cluster is there before anything is written to it)
    greedy_walk<INNER>(t, args, b, N, tid, nthr, rank == 0);       // every CTA of the cluster: same data, same path
    if constexpr (INNER) {
        if (t.last >= 0) {
            const size_t start = ((size_t)b * N + t.last) * args.V;
            const int ph = (int)(start & 3), each = (((args.V + 3 + C - 1) / C) + 3) & ~3;
            argmax_row(t, args.given + start, rank * each - ph, min(args.V, (rank + 1) * each - ph), tid, nthr);
            __syncthreads();
            if (tid == 0) *cluster.map_shared_rank(&peer_best[rank], 0) = t.best;  // (a word each: rank 0 clears its own t.best at a time of its own, and a maximum sent there might come before)
            cluster.sync();
            if (rank == 0 && tid == 0) {
                unsigned long long best = peer_best[0];
                for (int r = 1; r < C; ++r) best = max(best, peer_best[r]);
                args.bonus[b] = argmax_of(best);
            }
        }
    }
    if (args.kv_cache != nullptr) compact_accepted(args, t, b, rank, C, tid, nthr);
}

// INNER: the scan has gone by the trees.  (An instance of its own: the few instructions more cost a walk behind a scan of all rows half
// a microsecond, and this one has no use for the pieces' masses.)
template <int MAXN, bool INNER>
__global__ void __launch_bounds__(kWalkThreads, 1)
accept_walk_kernel(const __grid_constant__ WalkArgs args)
{
    typedef SharedT<MAXN, INNER> Shared;
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int N = args.N, V = args.V;

    __shared__ Shared sh;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    // mass of every (row, CTA) piece of the vocabulary scan, relative to the row maximum
    double (*piece_w)[kPieceSlots] = reinterpret_cast<double (*)[kPieceSlots]>(dyn_smem);

    fspad_pdl_trigger();
    int b = blockIdx.x / C;
    if (args.sampled_first) {
        // More clusters than the SMs hold at once: they are dispatched in index order, so the long walks should come first.
        // Every CTA takes the sequence whose place in that order (sampling ones, then greedy ones, by index) is its own.
        const bool samples = tid < args.B && args.temperature[tid] > 0.0f;
        const unsigned m = __ballot_sync(0xffffffffu, samples);
        if (lane == 0) sh.warp_off[wid] = (double)__popc(m);
        __syncthreads();
        int before = __popc(m & ((1u << lane) - 1u)), total = 0;
#pragma unroll 1
        for (int w = 0; w < kWarps; ++w) {
            const int n = (int)sh.warp_off[w];
            if (w < wid) before += n;
            total += n;
        }
        if (tid < args.B && (samples ? before : total + tid - before) == b) sh.cur = tid;
        __syncthreads();
        b = sh.cur;
    }
    // The vocabulary scan that precedes this kernel in the stream lets it start only after the scan's
    // own predecessor has completed, and the scan writes nothing of the caller's: only its partial
    // results and, of logits in host memory, the rows that it brings to the device.  So the
    // caller's arrays may be read before the scan has finished: the prologue's two round trips of
    // dependent loads run under the scan's tail.
    // Round trip 1: everything that depends on nothing - temperature, tree arrays, uniforms.
    float Tf = args.temperature[b];
    if (!(Tf > 0.0f) && rank > 0) return;        // a greedy sequence is one CTA's work: the others make room for the next cluster
    int p = -1, t = 0;
    float uval = 0.f;
    if (tid < N) {
        p = args.parent[(size_t)b * N + tid];
        t = args.tokens[(size_t)b * N + tid];
    }
    if (tid <= N) uval = args.uniforms[(size_t)b * (N + 1) + (tid == 0 ? N : tid)];   // thread c: node c's uniform; thread 0: the bonus uniform
    if (tid == 32 && args.kv_cache != nullptr) sh.t.kv_L = args.kv_prefix[b];
    // (the loads above are under way)
    if (tid < kExpTable) sh.exp_tbl[tid] = kExp2Tbl[tid];
    if (tid < MAXN) {
        sh.first_child[tid] = MAXN;
        if constexpr (INNER) sh.t.known[tid] = tid == 0;
    }
    if (tid == 0) {
        sh.fail = 0;
        for (int i = 0; i < 2; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_addr(&sh.bar[i])));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();
    // (the peers' barriers are initialised before anything is sent to them: waited for below)
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    if (!(Tf >= 0.0f)) {
        if (tid == 0 && rank == 0) fspad_report(args.status, FSPAD_ERR_RANGE);
        Tf = 0.0f;
    }
    const bool sampling = Tf > 0.0f;
    const size_t row0 = (size_t)b * N;           // the sequence's first row
    typedef typename Shared::Row Row;
    const Row lg{args.logits + row0 * V};
    const float *dp = args.draft + row0 * V;
    const float kT = kLog2eF / (sampling ? Tf : 1.0f);

    // Round trip 2: thread c owns node c (tree arrays, and the scalars its accept test needs: target logit and draft
    // probability of its token in its parent's row).
    float xv = 0.f, qv = 0.f;
    if (tid < N) {
        check_node(tid, V, p, t, args.status);
        sh.t.parent[tid] = p;
        sh.t.tok[tid] = t;
        if (tid >= 1) {
            atomicMin(&sh.first_child[p], tid);
            if constexpr (INNER) sh.t.known[p] = 1;
            if (sampling) {
                const size_t at = (size_t)p * V + t;
                xv = args.given[row0 * V + at];                        // (the scan may still be bringing the row)
                qv = dp[at];
            }
        }
    }
    // how a row is shared out (positions of the row plus up to three in front of it)
    const int per_cta = (((V + 3 + C - 1) / C) + 3) & ~3;
    const int per_thr = (((per_cta + kWalkThreads - 1) / kWalkThreads) + 3) & ~3;
    {
        // The root's draft row is the one most likely to be swept: ask for it now (a hint, no register
        // is tied up and nothing waits for it).
        const Chunk ck = chunk_of(row0 * V, V, per_cta, per_thr, rank, tid);
        if (sampling && !args.draft_far && ck.lo >= 0 && ck.lo < ck.hi) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(dp + ck.lo));
            if (per_thr > 8) asm volatile("prefetch.global.L2 [%0];" ::"l"(dp + min(ck.hi - 1, ck.lo + 8)));
        }
    }
    __syncthreads();
    const int l8 = tid & 7;
    if (sampling) {
        // eight lanes per node: the sibling after it, and whether one before it carries its token
#pragma unroll 1
        for (int c0 = 0; c0 < N; c0 += kWalkThreads / 8) {       // whole warps iterate together
            const int c = c0 + (tid >> 3);
            int nx = MAXN;
            unsigned d = 0;
            if (c >= 1 && c < N) {
                const int pc = sh.t.parent[c], tc = sh.t.tok[c];
                for (int o = 1 + l8; o < N; o += 8) {
                    const bool sib = sh.t.parent[o] == pc;
                    if (sib && o > c) nx = min(nx, o);
                    if (sib && o < c && sh.t.tok[o] == tc) d = 1;
                }
            }
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) {
                nx = min(nx, __shfl_xor_sync(0xffffffffu, nx, off));
                d |= __shfl_xor_sync(0xffffffffu, d, off);
            }
            if (l8 == 0 && c < N) { sh.next_sib[c] = nx < MAXN ? nx : 0; sh.dup[c] = (unsigned char)d; }
        }
    }

    fspad_pdl_wait();                            // from here on the scan's partial results may be read
#pragma unroll 1
    for (int r0 = 0; r0 < N; r0 += kWalkThreads / 8) {           // whole warps iterate together
        const int row = r0 + (tid >> 3), rs = row < N ? row : 0;
        float M; double S; int A;
        if constexpr (INNER) merge_row(args.parts, args.geom, b * N + row, row < N && sh.t.known[rs], kT, l8, M, S, A, nullptr, nullptr);
        else merge_row(args.parts, args.geom, b * N + row, row < N, kT, l8, M, S, A, piece_w[rs], &sh.piece_cnt[rs]);
        if (l8 == 0 && row < N) { sh.rowM[row] = M; sh.rowS[row] = S; sh.t.rowA[row] = A; }
    }
    const double invT = 1.0 / (double)(sampling ? Tf : 1.0f);
    __syncthreads();
    if (sampling && tid < N) {
        if (tid >= 1) {
            sh.cq[tid] = qv;
            sh.cu[tid] = uval;
            sh.cex[tid] = exp_neg(xv, exp_arg(sh.rowM[p], invT), sh.exp_tbl);
        } else {
            sh.ubonus = uval;
        }
        if (sh.first_child[tid] == MAXN) sh.first_child[tid] = 0;
    }
    // the peers' barriers are initialised (every CTA arrived at the top of the kernel)
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    __syncthreads();

    if (!sampling) {
        greedy_walk<INNER>(sh.t, args, b, N, tid, kWalkThreads, true);
        if constexpr (INNER) {
            if (sh.t.last >= 0) {
                const size_t start = (row0 + sh.t.last) * V;
                argmax_row(sh.t, args.given + start, -(int)(start & 3), V, tid, kWalkThreads);
                __syncthreads();
                if (tid == 0) args.bonus[b] = argmax_of(sh.t.best);
            }
        }
        if (args.kv_cache != nullptr) compact_accepted(args, sh.t, b, 0, 1, tid, kWalkThreads);
        return;   // (rank 0 of the cluster; no peer memory is touched)
    }

    // ---- sampling ----
    const bool cache_ok = args.cache_ok != 0, in_regs = cache_ok && per_thr <= kTile;
    // parked values: [k][thread] (k-th position of each thread's chunk), conflict-free
    unsigned char *node_cache = dyn_smem + (INNER ? 0 : N * kPieceBytes);
    double *se = reinterpret_cast<double *>(node_cache) + tid;
    float *sq = reinterpret_cast<float *>(node_cache + (size_t)per_thr * kWalkThreads * sizeof(double)) + tid;
    int n_exch = 0;                              // exchanges so far
    // Sums of NV values (one or five) over the cluster, in every lane of warp 0 (the other warps' values are not defined).
    // Every CTA performs the same operations on the same values.  The first four of five are summed in groups of eight lanes,
    // one value to a group, after two steps in which a lane passes on the values of the other groups; the fifth by all lanes
    // beside them.  A slot is written again two exchanges later, by peers that have by then received
    // this CTA's next totals, which it sends only after it has read the slot.
    // Warp 0 runs `meanwhile` while the peers' totals are on their way.
    auto exchange = [&](auto &v, auto meanwhile) {
        constexpr int NV = sizeof(v) / sizeof(double);
        constexpr bool kFive = NV == 5;
        static_assert(NV == 1 || kFive, "one value or five");
        constexpr int kGroup = kFive ? 8 : 32;   // lanes that end up with the same value
        const int item = lane / kGroup, sub = lane % kGroup;
        const int par = n_exch & 1;
        const uint32_t phase = (uint32_t)(n_exch >> 1) & 1u;
        ++n_exch;
        double one = v[0], fifth = v[NV - 1];
        if (kFive) {
            const bool up = (lane & 16) != 0, odd = (lane & 8) != 0;
            const double a0 = (up ? v[2 % NV] : v[0]) + __shfl_xor_sync(0xffffffffu, up ? v[0] : v[2 % NV], 16);
            const double a1 = (up ? v[3 % NV] : v[1 % NV]) + __shfl_xor_sync(0xffffffffu, up ? v[1 % NV] : v[3 % NV], 16);
            one = (odd ? a1 : a0) + __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 8);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) fifth += __shfl_xor_sync(0xffffffffu, fifth, off);
            if (lane == 0) sh.warp_v[4][wid] = fifth;
        }
#pragma unroll
        for (int off = kGroup / 2; off > 0; off >>= 1) one += __shfl_xor_sync(0xffffffffu, one, off);
        if (sub == 0) sh.warp_v[item][wid] = one;
        __syncthreads();
        if (wid == 0) {
            one = sub < kWarps ? sh.warp_v[item][sub] : 0.0;
            if (kGroup < kWarps) one += sh.warp_v[item][(sub + kGroup) % kWarps];
            static_assert(kGroup >= kWarps / 2 && kWarps == kMaxCluster, "at most two warp or CTA totals per lane");
#pragma unroll
            for (int off = (kGroup < kWarps ? kGroup : kWarps) / 2; off > 0; off >>= 1) one += __shfl_xor_sync(0xffffffffu, one, off);
            if (!kFive) one = __shfl_sync(0xffffffffu, one, 0);
            const uint32_t bar = smem_addr(&sh.bar[par]);
            if (lane == 0) expect_bytes(bar, C * NV * 8);
            if (sub < C) send_double(smem_addr(&sh.slot[par][item][rank]), bar, sub, one);
            if (kGroup < kMaxCluster && sub + kGroup < C) send_double(smem_addr(&sh.slot[par][item][rank]), bar, sub + kGroup, one);
            if (kFive) {
                fifth = lane < kWarps ? sh.warp_v[4][lane % kWarps] : 0.0;
#pragma unroll
                for (int off = kWarps / 2; off > 0; off >>= 1) fifth += __shfl_xor_sync(0xffffffffu, fifth, off);
                if (lane < C) send_double(smem_addr(&sh.slot[par][4][rank]), bar, lane, fifth);
            }
            meanwhile();
            if (!wait_cluster(bar, phase)) sh.fail = 1;
            __syncwarp();
            one = sub < C ? sh.slot[par][item][sub] : 0.0;
            if (kGroup < kMaxCluster && sub + kGroup < C) one += sh.slot[par][item][(sub + kGroup) % kMaxCluster];
            if (kFive) {
                fifth = lane < C ? sh.slot[par][4][lane % kMaxCluster] : 0.0;
#pragma unroll
                for (int off = kMaxCluster / 2; off > 0; off >>= 1) fifth += __shfl_xor_sync(0xffffffffu, fifth, off);
            }
#pragma unroll
            for (int off = (kGroup < kMaxCluster ? kGroup : kMaxCluster) / 2; off > 0; off >>= 1)
                one += __shfl_xor_sync(0xffffffffu, one, off);
            if (kFive) {
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k % NV] = __shfl_sync(0xffffffffu, one, k * 8);
                v[NV - 1] = __shfl_sync(0xffffffffu, fifth, 0);
            } else {
                v[0] = __shfl_sync(0xffffffffu, one, 0);
            }
        }
    };

    // Thread 0 of every CTA (all on identical data, so all take identical steps) walks ahead through
    // every decision that needs nothing but scalars, and stops only to ask the CTA for a sweep of the
    // current node's rows.
    WalkState w;
    Child nx;                                    // the child to be tested next, fetched ahead
    double fx = 0.0, next_rhs = 0.0;             // weight of the token being rejected; the next test's right side
    double next_D = 0.0, next_invD = 0.0;        // draft mass left when the child under test is rejected too
    auto fetch_child = [&](int c) {
        nx.ch = c;
        nx.next = sh.next_sib[c];
        nx.tok = sh.t.tok[c];
        nx.dup = sh.dup[c];
        nx.ex = sh.cex[c];
        nx.qx = (double)sh.cq[c];
        nx.rq = (double)sh.cu[c] * nx.qx;
    };
    // while a residual's total is on its way: the state, and everything that does not depend on that total
    auto fetch_ahead = [&]() {
        w = sh.state;
        fx = weight(sh.cex[w.ch], (double)sh.cq[w.ch], w.Cp);
        next_D = w.base + sh.later_q[w.ch];
        next_invD = 1.0 / next_D;
        fetch_child(sh.next_sib[w.ch]);          // (node 0 where there is none)
        next_rhs = weight(nx.ex, nx.qx, w.Cp) * (next_D > 0.0 ? next_D : w.D);
    };
    enum { GOT_NOTHING, GOT_SUM, GOT_RESIDUAL };
    int got = GOT_NOTHING;
    double R = 0.0;                              // warp 0: the sum asked for last
    double last_a = 0.0;                         // this thread's sum of weights in the latest residual sweep
    double er[kTile];                            // this thread's chunk of the node's rows, after the first rejection there
    float qr[kTile];
#pragma unroll
    for (int i = 0; i < kTile; ++i) { er[i] = 0.0; qr[i] = 0.f; }

    for (;;) {
        if (tid == 0) {
            int go = -1;                                      // node to be entered
            bool ahead = false;                               // nx and next_rhs hold for the next test
            if (got == GOT_NOTHING) {
                go = 0;
                w.len = 0;
                w.nrem = 0;
            } else if (got == GOT_SUM) {
                w.S = w.U = R;
                w.exact = 1;
            } else {
                // When this was the node's last child, the weights just summed (residual at the new coefficient, the
                // rejected tokens at the weights they keep) are the ones the bonus token is drawn from, thread by thread
                // in the same order: the draw reuses the sums (last_a).
                const double Wt = R + (w.ridx < 0 ? w.F + fx : w.F);
                double frozen = fx;
                if (Wt > 0.0) {
                    w.C = w.Cp;
                    w.U = Wt;
                    ahead = true;
                    sh.bonus_ok = nx.ch > 0 ? 0 : 1;
                } else {
                    frozen = weight(sh.cex[w.ch], (double)sh.cq[w.ch], w.C);   // residual vanished: p is kept
                    if (w.C == 0.0) w.U = w.S;
                }
                if (next_D > 0.0) { w.D = next_D; w.invD = next_invD; }
                if (w.ridx < 0 && w.nrem < MAXN) {
                    sh.rem_tok[w.nrem] = sh.t.tok[w.ch];
                    sh.rem_frozen[w.nrem] = frozen;
                    w.F += frozen;
                    w.nrem++;
                }
                w.ch = nx.ch;
            }
            int req = REQ_DONE;
#pragma unroll 1
            for (;;) {
                if (go >= 0) {
                    sh.t.path[w.len++] = go;
                    w.cur = go;
                    w.S = w.U = sh.rowS[go];
                    w.exact = w.parked = 0;
                    w.C = 0.0; w.D = 1.0; w.invD = 1.0; w.F = 0.0;
                    w.nrem = 0;
                    w.ch = sh.first_child[go];
                    sh.bonus_ok = 0;
                    go = -1;
                }
                if (w.ch == 0 || sh.fail != 0) break;
                if (!ahead) fetch_child(w.ch);
                w.ridx = -1;
                if (w.nrem > 0 && nx.dup)
#pragma unroll 1
                    for (int k = 0; k < w.nrem; ++k) if (sh.rem_tok[k] == nx.tok) w.ridx = k;
                // accept iff r * q_k(x) < p_k(x) with q_k = qx / D and p_k = u / U: compared as
                // r * qx * U < u * D (both normalisers are positive), so no division is needed
                double lhs = nx.rq * w.U, rhs = next_rhs;
                if (!ahead) rhs = weight(nx.ex, nx.qx, w.C) * w.D;
                if (w.ridx >= 0) {
                    lhs = 0.0;
                    rhs = sh.rem_frozen[w.ridx] * w.D;
                }
                ahead = false;
                if (!w.exact) {
                    // the scan's sum of exponentials is trusted only outside a margin around the boundary
                    const double big = fmax(lhs, rhs);
                    if (big > 0.0 && fabs(lhs - rhs) <= kAmbiguous * big) {
                        req = REQ_EXP;                        // exact denominator first
                        break;
                    }
                }
                if (lhs < rhs) {
                    go = nx.ch;
                    continue;
                }
                // rejected: a sweep gives the new residual mass
                w.Cp = fma(w.U, w.invD, w.C);
                req = w.parked ? REQ_RESID : REQ_FUSED;
                break;
            }
            sh.req = req;
            sh.C = req == REQ_DONE ? w.C : w.Cp;
            sh.xnew = nx.tok;
            sh.cur = w.cur;
            sh.S = w.S;
            sh.nrem = w.nrem;
            sh.t.len = w.len;
            sh.parked = w.parked && cache_ok;
            sh.state = w;
        }
        __syncthreads();
        w = WalkState{}; nx = Child{}; fx = next_rhs = next_D = next_invD = 0.0;   // (no register is tied up by the state during the sweeps)
        const int req = sh.req;
        if (req == REQ_DONE) break;                           // uniform
        const int cur = sh.cur, xn = sh.xnew;
        const Row x = lg + (size_t)cur * V;
        const float *q = dp + (size_t)cur * V;
        const Chunk ck = chunk_of((row0 + cur) * V, V, per_cta, per_thr, rank, tid);
        const ExpArg arg = exp_arg(sh.rowM[cur], invT);
        got = GOT_RESIDUAL;
        bool again = req != REQ_FUSED;
        if (req == REQ_FUSED) {
            // first rejection at this node, nothing exact yet (nothing removed, C = S)
            double v[5];
            const double s_scan = sh.S;
            fused_reject_sweep(sh, x, q, se, sq, kWalkThreads, ck, per_thr, cache_ok, arg, s_scan, xn, cur, N, v);
            double tot[5] = {v[0], v[1], v[2], v[3], v[4]};
            auto load_tile = [&]() {                          // (each thread its own values: nothing to wait for)
                if (in_regs) {
#pragma unroll
                    for (int i = 0; i < kTile; ++i) {
                        er[i] = i < per_thr ? se[i * kWalkThreads] : 0.0;
                        qr[i] = i < per_thr ? sq[i * kWalkThreads] : 0.f;
                    }
                }
            };
            exchange(tot, load_tile);
            if (wid > 0) load_tile();
            if (wid == 0) {
                const double s_exact = tot[0];
                R = tot[1] - (s_exact - s_scan) * tot[3];
                if (R < 0.0) R = 0.0;
                if (lane == 0) {
                    sh.state.S = sh.state.Cp = s_exact;
                    sh.state.base = tot[2];
                    sh.state.exact = sh.state.parked = 1;
                    const int c = sh.state.ch;
                    const double Wt = R + weight(sh.cex[c], (double)sh.cq[c], s_exact);
                    sh.sel = !(Wt > 0.0 && kScanRel * tot[4] <= kFusedTol * Wt);
                    sh.C = s_exact;                           // the coefficient of the repeated sweep
                    sh.S_exact = s_exact;
                }
            } else {
                // while warp 0 waits for the peers: for each child of the node, the draft mass of the tokens that only
                // siblings after it carry
                for (int c = tid - 31; c < N; c += kWalkThreads - 32) {
                    if (sh.t.parent[c] != cur) continue;
                    double later = 0.0;
#pragma unroll 1
                    for (int o = sh.next_sib[c]; o > 0; o = sh.next_sib[o])
                        if (!sh.dup[o]) later += (double)sh.cq[o];
                    sh.later_q[c] = later;
                }
            }
            __syncthreads();
            if (wid == 0) fetch_ahead();
            again = sh.sel != 0;
            // this thread's share of that sum (nothing rewrites S_exact before the next first rejection; thread 0 may
            // already be changing the rest of the walk's state)
            if (!again) last_a = v[1] - (sh.S_exact - s_scan) * v[3];
        }
        if (again) {
            const double Cn = sh.C;
            if (req == REQ_EXP) {
                // exact softmax denominator of this node; thread 0 then repeats the test with it
                last_a = sweep_row(MODE_EXP, sh, x, q, se, sq, kWalkThreads, ck, false, arg, 0.0, -1, 0.0, 0.0, nullptr);
                got = GOT_SUM;
            } else if (in_regs) {
                if (xn >= ck.lo && xn < ck.hi) {
#pragma unroll
                    for (int i = 0; i < kTile; ++i) {
                        er[i] = i == xn - ck.lo ? 0.0 : er[i];
                        qr[i] = i == xn - ck.lo ? 0.f : qr[i];
                    }
                }
                last_a = residual_of_tile(er, qr, per_thr, Cn);
            } else if (cache_ok) {
                last_a = parked_sweep(se, sq, kWalkThreads, ck, per_thr, Cn, xn);
            } else {
                last_a = sweep_row(MODE_RESID, sh, x, q, se, sq, kWalkThreads, ck, false, arg, Cn, xn, 0.0, 0.0, nullptr);
            }
            double v[1] = {last_a};
            exchange(v, fetch_ahead);
            R = v[0];
        }
        // no barrier here: only thread 0 touches the walk's state until the next request is published
    }
    if (sh.fail != 0) {
        // a wait ran out: nobody leaves while a peer may still write to its shared memory
        if (tid == 0) fspad_report(args.status, FSPAD_ERR_TIMEOUT);
        cluster.sync();
        return;
    }

    // ---- bonus token: inverse CDF of the current residual at the last node ----
    const int cur = sh.cur;
    const Row x = lg + (size_t)cur * V;
    const float *q = dp + (size_t)cur * V;
    const double c = sh.C;
    // A draw at a node where nothing was rejected (a leaf, typically) is taken from the softmax
    // of the row itself.  The scan left the mass of every piece of the row, accurate to kScanRel:
    // enough to name the piece the target falls into and the mass in front of it.  That piece is
    // then swept with single-precision exponentials - by every CTA on its own, all on the same
    // data with the same arithmetic, so all reach the same verdict and nothing is exchanged - and
    // the token is taken when the target clears both ends of its interval by more than the
    // uncertainty of all the approximations together.  Otherwise, and for every other kind of
    // draw, the cluster sweeps the whole row exactly.
    bool settled = false;
    if constexpr (INNER) {
        if (!sh.t.known[cur]) {                               // (a node without children: nothing was rejected there)
            const Chunk ck = chunk_of((row0 + cur) * V, V, per_cta, per_thr, rank, tid);
            const bool last = tid == kWalkThreads - 1 || ck.hi == V || ck.hi - ck.lo < per_thr || (tid + 1) * per_thr >= per_cta;
            if (!draw_from_row(sh, args.given + (row0 + cur) * V, cache_ok ? sq : nullptr, ck, per_thr, last, rank, C, n_exch & 1,
                               (uint32_t)(n_exch >> 1) & 1u, invT, V, args.bonus + b)) {
                if (tid == 0) fspad_report(args.status, FSPAD_ERR_TIMEOUT);
                cluster.sync();                               // nobody leaves while a peer may still write to its shared memory
                return;
            }
            settled = true;
        }
    }
    const int n_piece = INNER ? 0 : sh.piece_cnt[cur];
    if constexpr (!INNER) if (!sh.bonus_ok && c == 0.0 && sh.nrem == 0 && n_piece > 0) {
        // every warp scans the pieces' masses: prefix of the piece the target falls into
        double cum = lane < n_piece ? piece_w[cur][lane & (kPieceSlots - 1)] : 0.0;
        const double own = cum;
#pragma unroll
        for (int off = 1; off < kPieceSlots; off <<= 1) {
            const double t2 = __shfl_up_sync(0xffffffffu, cum, off);
            if (lane >= off) cum += t2;
        }
        const double Zs = __shfl_sync(0xffffffffu, cum, n_piece - 1), target = (double)sh.ubonus * Zs;
        const int pick = __ffs((int)__ballot_sync(0xffffffffu, lane < n_piece && cum > target)) - 1;
        const double top = __shfl_sync(0xffffffffu, cum, max(pick, 0)), mass = __shfl_sync(0xffffffffu, own, max(pick, 0));
        const double pre = top - mass;
        // error budget: the masses in front of the piece and the total (scan, kScanRel each, doubled
        // for slack) and the single-precision sums inside the piece (argument rounding of the
        // exponential 1.3e-7 per unit of |log2 e_j|, the approximation itself 2.4e-7, the partial sums)
        const double tol = 4.0 * kScanRel * Zs + 4e-6 * mass;
        if (pick >= 0 && target - pre > tol && top - target > tol) {
            int p_lo, p_hi;
            piece_bounds(args.geom, b * N + cur, pick, V, &p_lo, &p_hi);
            const int a_lo = p_lo - (int)(((row0 + cur) * V + p_lo) & 3);       // 16-byte aligned
            const int pt = ((((p_hi - a_lo) + kWalkThreads - 1) / kWalkThreads) + 3) & ~3;
            const int t_lo = min(p_hi, a_lo + tid * pt), t_hi = min(p_hi, t_lo + pt);
            const float Mf = sh.rowM[cur];
            // weights relative to the row maximum, as the table's: e_j = exp2((x_j - max) * log2(e) / T)
            auto e32 = [&](float xv2) {
                float y;
                asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"((xv2 - Mf) * kT));
                return xv2 == -INFINITY ? 0.f : y;
            };
            // (tokens of the piece only: what an aligned group of four holds before p_lo is left out)
            auto in4 = [&](int j) {
                if (j >= p_lo && j + 4 <= t_hi) return __ldg(reinterpret_cast<const float4 *>(x + j));
                const int sh_lo = max(p_lo - j, 0);
                float4 r = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                if (sh_lo <= 0 && j < t_hi) r.x = x[j];
                if (sh_lo <= 1 && j + 1 < t_hi) r.y = x[j + 1];
                if (sh_lo <= 2 && j + 2 < t_hi) r.z = x[j + 2];
                if (sh_lo <= 3 && j + 3 < t_hi) r.w = x[j + 3];
                return r;
            };
            double mine = 0.0;
#pragma unroll 1
            for (int j = t_lo; j < t_hi; j += 4) {
                const float4 xs = in4(j);
                mine += (double)((e32(xs.x) + e32(xs.y)) + (e32(xs.z) + e32(xs.w)));
            }
            double E, total;
            const double P = block_scan(sh, mine, &E, &total);
            const double tgt = target - pre;                  // within the piece
            if (tid == 0) { sh.sel = 0x7fffffff; sh.verdict = 2; }
            __syncthreads();
            if (P > tgt) atomicMin(&sh.sel, tid);
            __syncthreads();
            if (tid == sh.sel) {
                double run = E;
#pragma unroll 1
                for (int j = max(t_lo, p_lo); j < t_hi; ++j) {
                    const double before = run;
                    run += (double)e32(x[j]);
                    if (run > tgt) {
                        if (tgt - before > tol && run - tgt > tol) {
                            sh.verdict = 1;
                            if (rank == 0) args.bonus[b] = j;
                        }
                        break;
                    }
                }
            }
            __syncthreads();
            settled = sh.verdict == 1;                        // uniform over the cluster
        }
    }
    if (rank == 0) {
        if (tid == 0) args.n_acc[b] = sh.t.len;
        int *out_path = args.path + (size_t)b * args.path_stride;
#pragma unroll 1
        for (int i = tid; i < args.path_stride; i += kWalkThreads) out_path[i] = (i < sh.t.len) ? sh.t.path[i] : -1;
    }
    if (!settled) {
        // ---- exact draw over the whole row: every CTA a contiguous slice, every thread a contiguous chunk ----
        const Chunk ck = chunk_of((row0 + cur) * V, V, per_cta, per_thr, rank, tid);
        const ExpArg arg = exp_arg(sh.rowM[cur], invT);
        const bool parked = sh.parked != 0;
        // with nothing rejected at this node (c == 0) the weights are the e_j themselves and the
        // denominator cancels, so no separate exact-sum sweep is needed
        double mine = last_a;
        if (sh.bonus_ok) {
#pragma unroll 1
            for (int k = 0; k < sh.nrem; ++k)
                if (sh.rem_tok[k] >= ck.lo && sh.rem_tok[k] < ck.hi) mine += sh.rem_frozen[k];
        } else {
            mine = sweep_row(MODE_CDF, sh, x, q, se, sq, kWalkThreads, ck, parked, arg, c, -1, 0.0, 0.0, nullptr);
        }
        double E, total;
        const double P = block_scan(sh, mine, &E, &total);
        // the CTA total goes to every CTA of the cluster, as in exchange(); every thread waits for the peers' itself
        const int par = n_exch & 1;
        const uint32_t bar = smem_addr(&sh.bar[par]);
        if (tid == 0) expect_bytes(bar, C * 8);
        if (tid < C) send_double(smem_addr(&sh.slot[par][0][rank]), bar, tid, total);
        if (!wait_cluster_all(sh, bar, (uint32_t)(n_exch >> 1) & 1u)) {
            if (tid == 0) fspad_report(args.status, FSPAD_ERR_TIMEOUT);
            cluster.sync();                                   // nobody leaves while a peer may still write to its shared memory
            return;
        }
        // every warp scans the CTA totals side by side: mass in front of this CTA, whole mass, owner of the target
        double cum = (lane < C) ? sh.slot[par][0][lane & (kMaxCluster - 1)] : 0.0;
#pragma unroll
        for (int off = 1; off < kMaxCluster; off <<= 1) {
            const double t2 = __shfl_up_sync(0xffffffffu, cum, off);
            if (lane >= off) cum += t2;
        }
        const double Z = __shfl_sync(0xffffffffu, cum, C - 1), target = (double)sh.ubonus * Z;
        const double before = __shfl_sync(0xffffffffu, cum, rank > 0 ? rank - 1 : 0);
        const double base = rank > 0 ? before : 0.0;
        const int owner = __ffs((int)__ballot_sync(0xffffffffu, lane < C && cum > target)) - 1;
        if (owner == rank) {
            // the first thread (index order) whose inclusive prefix passes the target owns the draw
            if (tid == 0) sh.sel = 0x7fffffff;
            __syncthreads();
            if (base + P > target) atomicMin(&sh.sel, tid);
            __syncthreads();
            // rounding of the two-level prefix can leave no thread above the target although the
            // CTA total is: the last non-empty chunk then takes the draw
            const bool tail = sh.sel == 0x7fffffff && ck.lo < ck.hi && (tid == kWalkThreads - 1 || ck.hi == V || ck.hi - ck.lo < per_thr ||
                                                                       (tid + 1) * per_thr >= per_cta);
            if (tid == sh.sel || tail) {
                int found = -1;
                sweep_row(MODE_CDF, sh, x, q, se, sq, kWalkThreads, ck, parked, arg, c, -1, base + E, target, &found);
                args.bonus[b] = found < 0 ? min(max(ck.lo, 0), V - 1) : found;
            }
        }
        if (owner < 0 && rank == 0 && tid == 0) args.bonus[b] = 0;   // no positive weight anywhere
    }
    if (args.kv_cache != nullptr) compact_accepted(args, sh.t, b, rank, C, tid, kWalkThreads);   // (the CTAs that do not own the draw are at it meanwhile)
    // every CTA has received every peer's total by now, so each may leave on its own
}

// Self-test of the last wait: a pair of CTAs, of which the second sends nothing.  The first one's wait runs out after `polls`
// polls, all its threads leave the same way, and the kernel ends normally.
struct WaitTestShared {
    double slot;
    unsigned long long bar;
    int fail;
};
__global__ void __launch_bounds__(64) walk_wait_selftest_kernel(int *status, uint32_t polls)
{
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ WaitTestShared sh;
    const int rank = (int)cluster.block_rank();
    const uint32_t bar = smem_addr(&sh.bar);
    if (threadIdx.x == 0) {
        sh.fail = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    cluster.sync();
    if (threadIdx.x == 0) expect_bytes(bar, 8);
    if (rank == 0 && threadIdx.x == 0) send_double(smem_addr(&sh.slot), bar, 1, 1.0);
    if (!wait_cluster_all(sh, bar, 0u, rank == 0 ? polls : kPolls) && threadIdx.x == 0) fspad_report(status, FSPAD_ERR_TIMEOUT);
    cluster.sync();
}

}  // namespace

cudaError_t fspad_launch_walk_wait_selftest(fspad_ctx *ctx, int polls, cudaStream_t st)
{
    ctx->launches++;
    return fspad_launch_opt(false, walk_wait_selftest_kernel, dim3(2), dim3(64), 0, st, 2u, ctx->d_status, (uint32_t)polls);
}

// Shared memory that parks a CTA's slice of a row (as the kernel shares it out): e_j in double, q_j in float.
static size_t walk_parked_bytes(int cluster, int V)
{
    const size_t per_cta = (size_t)((((V + 3 + cluster - 1) / cluster) + 3) & ~3);
    const size_t per_thr = ((per_cta + kWalkThreads - 1) / kWalkThreads + 3) & ~(size_t)3;
    return per_thr * kWalkThreads * (sizeof(double) + sizeof(float));
}

typedef void (*WalkKernel)(const WalkArgs);
static WalkKernel walk_kernel(bool narrow, bool inner)
{
    if (narrow) return inner ? accept_walk_kernel<64, true> : accept_walk_kernel<64, false>;
    return inner ? accept_walk_kernel<FSPAD_MAX_NODES_WIDE, true> : accept_walk_kernel<FSPAD_MAX_NODES_WIDE, false>;
}

// Cluster size of the sampling walk.  Once per context: raise the dynamic shared-memory limit and find
// the largest cluster the device can co-schedule for these kernels: 16 (opt-in), else 8.  Small
// vocabularies do not need the whole cluster.  A cluster's CTAs lie side by side, so fewer fit than the SMs
// would hold: 7 of 16, 11 of 10, 15 of 8.  Where a batch may need more than the 7, clusters of 10 are taken, as long as a thread's
// share of a row can be parked in shared memory.  us a step at 128256 tokens, clusters of 16, 10 and 8: 8 sequences 71, 63, 70; 11 73, 65, 78;
// 16, half of them greedy, 124, 115, 145; 16 sampled 146, 129, 125; 10 at 50257 61, 53, 51.  (Of these only the last two are faster
// with eight, by 3 and 4 %.)
static int walk_cluster_size(fspad_ctx *ctx, int B, int V)
{
    if (ctx->walk_cluster == 0) {
        constexpr int most = kSmemBudget + 64 * kPieceBytes, most_wide = kSmemBudgetWide + FSPAD_MAX_NODES_WIDE * kPieceBytes;
        static_assert(most + sizeof(SharedT<64, true>) <= 227 * 1024 && most_wide + sizeof(SharedT<FSPAD_MAX_NODES_WIDE, true>) <= 227 * 1024,
                      "shared memory of a CTA");
        bool all = true;
        int fit = INT_MAX;
        for (int i = 0; i < 4; ++i) {
            const WalkKernel k = walk_kernel(i & 1, i & 2);
            const int bytes = i & 1 ? most : most_wide;
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
            if (!all || cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) { all = false; continue; }
            cudaLaunchConfig_t probe = {};
            probe.gridDim = dim3(kMaxCluster);
            probe.blockDim = dim3(kWalkThreads);
            probe.dynamicSmemBytes = bytes;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = kMaxCluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
            probe.attrs = at; probe.numAttrs = 1;
            int n = 0;
            all = cudaOccupancyMaxActiveClusters(&n, k, &probe) == cudaSuccess && n >= 1;
            fit = n < fit ? n : fit;
        }
        ctx->walk_cluster = all ? kMaxCluster : 8;
        ctx->walk_fit = all ? fit : ctx->sm_count / 8;
        (void)cudaGetLastError();
    }
    int cluster = ctx->walk_cluster;
    while (cluster > 1 && (V + cluster - 1) / cluster < 2048) cluster >>= 1;
    if (cluster == kMaxCluster && B > ctx->walk_fit &&
        walk_parked_bytes(kSmallerCluster, V) <= (size_t)(ctx->cfg.max_nodes <= 64 ? kSmemBudget : kSmemBudgetWide))
        cluster = kSmallerCluster;
    return cluster;
}

int fspad_walk_ctas(fspad_ctx *ctx, int B, int V) { return B * walk_cluster_size(ctx, B, V); }

cudaError_t fspad_launch_accept_walk(fspad_ctx *ctx, const float *logits, const float *draft,
                                     const int *tokens, const int *parent, const float *temperature,
                                     const float *uniforms, const FspadStatsGeom &geom, int N, int B, int V,
                                     int *path, int *n_acc, int *bonus, cudaStream_t st, FspadWalkCompact kv, bool draft_far)
{
    if (B == 0) return cudaSuccess;
    WalkArgs a;
    a.kv_cache = reinterpret_cast<uint4 *>(kv.cache); a.kv_prefix = kv.prefix_len; a.kv_new_len = kv.new_len;
    a.kv_layers = ctx->cfg.n_layers; a.kv_B = B; a.kv_H = ctx->cfg.n_kv_heads; a.kv_max_len = ctx->cfg.max_len;
    a.logits = geom.stage != nullptr ? geom.stage : logits; a.given = logits; a.draft = draft; a.temperature = temperature; a.uniforms = uniforms;
    a.tokens = tokens; a.parent = parent;
    a.parts = ctx->st_part; a.geom = geom;
    a.N = N; a.V = V; a.path_stride = ctx->cfg.max_nodes; a.cache_ok = 0; a.draft_far = draft_far ? 1 : 0; a.B = B; a.sampled_first = 0;
    a.path = path; a.n_acc = n_acc; a.bonus = bonus; a.status = ctx->d_status;

    const bool inner = geom.parent != nullptr;
    ctx->launches++;
    if (draft == nullptr || uniforms == nullptr) {               // every sequence greedy
        // a row that the scan has left out is looked at by a cluster of eight, 64 KB a CTA at 128256 tokens
        unsigned c = inner ? (unsigned)kGreedyCluster : 1u;
        while (c > 1 && (V + (int)c - 1) / (int)c < 4096) c >>= 1;
        return fspad_launch(N <= 64 ? inner ? accept_greedy_kernel<64, true> : accept_greedy_kernel<64, false>
                                    : inner ? accept_greedy_kernel<FSPAD_MAX_NODES_WIDE, true> : accept_greedy_kernel<FSPAD_MAX_NODES_WIDE, false>,
                            dim3((unsigned)B * c), dim3(kWalkThreads), 0, st, inner ? c : 0u, a);
    }
    const int cluster = walk_cluster_size(ctx, B, V);
    // (16 sequences, half of them sampling: the walk 75 -> 68 us beside the attention, the step 202 -> 199; with one wave of clusters
    // the order does not matter and the look at the temperatures is saved)
    a.sampled_first = B > 1 && B <= kWalkThreads && (B * cluster > ctx->sm_count || cluster == kSmallerCluster);     // (one thread looks at each sequence)
    const size_t need = walk_parked_bytes(cluster, V);
    size_t smem = inner ? 0 : (size_t)N * kPieceBytes;
    if (need <= (size_t)(N <= 64 ? kSmemBudget : kSmemBudgetWide)) { smem += need; a.cache_ok = 1; }
    // trees of up to 64 nodes and of up to FSPAD_MAX_NODES_WIDE nodes are two instances of the kernel
    return fspad_launch(walk_kernel(N <= 64, inner), dim3((unsigned)(B * cluster)), dim3(kWalkThreads), smem, st, (unsigned)cluster, a);
}
