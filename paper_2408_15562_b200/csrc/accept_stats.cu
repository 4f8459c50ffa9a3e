// Per-node vocabulary scan: the first stage of lossless tree acceptance.
// One streaming pass over every row of the target logits gives the row
// maximum, its lowest index and the sum of exponentials at the row's
// temperature.  The strict comparison of the paper's verification stage
// (Section "Preliminaries") needs the target's result for every tree node;
// this kernel produces all of them in one HBM-bound sweep.  The walk that follows an acceptance's scan reads only
// rows it comes to, and of a node without children only one, its last: on large arrays the scan of an acceptance
// goes by the trees and leaves those nodes' rows out (accept_stats_inner_kernel).
//
// Layout: logits [rows][V] fp32, viewed as one flat array that is cut into
// equal contiguous ranges, one per CTA (1024 threads per SM in a single wave:
// CTAs of 128 threads for a small array, of 256 otherwise), so the load is
// balanced whatever rows and V are.  Where the sizes allow, the ranges are cut at
// the rows; otherwise a range may cross row boundaries and runs the reductions
// once per row it touches.  Each (row, CTA) piece yields one partial (max, argmax, sum).
// A thread works in batches of four 128-bit loads, with the next batch already
// in flight: it takes the maximum of the 16 values in registers, rescales its
// running sum once and adds the 16 exponentials: no per-element branch.  Partials are merged per
// row by whoever needs them (the acceptance walk for the rows it visits, or
// the small merge kernel behind fspad_accept_stats).
#include <atomic>

#include "common.cuh"

namespace {

constexpr int kThreads = FSPAD_STATS_THREADS;   // 256; small arrays are scanned by CTAs of half that
constexpr int kDeep = 4;                  // load units per batch per thread (two batches in flight)
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct Acc {
    float m, s;
    int a;
};

__device__ __forceinline__ void acc_merge(Acc &p, float om, float os, float k)
{
    const float mn = fmaxf(p.m, om);
    const float sp = (p.m == -INFINITY) ? 0.f : p.s * ex2((p.m - mn) * k);
    const float so = (om == -INFINITY) ? 0.f : os * ex2((om - mn) * k);
    p.m = mn;
    p.s = sp + so;
}

// one load unit: a float4 (UNIT == 4) or a float (UNIT == 1)
template <int UNIT> struct Unit;
template <> struct Unit<4> {
    typedef float4 T;
    static __device__ __forceinline__ T pad() { return make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY); }
    static __device__ __forceinline__ float vmax(const T &v) { return fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)); }
    static __device__ __forceinline__ float vsum(const T &v, float m, float k)
    {
        return (ex2((v.x - m) * k) + ex2((v.y - m) * k)) + (ex2((v.z - m) * k) + ex2((v.w - m) * k));
    }
    // lowest position inside the unit equal to bm, or keep `a`
    static __device__ __forceinline__ int first_eq(const T &v, float bm, int j, int a)
    {
        if (v.w == bm) a = j + 3;
        if (v.z == bm) a = j + 2;
        if (v.y == bm) a = j + 1;
        if (v.x == bm) a = j;
        return a;
    }
};
template <> struct Unit<1> {
    typedef float T;
    static __device__ __forceinline__ T pad() { return -INFINITY; }
    static __device__ __forceinline__ float vmax(const T &v) { return v; }
    static __device__ __forceinline__ float vsum(const T &v, float m, float k) { return ex2((v - m) * k); }
    static __device__ __forceinline__ int first_eq(const T &v, float bm, int j, int a) { return v == bm ? j : a; }
};

// SHIFT: rows of a length that is no multiple of 4, one piece of one row per CTA; position j of unit i is 4 i + j - (up to three),
// aligned loads all the same (read float by float, 520 rows of 50257 took 39 us, now 23)
template <int UNIT, bool SHIFT, int kThreads>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads)
accept_stats_kernel(const float *__restrict__ logits, const float *__restrict__ temperature,
                    int rows_per_seq, int V, const FspadStatsGeom g, FspadStatsPart *__restrict__ parts)
{
    typedef typename Unit<UNIT>::T U;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int piece = SHIFT ? (int)blockIdx.x % g.per_row : 0;
    const long long lo = SHIFT ? ((long long)blockIdx.x / g.per_row) * g.upr + piece * g.chunk : (long long)blockIdx.x * g.chunk;
    const long long hi = SHIFT ? lo - piece * g.chunk + min((long long)g.upr, (piece + 1) * g.chunk) : min(g.total, lo + g.chunk);
    __shared__ Acc wacc[kThreads / 32];
    __shared__ float s_bmax;
    __shared__ int s_barg;
    // Wait first, then let the successor start: a kernel that follows this one in the stream (the
    // acceptance walk) can then rely on everything queued before the scan having completed, and may
    // read the caller's arrays, which the scan never writes, while the scan is still running.
    fspad_pdl_wait();
    fspad_pdl_trigger();

    long long seg_lo = lo;
    while (seg_lo < hi) {
        const int row = (int)(seg_lo / g.upr);
        const long long row_lo = (long long)row * g.upr;
        const long long seg_hi = min(hi, row_lo + g.upr);
        const int n = (int)(seg_hi - seg_lo);                 // units in this piece of the row
        const int off = (int)(seg_lo - row_lo);               // position of the piece inside the row
        const U *px = reinterpret_cast<const U *>(logits) + seg_lo;
        const float *xrow = logits + (size_t)row * V;         // SHIFT: unit i of this piece is xrow[j0 + 4 i ..], empty outside the row
        const int j0 = SHIFT ? 4 * off - (int)(((size_t)row * V) & 3) : 0;
        // units [i0, i1) lie inside the row; a first and a last one that do not are thread 0's and thread 32's to begin with.
        // (A row has room for one unit more than its tokens may fill, so a piece can begin past the row's end: it is empty.)
        const int i0 = SHIFT && j0 < 0 ? 1 : 0, i1 = SHIFT ? min(n, (V - j0) >> 2) : n;
        auto fetch = [&](int i) -> U {
            if constexpr (SHIFT) return __ldg(reinterpret_cast<const U *>(xrow + j0) + i);
            else return __ldg(px + i);
        };
        float T = temperature ? temperature[row / rows_per_seq] : 1.0f;
        if (!(T > 0.0f)) T = 1.0f;
        const float k = kLog2e / T;

        // software pipeline: the next batch of loads is in flight while this one is reduced
        Acc p{-INFINITY, 0.f, 0x7fffffff};
        int edge = -1;                                        // SHIFT: this thread's unit at an end of the row
        if constexpr (SHIFT) {
            if (tid == 0 && i0 > 0) edge = 0;
            if (tid == 32 && i1 >= i0 && i1 < n) edge = i1;   // (i1 < i0: the row is one unit, thread 0's, or the piece is empty)
            if (edge >= 0) {
                const U v = fspad_edge4(xrow, j0 + 4 * edge, V, -INFINITY);
                p.m = Unit<UNIT>::vmax(v);
                p.s = p.m == -INFINITY ? 0.f : Unit<UNIT>::vsum(v, p.m, k);
                p.a = -1;
            }
        }
        U cur[kDeep], nxt[kDeep];
#pragma unroll
        for (int u = 0; u < kDeep; ++u) {
            const int i = u * kThreads + tid;
            cur[u] = (i >= i0 && i < i1) ? fetch(i) : Unit<UNIT>::pad();
        }
        for (int base = 0; base < n; base += kThreads * kDeep) {
            const int nb = base + kThreads * kDeep;
            if (nb < n) {
#pragma unroll
                for (int u = 0; u < kDeep; ++u) {
                    const int i = nb + u * kThreads + tid;
                    nxt[u] = (i < i1) ? fetch(i) : Unit<UNIT>::pad();
                }
            }
            float bm = Unit<UNIT>::vmax(cur[0]);
#pragma unroll
            for (int u = 1; u < kDeep; ++u) bm = fmaxf(bm, Unit<UNIT>::vmax(cur[u]));
            if (bm > p.m || (SHIFT && p.a < 0 && bm == p.m)) {        // (an equal value in a batch comes before the row's last unit)
                // only the batch is remembered; the position inside it is looked up once, at the
                // end, by the threads that hold the block's maximum
                p.s = (p.m == -INFINITY) ? 0.f : p.s * ex2((p.m - bm) * k);
                p.m = bm;
                p.a = base;
            }
            if (p.m != -INFINITY) {
                float s0 = 0.f;
#pragma unroll
                for (int u = 0; u < kDeep; ++u) s0 += Unit<UNIT>::vsum(cur[u], p.m, k);
                p.s += s0;
            }
            if (nb < n) {
#pragma unroll
                for (int u = 0; u < kDeep; ++u) cur[u] = nxt[u];
            }
        }
        // block reduction of (m, s); then the lowest index of the block's maximum
        const float my_m = p.m;
        const int my_base = p.a;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float om = __shfl_xor_sync(0xffffffffu, p.m, o);
            const float os = __shfl_xor_sync(0xffffffffu, p.s, o);
            acc_merge(p, om, os, k);
        }
        if (lane == 0) wacc[wid] = p;
        if (tid == 0) s_barg = 0x7fffffff;
        __syncthreads();
        if (wid == 0) {
            Acc q = (lane < kThreads / 32) ? wacc[lane] : Acc{-INFINITY, 0.f, 0};
#pragma unroll
            for (int o = kThreads / 64; o > 0; o >>= 1) {
                const float om = __shfl_xor_sync(0xffffffffu, q.m, o);
                const float os = __shfl_xor_sync(0xffffffffu, q.s, o);
                acc_merge(q, om, os, k);
            }
            if (lane == 0) { wacc[0] = q; s_bmax = q.m; }
        }
        __syncthreads();
        const float bmax = s_bmax;
        if (my_m == bmax && bmax != -INFINITY) {
            // this thread's batch `my_base` holds the maximum: fetch it again (cache hit) and scan it
            int a = 0x7fffffff;
            if constexpr (SHIFT)                              // (only a batch with a larger value has displaced it: it may hold the maximum too)
                if (edge >= 0) a = Unit<UNIT>::first_eq(fspad_edge4(xrow, j0 + 4 * edge, V, -INFINITY), bmax, j0 + 4 * edge, a);
            int b = 0x7fffffff;
#pragma unroll
            for (int u = kDeep - 1; u >= 0; --u) {
                const int i = my_base + u * kThreads + tid;
                if (my_base >= 0 && i >= i0 && i < i1) b = Unit<UNIT>::first_eq(fetch(i), bmax, SHIFT ? j0 + 4 * i : (off + i) * UNIT, b);
            }
            atomicMin(&s_barg, min(a, b));
        }
        __syncthreads();
        if (tid == 0) {
            const int slot = SHIFT ? piece : (int)(blockIdx.x - (int)(row_lo / g.chunk));
            FspadStatsPart out;
            out.m = wacc[0].m; out.s = wacc[0].s; out.a = s_barg; out.pad = 0;
            parts[(size_t)row * g.slots + slot] = out;
        }
        __syncthreads();
        seg_lo = seg_hi;
    }
}

// The largest of a warp's values.
static __device__ __forceinline__ float warp_max(float v)
{
    float m;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
    return m;
}

// Positions j .. j + 3 of a row, from memory this thread has written itself.  (Past the first-level cache: the other half of a line's
// 32 bytes may be another CTA's and not there yet.)
static __device__ __noinline__ float4 own4(const float *x, int j, int V)
{
    float4 r = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (j >= 0 && j < V) r.x = __ldcg(x + j);
    if (j + 1 >= 0 && j + 1 < V) r.y = __ldcg(x + j + 1);
    if (j + 2 >= 0 && j + 2 < V) r.z = __ldcg(x + j + 2);
    if (j + 3 >= 0 && j + 3 < V) r.w = __ldcg(x + j + 3);
    return r;
}

// The same scan over the rows of the nodes that have children (a quarter of a 60-node tree's): the walk stops at a node without
// children at most once, at its end, and looks at that row itself.  A parent that is no lower node counts as the root, as in the
// walk.  Two ways of finding the rows:
//   SHARED = false  few rows: a CTA for every piece of every row, gridDim.x pieces by gridDim.y rows, and those of a row that is
//                   nobody's parent leave at once
//   SHARED = true   every CTA marks the nodes that are somebody's parent, a bit a row, and every warp numbers them for itself.  A row is
//                   cut into as many pieces as give every CTA one, up to g.per_row; where that leaves two fifths of the CTAs idle, or
//                   there are more rows than CTAs, each takes an equal share of the rows laid end to end instead, the first loads of
//                   a run being in flight while the one before it is reduced
// Bound by HBM where the rows are many, else by the chain of launch, parents, loads and reduction: parents marked 0.7 us after the start,
// piece known 1.3 to 1.6, loads back 2.2 to 2.7, partials written 3.3 to 3.8 (60 nodes of 50257 and 128256 tokens).  One piece to a CTA wherever
// that fills three fifths of them, because a second run costs a reduction (1.1 us) more than the idle CTAs do.  Acceptance alone, greedy, us
// from a graph, all rows / shares with pairs of (maximum, sum) merged step by step / this: 60 x 32000 eight times 18.0 / 15.3 / 11.7, 25 x 32001
// six times 8.2 / 13.0 / 9.8, 60 x 128256 16 times 83.5 / 33.8 / 32.3, a chain of 60 x 128256 12.3 / 15.6 / 12.3.
//   The run of a row that a CTA takes is reduced as a whole.  Of a share its result goes to slot 0 if the run begins the row, else to the
// one behind the stretch of `wide` units it starts in: every share is at least that long, so no two meet.  Slots without a run of their
// own are empty.
// STAGE: the logits are in host memory, and the rows read are left at g.stage for the walk.
template <bool SHARED, bool STAGE>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads)
accept_stats_inner_kernel(const float *__restrict__ logits, const float *__restrict__ temperature, int N, int rows, int V,
                          const FspadStatsGeom g, int wide, FspadStatsPart *__restrict__ parts)
{
    typedef Unit<4> U4;
    constexpr int kStep = kThreads * kDeep, kWords = SHARED ? FSPAD_INNER_MAX_ROWS / 32 : 1, kList = SHARED ? FSPAD_INNER_LIST : 1;
    constexpr int kWarps = kThreads / 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, upr = g.upr;
    __shared__ unsigned word[kWords];            // SHARED: a bit a row, set where it is somebody's parent
    __shared__ int list[kList];                  // the rows of the CTA's share
    __shared__ float2 wacc[2][kWarps];           // (by the parity of the run, as s_at: what one run leaves is read while the next begins)
    __shared__ int s_at[2];
    static_assert(kWords <= kThreads, "a word to a thread");
    if constexpr (SHARED)
        if (tid < kWords) word[tid] = 0u;
    if (tid < 2) s_at[tid] = 0x7fffffff;
    __syncthreads();
    struct Run {
        const float4 *x;                         // its units off .. off + n - 1 of the row, from token j0 on (up to three in front of the row)
        int row, off, j0, n, n_load;             // n_load: how many of them can be loaded whole (the rest has no token or ends the array)
        float k;
    };
    auto open = [&](int row, int off, int n) {
        Run q;
        q.row = row;
        q.off = off;
        q.n = n;
        q.j0 = 4 * off - (int)(((size_t)row * V) & 3);
        q.x = reinterpret_cast<const float4 *>(logits + (size_t)row * V + q.j0);
        q.n_load = fspad_whole_units(rows, row, V, q.j0, n);
        const float T = temperature ? temperature[(unsigned)row / (unsigned)N] : 1.0f;
        q.k = kLog2e / (T > 0.0f ? T : 1.0f);
        return q;
    };
    // A unit that reaches out of its row is loaded whole, but for one that ends the array, and clipped when it is used: the threads
    // that have one do not hold up their warp's loads.
    auto batch = [&](float4 (&v)[kDeep], const Run &q, int base) {
#pragma unroll
        for (int u = 0; u < kDeep; ++u) {
            const int i = base + u * kThreads + tid;
            v[u] = i < q.n_load ? __ldg(q.x + i) : U4::pad();
        }
    };
    fspad_pdl_wait();                            // (the order of the two: see the scan of all rows)
    fspad_pdl_trigger();
    unsigned hi = 0;                             // end of the share, in units of the rows laid end to end (below 2^31)
    int first = 0, last = 0;                     // the rows it touches, by number
    int piece = (int)blockIdx.x, pieces = g.per_row;   // pieces: 0 where the rows are shared out laid end to end
    Run q;
    if constexpr (SHARED) {
        int c = (int)((unsigned)tid % (unsigned)N);
        const int step = (int)((unsigned)kThreads % (unsigned)N);
#pragma unroll 4
        for (int i = tid; i < rows; i += kThreads) {
            const int p = __ldg(g.parent + i), r = i - c + ((unsigned)p < (unsigned)c ? p : 0);
            atomicOr(&word[r >> 5], 1u << (r & 31));
            c += step;
            c -= c >= N ? N : 0;
        }
        __syncthreads();
        // the marked rows, numbered by every warp for itself: a lane has `wpl` words of marks, `incl` rows up to its last
        const int wpl = (rows + 1023) >> 10;
        int cnt = 0;
#pragma unroll 1
        for (int u = 0; u < wpl; ++u) cnt += __popc(word[lane * wpl + u]);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int n_inner = __shfl_sync(0xffffffffu, incl, 31);
        auto row_of = [&](int number) {          // (whole warps)
            const int owner = __ffs((int)__ballot_sync(0xffffffffu, incl > number)) - 1;
            int nth = number - __shfl_sync(0xffffffffu, incl - cnt, owner), w = owner * wpl;
            unsigned bits = word[w];
#pragma unroll 1
            for (int c = __popc(bits); nth >= c; c = __popc(bits)) {
                nth -= c;
                bits = word[++w];
            }
            const bool is = ((bits >> lane) & 1u) != 0u && __popc(bits & ((1u << lane) - 1u)) == nth;
            return 32 * w + __ffs((int)__ballot_sync(0xffffffffu, is)) - 1;
        };
        const unsigned ctas = gridDim.x;
        pieces = min(g.per_row, (int)(ctas / (unsigned)n_inner));
        if (pieces < g.per_row && 10u * (unsigned)(pieces * n_inner) < 6u * ctas) pieces = 0;
        int off, n;
        if (pieces > 0) {
            const int chunk = (int)((unsigned)(upr + pieces - 1) / (unsigned)pieces);
            first = last = (int)((unsigned)blockIdx.x / (unsigned)pieces);
            if (first >= n_inner) return;
            piece = (int)blockIdx.x - first * pieces;
            off = piece * chunk;
            n = min(chunk, upr - off);
        } else {
            const unsigned total = (unsigned)(n_inner * upr), each = max((total + ctas - 1) / ctas, (unsigned)wide);
            const unsigned lo = min(total, blockIdx.x * each);
            hi = min(total, lo + each);
            if (lo >= hi) return;
            first = (int)(lo / (unsigned)upr);
            last = (int)((hi - 1) / (unsigned)upr);
            off = (int)(lo - (unsigned)(first * upr));
            n = min(upr - off, (int)(hi - lo));
            for (int r = first + wid; r <= last; r += kWarps) {
                const int row = row_of(r);
                if (lane == 0) list[r - first] = row;
            }
            __syncthreads();
        }
        q = open(row_of(first), off, n);
    } else {
        const int row = (int)blockIdx.y, root = row - (int)((unsigned)row % (unsigned)N);
        bool inner = row == root;
        for (int c = tid + 1; c < N; c += kThreads) {
            const int p = __ldg(g.parent + root + c);
            inner |= p == row - root && p < c;
        }
        const int off = piece * (int)g.chunk;
        if (!__syncthreads_or(inner)) return;
        q = open(row, off, min((int)g.chunk, upr - off));          // (n below 1: the piece is empty)
    }
    float4 cur[kDeep], nxt[kDeep];
    batch(cur, q, 0);
    for (int r = first, par = 0;; par ^= 1) {
        Run following = q;
        Acc p{-INFINITY, 0.f, 0x7fffffff};
        for (int base = 0; base < q.n; base += kStep) {
            if (base + kStep < q.n) {
                batch(nxt, q, base + kStep);
            } else if (SHARED && r < last) {
                following = open(list[r + 1 - first], 0, min(upr, (int)(hi - (unsigned)((r + 1) * upr))));
                batch(nxt, following, 0);
            }
            if (g.shift && ((base == 0 && q.j0 < 0) || q.j0 + 4 * (base + kStep) > V)) {         // (the row's first or last batch)
#pragma unroll
                for (int u = 0; u < kDeep; ++u) {
                    const int i = base + u * kThreads + tid, j = q.j0 + 4 * i;
                    if (i < q.n && j < V && (j < 0 || j + 4 > V)) {
                        if (i >= q.n_load) {
                            cur[u] = fspad_edge4(logits + (size_t)q.row * V, j, V, -INFINITY);
                        } else {
                            if (j < 0) cur[u].x = -INFINITY;
                            if (j < -1 || j + 1 >= V) cur[u].y = -INFINITY;
                            if (j < -2 || j + 2 >= V) cur[u].z = -INFINITY;
                            if (j + 3 >= V) cur[u].w = -INFINITY;
                        }
                    }
                }
            }
            if constexpr (STAGE) {
                float *to = g.stage + (size_t)q.row * V;
#pragma unroll
                for (int u = 0; u < kDeep; ++u) {
                    const int i = base + u * kThreads + tid, j = q.j0 + 4 * i;
                    if (i < q.n && j >= 0 && j + 4 <= V) {
                        *reinterpret_cast<float4 *>(to + j) = cur[u];
                    } else if (i < q.n) {
                        if (j >= 0 && j < V) to[j] = cur[u].x;
                        if (j + 1 >= 0 && j + 1 < V) to[j + 1] = cur[u].y;
                        if (j + 2 >= 0 && j + 2 < V) to[j + 2] = cur[u].z;
                        if (j + 3 >= 0 && j + 3 < V) to[j + 3] = cur[u].w;
                    }
                }
            }
            float bm = U4::vmax(cur[0]);
#pragma unroll
            for (int u = 1; u < kDeep; ++u) bm = fmaxf(bm, U4::vmax(cur[u]));
            if (bm > p.m) {
                p.s = (p.m == -INFINITY) ? 0.f : p.s * ex2((p.m - bm) * q.k);
                p.m = bm;
                p.a = base;
            }
            if (p.m != -INFINITY) {
                float s0 = 0.f;
#pragma unroll
                for (int u = 0; u < kDeep; ++u) s0 += U4::vsum(cur[u], p.m, q.k);
                p.s += s0;
            }
#pragma unroll
            for (int u = 0; u < kDeep; ++u) cur[u] = nxt[u];
        }
        // The run's maximum first, by warps and then by all warps' results, then the sums, brought to it once each: half the time of
        // merging pairs of (maximum, sum) step by step.
        const float wm = warp_max(p.m);
        float ws = p.m == -INFINITY ? 0.f : p.s * ex2((p.m - wm) * q.k);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ws += __shfl_xor_sync(0xffffffffu, ws, o);
        if (lane == 0) wacc[par][wid] = make_float2(wm, ws);
        __syncthreads();
        float bmax = wacc[par][0].x;
#pragma unroll
        for (int w = 1; w < kWarps; ++w) bmax = fmaxf(bmax, wacc[par][w].x);
        if (p.m == bmax && bmax != -INFINITY) {
            // the batch at p.a holds the maximum: fetch it again (cache hit) and look for it
            const float *from = (STAGE ? g.stage : logits) + (size_t)q.row * V;      // (what this thread has stored there itself)
            float4 v[kDeep];
#pragma unroll
            for (int u = 0; u < kDeep; ++u) {
                const int i = p.a + u * kThreads + tid, j = q.j0 + 4 * i;
                v[u] = U4::pad();
                if (i < q.n) v[u] = STAGE ? own4(from, j, V) : fspad_load4(from, j, V, -INFINITY);
            }
            int at = 0x7fffffff;
#pragma unroll
            for (int u = kDeep - 1; u >= 0; --u) at = U4::first_eq(v[u], bmax, q.j0 + 4 * (p.a + u * kThreads + tid), at);
            atomicMin(&s_at[par], at);
        }
        __syncthreads();
        int own = piece, stop = piece + 1;
        if (SHARED && pieces > 0 && stop == pieces) stop = g.per_row;
        if (SHARED && pieces == 0) {
            const int end = q.off + q.n;
            own = q.off == 0 ? 0 : 1 + q.off / wide;
            stop = end >= upr ? g.per_row : 1 + end / wide;
        }
        if (tid >= own && tid < stop) {
            FspadStatsPart out;
            out.m = -INFINITY; out.s = 0.f; out.a = 0x7fffffff; out.pad = 0;
            if (tid == own) {
                out.m = bmax;
                out.a = s_at[par];
                s_at[par] = 0x7fffffff;                          // (for the run after next)
#pragma unroll
                for (int w = 0; w < kWarps; ++w) {
                    const float2 t = wacc[par][w];
                    out.s += t.x == -INFINITY ? 0.f : t.y * ex2((t.x - bmax) * q.k);
                }
            }
            parts[(size_t)q.row * g.slots + tid] = out;
        }
        if (!SHARED || r == last) break;
        ++r;
        q = following;
    }
}

// rows -> (max, sum, argmax) from the partials; one warp per row
__global__ void __launch_bounds__(128)
accept_stats_merge_kernel(const FspadStatsPart *__restrict__ parts, const FspadStatsGeom g,
                          const float *__restrict__ temperature, int rows, int rows_per_seq,
                          float *__restrict__ row_max, double *__restrict__ row_sum, int *__restrict__ row_arg)
{
    fspad_pdl_trigger();
    fspad_pdl_wait();
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (row >= rows) return;
    float T = temperature ? temperature[row / rows_per_seq] : 1.0f;
    if (!(T > 0.0f)) T = 1.0f;
    float M;
    double S;
    int A;
    fspad_stats_merge_warp(parts, g, row, kLog2e / T, lane, M, S, A);
    if (lane == 0) {
        row_max[row] = M;
        row_sum[row] = S;
        row_arg[row] = A;
    }
}

template <int kT>
cudaError_t launch_partials_t(const float *logits, const float *temperature, int rows_per_seq, int V, const FspadStatsGeom &g,
                              FspadStatsPart *parts, cudaStream_t st, bool pdl)
{
    const dim3 grid(g.n_cta), block(kT);
    if (g.shift) return fspad_launch_opt(pdl, accept_stats_kernel<4, true, kT>, grid, block, 0, st, 0, logits, temperature, rows_per_seq, V, g, parts);
    if (g.unit == 4) return fspad_launch_opt(pdl, accept_stats_kernel<4, false, kT>, grid, block, 0, st, 0, logits, temperature, rows_per_seq, V, g, parts);
    return fspad_launch_opt(pdl, accept_stats_kernel<1, false, kT>, grid, block, 0, st, 0, logits, temperature, rows_per_seq, V, g, parts);
}
cudaError_t launch_partials(const float *logits, const float *temperature, int rows_per_seq, int V,
                            const FspadStatsGeom &g, FspadStatsPart *parts, cudaStream_t st, bool pdl = true)
{
    return g.threads == kThreads / 2 ? launch_partials_t<kThreads / 2>(logits, temperature, rows_per_seq, V, g, parts, st, pdl)
                                     : launch_partials_t<kThreads>(logits, temperature, rows_per_seq, V, g, parts, st, pdl);
}

}  // namespace

cudaError_t fspad_launch_stats_partials(fspad_ctx *ctx, const float *logits, const float *temperature,
                                        int rows, int rows_per_seq, int V, FspadStatsGeom *geom,
                                        cudaStream_t st, bool pdl, int sms)
{
    const bool aligned = (reinterpret_cast<uintptr_t>(logits) & 15) == 0;
    if (sms <= 0 || sms > ctx->sm_count) sms = ctx->sm_count;
    if (geom->parent != nullptr && aligned && rows % rows_per_seq == 0 && fspad_scan_inner_fits(sms, rows, V)) {
        *geom = fspad_stats_geom_inner(sms, rows, V, ctx->stats_slots, geom->parent, geom->stage);
        const FspadStatsGeom &g = *geom;
        const int wide = (g.upr + g.per_row - 2) / (g.per_row - 1);
        ctx->launches++;
        const bool pieces = g.n_cta == rows * g.per_row, stage = g.stage != nullptr;
        return fspad_launch_opt(pdl, pieces ? stage ? accept_stats_inner_kernel<false, true> : accept_stats_inner_kernel<false, false>
                                            : stage ? accept_stats_inner_kernel<true, true> : accept_stats_inner_kernel<true, false>,
                                pieces ? dim3(g.per_row, rows) : dim3(g.n_cta), dim3(kThreads), 0, st, 0, logits, temperature, rows_per_seq,
                                rows, V, g, wide, ctx->st_part);
    }
    if (geom->stage != nullptr) return cudaErrorInvalidValue;        // (the caller looks first)
    *geom = fspad_stats_geom(sms, rows, V, aligned, ctx->stats_slots, true);
    ctx->launches++;
    return launch_partials(logits, temperature, rows_per_seq, V, *geom, ctx->st_part, st, pdl);
}

cudaError_t fspad_launch_accept_stats(fspad_ctx *ctx, const float *logits, const float *temperature,
                                      int rows, int rows_per_seq, int V, float *row_max,
                                      double *row_sum, int *row_arg, cudaStream_t st)
{
    if (rows == 0) return cudaSuccess;
    FspadStatsGeom g;
    cudaError_t e = fspad_launch_stats_partials(ctx, logits, temperature, rows, rows_per_seq, V, &g, st);
    if (e != cudaSuccess) return e;
    ctx->launches++;
    return fspad_launch(accept_stats_merge_kernel, dim3((rows + 3) / 4), dim3(128), 0, st, 0,
                        (const FspadStatsPart *)ctx->st_part, g, temperature, rows, rows_per_seq, row_max, row_sum,
                        row_arg);
}

// ---------------------------------------------------------------------------
// The same scan for callers that must not allocate device memory.
//
// Some hosts of this library run where cudaMalloc is off limits: inside a
// serving process whose memory pool owns the whole device and forbids outside
// allocations, or in a start-up path where an allocation (which synchronises
// the device) is not acceptable.  They cannot create an fspad_ctx, so this entry
// point needs none: the per-CTA partials live in the fixed device array below,
// which every GPU that loads the library holds until the process exits (0.5 MB).
// ---------------------------------------------------------------------------
namespace {

constexpr int kNoAllocMaxRows = 1024;     // e.g. 16 sequences x 64 nodes
constexpr int kNoAllocSlots = 32;         // partial slots per row
constexpr size_t kNaBytes = (size_t)kNoAllocMaxRows * kNoAllocSlots * sizeof(FspadStatsPart);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

constexpr int kMaxDevices = 64;
struct NoAllocDevice {
    std::atomic<unsigned char *> scratch;   // device address of g_noalloc_scratch on this device (NULL = not set up)
    int sm_count;                            // written before `scratch` is published
};
NoAllocDevice g_na_dev[kMaxDevices];

}  // namespace

extern "C" int fspad_accept_stats_noalloc(const float *logits, const float *temperature, int rows,
                                          int rows_per_seq, int vocab, float *row_max, double *row_sum,
                                          int32_t *row_arg, void *stream)
{
    if (!logits || !row_max || !row_sum || !row_arg) return FSPAD_ERR_NULL;
    if (rows < 0 || rows_per_seq < 1 || vocab < 1) return FSPAD_ERR_SHAPE;
    if (rows > kNoAllocMaxRows) return FSPAD_ERR_TOO_LARGE;
    if (rows == 0) return FSPAD_OK;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return FSPAD_ERR_CUDA;
    NoAllocDevice &nd = g_na_dev[dev];
    unsigned char *scratch = nd.scratch.load(std::memory_order_acquire);
    if (!scratch) {
        // First call on this device: g_noalloc_scratch is only a host-side handle here, the
        // kernels need the array's address in this device's memory.  Host threads that race on
        // this first call all compute the same two values; the address is published last, so a
        // thread that sees it also sees the SM count.
        void *p = nullptr;
        int sms = 0;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return FSPAD_ERR_CUDA;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
            return FSPAD_ERR_CUDA;
        nd.sm_count = sms;
        scratch = static_cast<unsigned char *>(p);
        nd.scratch.store(scratch, std::memory_order_release);
    }
    cudaStream_t st = fspad_stream(stream);
    const bool aligned = (reinterpret_cast<uintptr_t>(logits) & 15) == 0;
    const FspadStatsGeom g = fspad_stats_geom(nd.sm_count, rows, vocab, aligned, kNoAllocSlots);
    FspadStatsPart *parts = reinterpret_cast<FspadStatsPart *>(scratch);
    // every slot the merge reads is rewritten by this call's first kernel, so the contents an
    // earlier call left in the shared array never need clearing
    if (launch_partials(logits, temperature, rows_per_seq, vocab, g, parts, st) != cudaSuccess) return FSPAD_ERR_CUDA;
    return fspad_launch(accept_stats_merge_kernel, dim3((rows + 3) / 4), dim3(128), 0, st, 0,
                        (const FspadStatsPart *)parts, g, temperature, rows, rows_per_seq, row_max, row_sum,
                        (int *)row_arg) == cudaSuccess ? FSPAD_OK : FSPAD_ERR_CUDA;
}
