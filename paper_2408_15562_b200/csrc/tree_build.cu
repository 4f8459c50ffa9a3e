// Dynamic token tree, final stage (paper, Section "Preliminaries", last
// paragraph: every draft step is cut to its top-k, each token carries the joint
// probability of its path, and one top-k over all tokens after the draft phase
// gives a valid tree of bounded size; Section "Performance on Fewer Candidate
// Tokens" halves both budgets).
//
// One CTA per sequence, one thread per candidate (at most 1024, level by level, joint
// log-probabilities that never grow along a path).  The N - 1 largest are found
// without sorting: the value of the last one is settled bit by bit from the top (one
// CTA-wide count per bit, over as soon as exactly N - 1 candidates reach what is settled),
// and among candidates that equal it the lower indices are kept, so parents stay
// ahead of their children.  The thread of a kept candidate walks
// its parent chain (depth, and that every ancestor was kept), takes its
// breadth-first position by counting the kept candidates that come before it in
// (depth, index) order, and writes the flattened tree the verification step
// consumes, with (optionally) each node's ancestor-or-self mask.  Integer work throughout; no arithmetic on the
// probabilities.  What bounds it is latency: with the candidates sorted by a 1024-entry network first, 410 candidates
// took 7.6 us, now 4.7.
#include "common.cuh"
#include "sort_key.cuh"

namespace {

__global__ void __launch_bounds__(FSPAD_MAX_CANDIDATES)
tree_build_kernel(const int *__restrict__ cand_parent, const int *__restrict__ cand_token,
                  const float *__restrict__ cand_logp, const int *__restrict__ root_token, int C, int N,
                  int *__restrict__ parent_out, int *__restrict__ token_out, int *__restrict__ cand_out,
                  unsigned long long *__restrict__ anc_out, int *__restrict__ n_out, int *__restrict__ status)
{
    __shared__ short s_par[FSPAD_MAX_CANDIDATES];                // parent candidate (-1: child of the root)
    __shared__ short s_node[FSPAD_MAX_CANDIDATES];               // node number of a kept candidate, else -1
    __shared__ int s_eq[FSPAD_MAX_CANDIDATES / 32], s_kept[FSPAD_MAX_CANDIDATES / 32];   // per warp: ties, kept candidates
    __shared__ unsigned char s_kd[FSPAD_MAX_NODES];              // depths of the kept candidates, in index order
    fspad_pdl_trigger();
    fspad_pdl_wait();
    const int b = blockIdx.x, c = threadIdx.x, lane = c & 31, warp = c >> 5;
    const bool mine = c < C;
    bool bad = false;
    uint32_t key = 0u;                                           // order-preserving image of the value
    int p = -1, tok = 0;
    if (mine) {
        key = fspad_orderable(cand_logp[(size_t)b * C + c] + 0.0f);      // (-0.0 counts as +0.0)
        p = cand_parent[(size_t)b * C + c];
        tok = cand_token[(size_t)b * C + c];
        if (p < -1 || p >= c) { bad = true; p = -1; }
        s_par[c] = (short)p;
    }
    const int want = min(N - 1, C);
    // the largest t that `want` candidates reach
    uint32_t t = 0u;
    bool exact = want == C;
    for (int bit = 31; bit >= 0 && !exact; --bit) {
        const uint32_t with = t | (1u << bit);
        const int n = __syncthreads_count(mine && key >= with);
        if (n >= want) { t = with; exact = n == want; }
    }
    bool keep = mine && key >= t && want > 0;
    if (!exact) {
        // more candidates equal t than there is room for: the lower indices are kept
        const unsigned eq = __ballot_sync(0xffffffffu, mine && key == t);
        if (lane == 0) s_eq[warp] = __popc(eq);
        const int above = __syncthreads_count(mine && key > t);
        if (keep && key == t) {
            int before = __popc(eq & ((1u << lane) - 1u));
            for (int w = 0; w < warp; ++w) before += s_eq[w];
            keep = above + before < want;
        }
    }
    const unsigned km = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) s_kept[warp] = __popc(km);
    if (mine) s_node[c] = keep ? 0 : -1;                         // kept (number follows)
    __syncthreads();
    int slot = 0, depth = 0;
    if (keep) {
        slot = __popc(km & ((1u << lane) - 1u));                 // kept candidates before this one
        for (int w = 0; w < warp; ++w) slot += s_kept[w];
        for (int a = c; a >= 0; a = s_par[a]) {                  // indices strictly decrease: the walk ends
            if (s_node[a] < 0) bad = true;                       // an ancestor was not kept
            ++depth;
        }
        s_kd[slot] = (unsigned char)min(depth, 255);
    }
    __syncthreads();
    int pos = 1;
    if (keep) {
        depth = min(depth, 255);
        for (int o = 0; o < want; ++o) {
            const int od = s_kd[o];
            pos += (od < depth || (od == depth && o < slot)) ? 1 : 0;
        }
        s_node[c] = (short)pos;
    }
    __syncthreads();
    int *po = parent_out + (size_t)b * N, *to = token_out + (size_t)b * N, *co = cand_out + (size_t)b * N;
    if (keep) {
        po[pos] = (p < 0) ? 0 : (int)s_node[p];
        to[pos] = tok;
        co[pos] = c;
        if (anc_out) {                                           // the node, its ancestors and the root
            unsigned long long mask = 1ull;
            for (int a = c; a >= 0; a = s_par[a])
                if (s_node[a] > 0) mask |= 1ull << s_node[a];
            anc_out[(size_t)b * N + pos] = mask;
        }
    }
    if (c == 0) {
        po[0] = -1; to[0] = root_token[b]; co[0] = -1; n_out[b] = want + 1;
        if (anc_out) anc_out[(size_t)b * N] = 1ull;
    }
    for (int i = want + 1 + c; i < N; i += blockDim.x) {
        po[i] = -1; to[i] = -1; co[i] = -1;
        if (anc_out) anc_out[(size_t)b * N + i] = 0ull;
    }
    if (bad) fspad_report(status, FSPAD_ERR_BAD_TREE);
}

}  // namespace

cudaError_t fspad_launch_tree_build(fspad_ctx *ctx, const int *cand_parent, const int *cand_token,
                                    const float *cand_logp, const int *root_token, int n_cand, int n_nodes,
                                    int B, int *parent_out, int *token_out, int *cand_out,
                                    unsigned long long *anc_out, int *n_out, cudaStream_t st)
{
    if (B == 0) return cudaSuccess;
    ctx->launches++;
    return fspad_launch(tree_build_kernel, dim3(B), dim3((n_cand + 31) / 32 * 32), 0, st, 0, cand_parent, cand_token, cand_logp,
                        root_token, n_cand, n_nodes, parent_out, token_out, cand_out, anc_out, n_out, ctx->d_status);
}
