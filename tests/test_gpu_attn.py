"""CUDA tree-masked attention (through the C ABI) against the fp64 oracle.
Bound (bf16 inputs, fp32 accumulate, bf16 output): max abs error <= 1e-2,
mean abs error <= 1e-3."""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_15562_b200 import binding, synth
from tests import helpers

pytestmark = pytest.mark.gpu

W = synth.WORKLOADS
MAX_ABS, MEAN_ABS = 1e-2, 1e-3


def _shrink_values(inp, factor_log2=2):
    """Divide every V entry by 2**factor_log2 (exact in bf16).  With only a handful of
    keys the outputs are as large as single N(0,1) draws (|v| up to 4), where bf16
    output rounding alone (2^-9 relative) reaches the absolute bound; the bound is
    stated for outputs of order one and below, as the named workloads produce."""
    for arr in (inp.v_cache, inp.tree_v):
        nz = arr & 0x7FFF != 0
        arr[nz] -= np.uint16(factor_log2 << 7)


def _check(inp, seqs=None, alias_cache=False):
    ctx = helpers.make_ctx(inp)
    d = helpers.upload_attn(inp)
    out = ctx.tree_attn(d["q"], d["k_cache"], d["v_cache"], None if alias_cache else d["tree_k"],
                        None if alias_cache else d["tree_v"], d["parent"], d["prefix_len"])
    ctx.check()
    seqs = list(range(inp.q.shape[0])) if seqs is None else seqs
    for b in seqs:
        sl = slice(b, b + 1)
        ref = oracle.tree_attn(inp.q[sl], inp.k_cache[sl], inp.v_cache[sl], inp.tree_k[sl], inp.tree_v[sl],
                               inp.parent[sl], inp.prefix_len[sl])
        mx, mean = helpers.attn_errors(out[sl], ref)
        assert mx <= MAX_ABS and mean <= MEAN_ABS, (b, mx, mean)
    return out


@pytest.mark.parametrize("hq,hkv", [(4, 4), (8, 2), (16, 2)])
@pytest.mark.parametrize("prefix", [0, 1, 63, 64, 65, 200, 333])
def test_small_shapes_ragged_tails(hq, hkv, prefix):
    w = synth.scaled(W["llama3_8b_2k"], n_q_heads=hq, n_kv_heads=hkv, prefix=(prefix, prefix), n_nodes=19,
                     depth=4, branch=3, vocab=16)
    inp = synth.generate(w, 0, with_accept=False)
    if prefix < 64:
        _shrink_values(inp)
    _check(inp)


@pytest.mark.parametrize("tree,n", [("chain", 7), ("star", 33), ("bfs", 26), ("pruned", 64), ("chain", 1)])
def test_tree_shapes(tree, n):
    w = synth.scaled(W["llama3_8b_2k"], n_q_heads=8, n_kv_heads=2, prefix=(150, 150), n_nodes=n, tree=tree,
                     depth=6 if n > 1 else 1, branch=4, vocab=16)
    _check(synth.generate(w, 1, with_accept=False))


def test_tree_rows_taken_from_cache_when_no_tree_arrays():
    w = synth.scaled(W["llama3_8b_2k"], n_q_heads=8, n_kv_heads=2, prefix=(100, 300), batch=3, n_nodes=20,
                     depth=4, branch=3, vocab=16, temperatures=(0.0,) * 3)
    inp = synth.generate(w, 2, with_accept=False)
    a = _check(inp, alias_cache=False)
    b = _check(inp, alias_cache=True)
    assert torch.equal(a, b)


@pytest.mark.parametrize("prefix", [0, 100, 128, 200, 256, 300, 511, 640, 1000])
def test_every_chunk_count_per_cta(prefix):
    """80 kv heads fill the GPU with one key range per head, so a CTA walks all of the sequence's
    1 .. 9 chunks itself: every wrap state of a lone CTA's three-deep K/V ring and of the parity-doubled
    score barriers, with the gathered boundary chunk first, in the middle of the ring, or last."""
    w = synth.scaled(W["llama3_8b_2k"], n_q_heads=80, n_kv_heads=80, prefix=(prefix, prefix), n_nodes=9,
                     depth=3, branch=3, vocab=16)
    inp = synth.generate(w, 3, with_accept=False)
    if prefix < 64:
        _shrink_values(inp)
    _check(inp)


@pytest.mark.parametrize("hq,hkv,n", [(16, 2, 60), (24, 2, 33), (12, 4, 64)])
def test_gqa_row_tiles(hq, hkv, n):
    """Rows per kv head beyond one 128-row tile: 480 (four tiles, the last ragged), 396, 192."""
    w = synth.scaled(W["llama3_8b_2k"], n_q_heads=hq, n_kv_heads=hkv, prefix=(700, 700), n_nodes=n,
                     depth=6, branch=4, vocab=16)
    _check(synth.generate(w, 4, with_accept=False))


def test_batched_ragged_small():
    w = synth.scaled(W["batch16_ragged"], batch=5, prefix=(10, 700), temperatures=(0.0,) * 5, vocab=16)
    _check(synth.generate(w, 0, with_accept=False))


@pytest.mark.parametrize("lengths", ["equal", "pairs", "descending", "ascending"])
def test_more_ctas_than_sms_sequences_taken_longest_first(lengths):
    """24 sequences x 8 kv heads x 2 row tiles = 384 CTAs: more than the SMs, so the kernel hands the sequences
    out longest first by a rank it computes from the lengths on the device.  Equal lengths (every rank decided by
    the index), equal pairs, and lengths already in either order must all give every sequence its own output."""
    B = 24
    L = {"equal": np.full(B, 200), "pairs": 60 + 40 * (np.arange(B) // 2), "descending": 600 - 20 * np.arange(B),
         "ascending": 50 + 20 * np.arange(B)}[lengths].astype(np.int32)
    w = synth.scaled(W["batch16_ragged"], batch=B, prefix=(int(L.max()), int(L.max())), temperatures=(0.0,) * B,
                     vocab=16, n_layers=1)
    inp = synth.generate(w, 3, with_accept=False)
    inp.prefix_len[:] = L                       # the cache is generated for the longest; shorter ones use its head
    _check(inp)


@pytest.mark.parametrize("n_nodes,group", [(33, 4), (64, 4), (60, 5), (60, 8), (130, 3), (200, 2)])
@pytest.mark.parametrize("alias", [False, True])
def test_row_tiles_in_pairs(n_nodes, group, alias):
    """Calls whose row tiles alone fill the SMs run on pairs of CTAs: 2 to 4 row tiles of a kv head (an empty half of the last pair
    with 3), the boundary between the tiles inside a node's heads, 1 .. 12 chunks a sequence (every wrap state of the pair's
    five-deep ring), the gathered boundary chunks first, in the middle and last; tree rows apart and in the cache."""
    B = 12
    L = np.array([0, 100, 128, 129, 383, 500, 640, 700, 900, 1151, 1280, 1400], np.int32)
    w = synth.scaled(W["batch16_ragged"], batch=B, n_q_heads=8 * group, n_kv_heads=8, n_nodes=n_nodes, depth=6, branch=12,
                     prefix=(int(L.max()), int(L.max())), temperatures=(0.0,) * B, vocab=16, n_layers=1)
    inp = synth.generate(w, n_nodes, with_accept=False)
    if inp.parent.shape[1] != n_nodes:
        pytest.skip("the expansion gave fewer nodes")
    inp.prefix_len[:] = L
    _shrink_values(inp)                         # (the first sequences have few keys)
    if alias:
        for b in range(B):
            inp.k_cache[b, :, L[b]:L[b] + n_nodes] = inp.tree_k[b]
            inp.v_cache[b, :, L[b]:L[b] + n_nodes] = inp.tree_v[b]
    _check(inp, alias_cache=alias)


def test_equal_value_rows_reproduce_exactly():
    """All V rows equal to one bf16 row: the softmax weights sum to 1, so the output is that row."""
    w = synth.scaled(W["llama3_8b_2k"], prefix=(300, 300), vocab=16)
    inp = synth.generate(w, 0, with_accept=False)
    row = inp.v_cache[0, 0, 0].copy()
    inp.v_cache[...] = row
    inp.tree_v[...] = row
    ctx = helpers.make_ctx(inp)
    d = helpers.upload_attn(inp)
    out = ctx.tree_attn(d["q"], d["k_cache"], d["v_cache"], d["tree_k"], d["tree_v"], d["parent"], d["prefix_len"])
    ref = synth.bf16_bits_to_f32(row).astype(np.float64)
    err = np.abs(out.float().cpu().numpy() - ref)
    assert err.max() <= 2.0 ** -7 * np.abs(ref).max()


@pytest.mark.parametrize("name", ["tiny_greedy", "llama3_8b_2k", "vicuna_33b_4k_greedy"])
def test_full_size_configs(name):
    _check(synth.generate(W[name], 0, with_accept=False))


def test_full_size_llama3_70b_8k_sampled_heads():
    """Full launch configuration; the oracle checks every output of the sequence
    (64 query heads x 60 nodes) - about ten seconds of fp64 CPU work."""
    _check(synth.generate(W["llama3_70b_8k"], 0, with_accept=False))


def test_full_size_batch16_every_sequence():
    """The batched ragged workload in its full launch configuration; the oracle checks every
    output of all sixteen sequences (about a minute of fp64 CPU work on all host cores)."""
    inp = synth.generate(W["batch16_ragged"], 0, with_accept=False)
    _check(inp)


def test_prefix_out_of_range_is_reported():
    w = synth.scaled(W["llama3_8b_2k"], n_q_heads=8, n_kv_heads=2, prefix=(50, 50), n_nodes=10, depth=3,
                     branch=3, vocab=16)
    inp = synth.generate(w, 0, with_accept=False)
    ctx = helpers.make_ctx(inp)
    d = helpers.upload_attn(inp)
    bad = torch.tensor([inp.max_len], dtype=torch.int32, device="cuda")
    ctx.tree_attn(d["q"], d["k_cache"], d["v_cache"], d["tree_k"], d["tree_v"], d["parent"], bad)
    assert ctx.status() == -5
    with pytest.raises(binding.FspadError) as e:          # a pointer that is not 16-byte aligned
        ctx.tree_attn(d["q"], d["k_cache"], d["v_cache"], d["tree_k"], d["tree_v"].flatten()[1:], d["parent"],
                      d["prefix_len"])
    assert e.value.code == -2


@pytest.mark.parametrize("hq,hkv,prefix,n", [
    (2, 2, 128, 60),       # the prefix ends with a chunk: the tree's chunk holds nothing but tree rows and padding
    (6, 2, 127, 1),        # Q gathered (three heads a group); the last chunk is exactly full
    (14, 2, 129, 60),      # Q gathered, rows of a tile begin within a node
    (2, 1, 255, 129),      # three chunks with tree rows, one of them full
    (4, 1, 127, 256),      # three chunks with tree rows, the first with a single one
    (120, 40, 300, 60),    # pairs of CTAs, Q gathered
    (80, 40, 383, 65),     # pairs of CTAs, the last chunk is exactly full
])
def test_rows_behind_the_tree_may_hold_anything(hq, hkv, prefix, n):
    """Chunks with tree rows or padding are gathered, the others copied by TMA: what lies behind the last tree row (or, where the
    tree rows come apart, behind the prefix) is NaN here and must not get into any sum."""
    w = synth.scaled(W["llama3_8b_2k"], n_q_heads=hq, n_kv_heads=hkv, prefix=(prefix, prefix), n_nodes=n,
                     tree="pruned" if n > 1 else "chain", depth=8 if n > 1 else 1, branch=10, vocab=16)
    inp = synth.generate(w, 3, with_accept=False)
    for alias in (True, False):
        for plane in (inp.k_cache, inp.v_cache):
            plane[:, :, prefix + (n if alias else 0):] = 0x7FC0
        _check(inp, alias_cache=alias)


@pytest.mark.parametrize("hq,hkv,n,batch,prefix", [
    (32, 8, 60, 2, 300),       # lone CTAs: 240 rows, half of a warp's rows do not exist
    (32, 8, 60, 2, 768),       # a chunk of tree rows alone
    (16, 2, 33, 3, 700),       # 264 rows
    (8, 8, 19, 2, 200),        # one head a group: 19 rows
    (24, 8, 33, 2, 300),       # Q gathered
    (32, 8, 60, 12, 300),      # pairs of CTAs
])
def test_a_sequence_does_not_depend_on_its_neighbours_queries(hq, hkv, n, batch, prefix):
    """Rows of a tile past a sequence's last node hold the next sequence's queries: whatever these are, the sequence's own
    output stays the same bit for bit."""
    w = synth.scaled(W["batch16_ragged"], batch=batch, n_q_heads=hq, n_kv_heads=hkv, prefix=(prefix, prefix), n_nodes=n, depth=6,
                     branch=10, vocab=16, temperatures=(0.0,) * batch, n_layers=1)
    inp = synth.generate(w, 5, with_accept=False)
    ctx = helpers.make_ctx(inp)
    d = helpers.upload_attn(inp)

    def call(q):
        out = ctx.tree_attn(q, d["k_cache"], d["v_cache"], d["tree_k"], d["tree_v"], d["parent"], d["prefix_len"])
        ctx.check()
        return out

    ref = call(d["q"])
    for fill in (float("nan"), float("inf"), None):
        q = d["q"].clone()
        q[1::2] = q[1::2] * 64 if fill is None else fill
        assert torch.equal(call(q)[0::2], ref[0::2]), fill


@pytest.mark.parametrize("batch,n", [(1, 60), (12, 60), (1, 200)])
def test_the_largest_weight_is_exact_behind_chunks_of_tree_rows(batch, n):
    """The first 128 keys are the prefix, one of them 5 to 7.7 in log2 above the tree's keys (whose V is 0), the others 25 and more
    below.  Taken against the largest score its weight is exactly 1, and the result is its V row over a sum kept in 32 bits: what is
    left is the output's own rounding, half a unit in the last place of bf16, and a few of 32 bits."""
    hq, hkv, L, j = 32, 8, 128, 10
    w = synth.scaled(W["batch16_ragged"], batch=batch, n_q_heads=hq, n_kv_heads=hkv, prefix=(L, L), n_nodes=n, depth=8, branch=10,
                     vocab=16, temperatures=(0.0,) * batch, n_layers=1)
    inp = synth.generate(w, 7, with_accept=False)
    n = inp.parent.shape[1]
    rng = np.random.default_rng(3)
    bf = lambda x: (np.ascontiguousarray(x, np.float32).view(np.uint32) >> 16).astype(np.uint16)      # (exact values only)
    inp.q[...] = 0
    inp.q[..., 0] = bf(40 + 0.25 * rng.integers(0, 80, inp.q.shape[:-1]))
    inp.k_cache[...] = 0
    inp.k_cache[:, :, :L, 0] = bf([-4.0])
    inp.k_cache[:, :, j, 0] = bf([1.0])
    inp.tree_k[...] = 0
    inp.tree_v[...] = 0
    ctx = helpers.make_ctx(inp)
    d = helpers.upload_attn(inp)
    out = ctx.tree_attn(d["q"], d["k_cache"], d["v_cache"], d["tree_k"], d["tree_v"], d["parent"], d["prefix_len"])
    ctx.check()
    ref = oracle.tree_attn(inp.q, inp.k_cache, inp.v_cache, inp.tree_k, inp.tree_v, inp.parent, inp.prefix_len)
    err = np.abs(out.float().cpu().numpy().astype(np.float64) - ref)
    half_ulp = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(ref), 2.0 ** -20))) - 8)
    assert (err <= half_ulp + 4e-6).all(), (err / half_ulp).max()
