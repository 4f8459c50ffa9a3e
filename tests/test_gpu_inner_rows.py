"""Acceptance on arrays that are scanned by the trees: the rows of nodes without children have no scan results, and the walk looks
at the one it ends in itself.  Against the oracle, bit-exact (the 1e-6 band excepted and counted)."""
import numpy as np
import pytest
import torch

import oracle

from paper_2408_15562_b200 import binding, synth
from tests import helpers
from tests.test_gpu_accept import _run

pytestmark = pytest.mark.gpu

W = synth.WORKLOADS


def _parity(inp, allow_near=1):
    path, n_acc, bonus = _run(inp)
    hard, near, msgs = helpers.compare_accept(inp, path, n_acc, bonus)
    assert hard == 0, msgs
    assert near <= allow_near, msgs
    return path, n_acc, bonus


def _leaf_ends(inp, path, n_acc):
    return sum(int(path[b, n_acc[b] - 1]) not in set(inp.parent[b].tolist()) for b in range(len(n_acc)))


# one CTA per sequence up to clusters of 16; rows that start on and off 16-byte boundaries; trees on either side of 64 nodes;
# fewer and more items than CTAs; up to nine rows
@pytest.mark.parametrize("vocab,nodes,batch", [(4000, 64, 30), (4099, 80, 30), (8192, 200, 6), (16381, 130, 5), (32000, 60, 5), (50257, 60, 4), (128256, 33, 3),
                                                (128256, 60, 1), (5003, 64, 30), (8193, 9, 1), (8196, 3, 3), (50257, 1, 9), (128256, 4, 2)])
@pytest.mark.parametrize("mode", ["greedy", "sample", "mixed"])
def test_rows_without_children(vocab, nodes, batch, mode):
    temps = {"greedy": (0.0,) * 16, "sample": (1.0, 0.7) * 8, "mixed": (0.0, 1.0, 0.6) * 6}[mode]
    temps = (temps * 2)[:batch]
    at_leaf = 0
    for variant in range(3):
        w = synth.scaled(W["llama3_8b_2k"], batch=batch, vocab=vocab, n_nodes=nodes, depth=3, branch=8 if nodes <= 64 else 16,
                         temperatures=temps, prefix=(8, 8))
        if nodes == 1:
            w = synth.scaled(w, depth=1)
        inp = synth.generate(w, variant, with_attention=False)
        assert inp.parent.size * vocab >= 9.5e6 or (nodes >= 32 and vocab % 4 == 0 and inp.parent.size * vocab >= 5e6) or \
            (inp.parent.size < 10 and vocab > 8192)                                                        # (else every row is scanned)
        path, n_acc, _ = _parity(inp)
        at_leaf += _leaf_ends(inp, path, n_acc)
    assert at_leaf > 0 or batch == 1 or inp.parent.size < 10


@pytest.mark.parametrize("temps", [(0.0, 0.0), (1.0, 0.0), (0.3, 2.0)])
@pytest.mark.parametrize("where", [0, 1, 31998, 49999, 50256])
def test_ends_of_the_row(temps, where):
    """A star whose only child is certain to be accepted; the leaf's mass lies at one token, also twice (the lower index counts), or
    nowhere."""
    w = synth.scaled(W["tiny_greedy"], batch=2, vocab=50257, n_nodes=100, tree="star", temperatures=temps, prefix=(8, 8))
    inp = synth.generate(w, 0, with_attention=False)
    inp.target_logits[:, 0] = -np.inf
    inp.target_logits[0, 0, inp.draft_tokens[0, 1]] = 1.0
    inp.target_logits[1, 0, inp.draft_tokens[1, 1]] = 1.0
    for b in range(2):
        inp.target_logits[b, 1] = -np.inf
        if b == 0:
            inp.target_logits[b, 1, where] = -3.0
        else:
            inp.target_logits[b, 1, where] = 4.0
            inp.target_logits[b, 1, 50256] = 4.0
    path, n_acc, bonus = _parity(inp, allow_near=0)
    assert n_acc.tolist() == [2, 2] and bonus[0] == where
    if temps[1] == 0.0:
        assert bonus[1] == where
    inp.target_logits[:, 1] = -np.inf
    _, _, bonus = _run(inp)
    assert bonus.tolist() == [0, 0]


def test_zeros_of_either_sign_and_chains():
    w = synth.scaled(W["tiny_greedy"], batch=1, vocab=65536, n_nodes=80, tree="star", temperatures=(0.0,), prefix=(8, 8))
    inp = synth.generate(w, 0, with_attention=False)
    inp.target_logits[:] = -1.0
    inp.target_logits[0, 0, inp.draft_tokens[0, 5]] = 1.0
    inp.target_logits[0, :, 40000] = 0.0
    inp.target_logits[0, :, 123] = -0.0
    path, n_acc, bonus = _parity(inp, allow_near=0)
    assert path[0, 1] in (1, 2, 3, 4, 5) and bonus[0] == 123
    for temps in ((0.0, 0.0), (1.0, 1.0)):
        w = synth.scaled(W["tiny_greedy"], batch=2, vocab=32000, n_nodes=80, tree="chain", temperatures=temps, prefix=(8, 8))
        for variant in range(3):
            _parity(synth.generate(w, variant, with_attention=False))


@pytest.mark.parametrize("vocab,nodes,batch", [(1000, 9, 1), (3001, 70, 3), (4099, 256, 2), (50257, 40, 2)])
@pytest.mark.parametrize("mode", ["greedy", "mixed"])
def test_logits_read_where_they_are(vocab, nodes, batch, mode):
    """The host entry point on logits that the kernels read over the link (pinned, on a 16-byte boundary) and on ones that are copied
    (pinned off the boundary; pageable): the oracle's acceptance each time, also in a second call with other logits in the same memory."""
    w = synth.scaled(W["llama3_8b_2k"], batch=batch, prefix=(40, 300), n_nodes=nodes, depth=4, branch=16, vocab=vocab,
                     temperatures=((0.0,) * 3 if mode == "greedy" else (1.0, 0.0, 0.7))[:batch])
    inps = [synth.generate(w, v) for v in (3, 4)]
    ctx = helpers.make_ctx(inps[0], n_layers=1)
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()   # noqa: E731
    flat = torch.from_numpy(inps[0].target_logits)
    for where in (flat.clone().pin_memory(), torch.empty(flat.numel() + 4).pin_memory()[1:1 + flat.numel()].view(flat.shape), flat.clone()):
        for inp in inps:
            where.copy_(torch.from_numpy(inp.target_logits))
            sampling = inp.draft_probs is not None
            cache = binding.bf16_tensor(synth.make_cache(inp, 1))
            out = torch.empty(inp.q.shape, dtype=torch.bfloat16).pin_memory()
            path = torch.empty(inp.parent.shape, dtype=torch.int32)
            n, bonus, new_len = (torch.empty((batch,), dtype=torch.int32) for _ in range(3))
            ctx.verify_step_host(cache, *(binding.bf16_tensor(a, "cpu").pin_memory() for a in (inp.q, inp.tree_k, inp.tree_v)),
                                 pin(inp.parent), pin(inp.prefix_len), where, pin(inp.draft_probs) if sampling else None,
                                 pin(inp.draft_tokens), pin(inp.temperature), pin(inp.uniforms) if sampling else None, out, path, n, bonus,
                                 new_len)
            hard, near, msgs = helpers.compare_accept(inp, path.numpy(), n.numpy(), bonus.numpy())
            assert hard == 0 and near == 0, msgs
            assert np.array_equal(new_len.numpy(), inp.prefix_len + n.numpy())


@pytest.mark.parametrize("vocab,nodes,batch", [(32753, 20, 7), (32753, 20, 8), (50257, 12, 9), (128256, 10, 12), (151936, 66, 8)])
@pytest.mark.parametrize("mode", ["sample", "mixed"])
def test_batches_of_more_clusters_than_fit_at_once(vocab, nodes, batch, mode):
    """Clusters of 16 up to seven sequences, of ten beyond (but where a slice of the row would not fit into shared memory), sampling
    sequences first: every number of rejections, draws at leaves and inside."""
    temps = ((1.0, 0.7) * 8 if mode == "sample" else (0.0, 1.0, 0.6, 1.0) * 4)[:batch]
    for variant in range(2):
        w = synth.scaled(W["llama3_8b_2k"], batch=batch, vocab=vocab, n_nodes=nodes, depth=3, branch=9 if nodes <= 64 else 12,
                         temperatures=temps, prefix=(8, 8))
        _parity(synth.generate(w, variant, with_attention=False))


@pytest.mark.parametrize("hq,hkv,prefix,nodes,batch,vocab,temps", [
    (32, 8, 1500, 60, 1, 50257, (1.0,)),                 # several key ranges behind the walk in one stream, from a graph forked behind the scan
    (52, 52, 700, 52, 1, 50257, (1.0,)),                 # an attention on most SMs: one stream either way
    (32, 8, 700, 40, 2, 50257, (0.8, 0.0)),
    (32, 8, 300, 24, 9, 32753, (1.0, 0.0, 0.7) * 3),     # more clusters than fit at once: forked
])
def test_step_called_and_captured(hq, hkv, prefix, nodes, batch, vocab, temps):
    """The step behind a scan by the trees: called, and replayed from a graph twice, it gives the same bits, and the acceptance and the
    compacted cache are those of the separate calls."""
    w = synth.scaled(W["llama3_8b_2k"], batch=batch, prefix=(prefix, prefix + 40), n_q_heads=hq, n_kv_heads=hkv, n_nodes=nodes, depth=4,
                     branch=12, vocab=vocab, temperatures=temps, n_layers=1)
    inp = synth.generate(w, 6)
    assert inp.parent.size * vocab >= 1 << 21
    B, N = inp.parent.shape
    ctx = helpers.make_ctx(inp, n_layers=1)
    cache0 = binding.bf16_tensor(synth.make_cache(inp, 1))
    d, a = helpers.upload_accept(inp), helpers.upload_attn(inp)
    L = inp.prefix_len
    for b in range(B):
        cache0[0, 0, b, :, L[b]:L[b] + N] = a["tree_k"][b]
        cache0[0, 1, b, :, L[b]:L[b] + N] = a["tree_v"][b]
    i32 = dict(dtype=torch.int32, device="cuda")

    def outputs():
        return [torch.zeros_like(a["q"]), torch.zeros((B, N), **i32)] + [torch.zeros((B,), **i32) for _ in range(3)]

    def step(cache, out):
        ctx.verify_step(cache, a["q"], a["tree_k"], a["tree_v"], d["parent"], a["prefix_len"], d["target_logits"], d["draft_probs"],
                        d["draft_tokens"], d["temperature"], d["uniforms"], *out)

    called, cache = outputs(), cache0.clone()
    step(cache, called)
    ctx.check()
    path, n, bonus = ctx.tree_accept(d["target_logits"], d["draft_probs"], d["draft_tokens"], d["parent"], d["temperature"], d["uniforms"])
    want = cache0.clone()
    new_len = ctx.kv_compact(want, path, n, a["prefix_len"])
    for got, ref in zip(called[1:] + [cache], [path, n, bonus, new_len, want]):
        assert torch.equal(got.view(torch.int16), ref.view(torch.int16))
    hard, near, msgs = helpers.compare_accept(inp, path.cpu().numpy(), n.cpu().numpy(), bonus.cpu().numpy())
    assert hard == 0, msgs
    replayed, cache_g = outputs(), cache0.clone()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        step(cache_g, replayed)
    for _ in range(2):
        cache_g.copy_(cache0)
        for t in replayed:
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        ctx.check()
        for got, ref in zip(replayed + [cache_g], called + [cache]):
            assert torch.equal(got.view(torch.int16), ref.view(torch.int16))
    ref_o = oracle.tree_attn(inp.q, inp.k_cache, inp.v_cache, inp.tree_k, inp.tree_v, inp.parent, L)
    mx, mean = helpers.attn_errors(called[0], ref_o)
    assert mx <= 1e-2 and mean <= 1e-3


def _host_step(ctx, inp, logits):
    """The host entry point on `inp` with its logits in `logits`: the outputs and the cache."""
    B, N = inp.parent.shape
    sampling = inp.draft_probs is not None
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()   # noqa: E731
    cache = binding.bf16_tensor(synth.make_cache(inp, 1))
    out = torch.empty(inp.q.shape, dtype=torch.bfloat16).pin_memory()
    path = torch.empty((B, N), dtype=torch.int32)
    n, bonus, new_len = (torch.empty((B,), dtype=torch.int32) for _ in range(3))
    ctx.verify_step_host(cache, *(binding.bf16_tensor(a, "cpu").pin_memory() for a in (inp.q, inp.tree_k, inp.tree_v)), pin(inp.parent),
                         pin(inp.prefix_len), logits, pin(inp.draft_probs) if sampling else None, pin(inp.draft_tokens),
                         pin(inp.temperature), pin(inp.uniforms) if sampling else None, out, path, n, bonus, new_len)
    return out, path, n, bonus, new_len, cache


# every other row has children, or all but one of few: a CTA for every piece, fewer pieces a row than 16, shares of rows laid end to end
@pytest.mark.parametrize("tree,branch,nodes,batch,vocab", [("chain", 1, 8, 1, 50257), ("bfs", 2, 120, 1, 32753), ("bfs", 2, 200, 3, 8001),
                                                           ("bfs", 2, 250, 5, 2003)])
@pytest.mark.parametrize("mode", ["greedy", "sample"])
def test_most_rows_read_where_they_are(tree, branch, nodes, batch, vocab, mode):
    """Rows that the scan brings to the device while the walk that sweeps them is already resident: other logits in the same memory at
    every call, and the oracle's acceptance each time (children are rejected at the root at least once)."""
    w = synth.scaled(W["llama3_8b_2k"], batch=batch, prefix=(40, 300), n_nodes=nodes, tree=tree, branch=branch, vocab=vocab,
                     temperatures=((0.0,) * 5 if mode == "greedy" else (1.0, 0.7, 1.0, 0.0, 0.7))[:batch])
    inps = [synth.generate(w, v) for v in (1, 2, 3, 4)]
    ctx = helpers.make_ctx(inps[0], n_layers=1)
    logits = torch.empty(inps[0].target_logits.shape).pin_memory()
    rejected = 0
    for inp in inps:
        logits.copy_(torch.from_numpy(inp.target_logits))
        _, path, n, bonus, new_len, _ = _host_step(ctx, inp, logits)
        hard, near, msgs = helpers.compare_accept(inp, path.numpy(), n.numpy(), bonus.numpy())
        assert hard == 0 and near == 0, msgs
        assert np.array_equal(new_len.numpy(), inp.prefix_len + n.numpy())
        rejected += int((n.numpy() < 2).sum())
    assert rejected > 0


@pytest.mark.parametrize("vocab", [1, 2, 3, 5])
@pytest.mark.parametrize("mode", ["greedy", "sample"])
def test_rows_of_less_than_a_unit(vocab, mode):
    """The host entry point on rows shorter than the unit they are read by, from logits that end where their allocation ends."""
    nodes, batch = 6, 3
    w = synth.scaled(W["llama3_8b_2k"], batch=batch, prefix=(8, 40), n_nodes=nodes, tree="chain", vocab=vocab,
                     temperatures=(0.0,) * batch if mode == "greedy" else (1.0, 0.0, 0.7))
    for variant in range(3):
        inp = synth.generate(w, variant)
        ctx = helpers.make_ctx(inp, n_layers=1)
        _, path, n, bonus, _, _ = _host_step(ctx, inp, torch.from_numpy(inp.target_logits).pin_memory())
        hard, near, msgs = helpers.compare_accept(inp, path.numpy(), n.numpy(), bonus.numpy())
        assert hard == 0 and near == 0, msgs


# rows with children and the CTAs of the scan (592): fewer pieces a row than 16; one piece a row; shares laid end to end, of two rows, of
# several whole ones, with more rows than one word of marks a lane
@pytest.mark.parametrize("tree,branch,nodes,batch,vocab", [
    ("chain", 1, 64, 2, 40000), ("chain", 1, 80, 5, 12800), ("bfs", 2, 200, 3, 16384), ("chain", 1, 62, 5, 31001), ("chain", 1, 256, 6, 4100),
    ("bfs", 2, 250, 10, 3802), ("chain", 1, 256, 32, 1161)])
@pytest.mark.parametrize("mode", ["greedy", "mixed"])
def test_many_rows_with_children(tree, branch, nodes, batch, vocab, mode):
    """Trees most of whose nodes have children, on which the walk goes some way: every draft token has the largest logit of its parent's
    row, at the very first, at the very last or at some other position, and a few of them do not."""
    w = synth.scaled(W["llama3_8b_2k"], batch=batch, vocab=vocab, n_nodes=nodes, tree=tree, branch=branch, prefix=(8, 8),
                     temperatures=(0.0,) * batch if mode == "greedy" else ((1.0, 0.0, 0.7) * 11)[:batch])
    rng = np.random.default_rng(vocab)
    for variant in range(2):
        inp = synth.generate(w, variant, with_attention=False)
        assert inp.parent.size * vocab >= (9.5e6 if vocab % 4 else 5e6)                                        # (else every row is scanned)
        for b in range(batch):
            for c in range(1, nodes):
                p = inp.parent[b, c]
                at = inp.draft_tokens[b, c]
                if rng.random() < 0.15 and (inp.parent[b, 1:c] != p).all():
                    at = inp.draft_tokens[b, c] = (0, vocab - 1)[int(rng.integers(2))]
                if rng.random() < 0.97:
                    inp.target_logits[b, p, at] = 20.0 + 10.0 * float(inp.temperature[b] > 0)
        path, n_acc, _ = _parity(inp, allow_near=2)
        assert n_acc.max() > 4


@pytest.mark.parametrize("vocab,nodes", [(270000, 24), (262148, 33), (200001, 70)])
def test_rows_that_shared_memory_does_not_hold(vocab, nodes):
    """A slice of the row of more tokens than can be parked: every sweep and the draw at a leaf read the row itself."""
    w = synth.scaled(W["llama3_8b_2k"], batch=1, vocab=vocab, n_nodes=nodes, depth=3, branch=12, temperatures=(1.0,), prefix=(8, 8))
    at_leaf = 0
    for variant in range(4):
        inp = synth.generate(w, variant, with_attention=False)
        assert inp.parent.size * vocab >= 4e6
        if variant % 2:                                                  # the first child of the root is accepted, and is a leaf or is not
            inp.target_logits[0, 0, inp.draft_tokens[0, 1 if variant == 1 else nodes - 1]] = 40.0
        path, n_acc, _ = _parity(inp)
        at_leaf += _leaf_ends(inp, path, n_acc)
    assert at_leaf > 0


@pytest.mark.parametrize("nodes,batch,vocab", [(60, 1, 65536), (130, 3, 32001), (32, 2, 128256), (9, 1, 50257)])      # (the last in one stream)
def test_greedy_step_whose_clusters_compact(nodes, batch, vocab):
    """All sequences greedy, few slices: the CTAs that share a leaf's row share the moves of the cache rows, too."""
    w = synth.scaled(W["llama3_8b_2k"], batch=batch, prefix=(300, 500), n_nodes=nodes, depth=5, branch=8 if nodes <= 64 else 16, vocab=vocab,
                     temperatures=(0.0,) * batch, n_layers=2)
    for variant in range(3):
        inp = synth.generate(w, variant)
        B, N = inp.parent.shape
        ctx = helpers.make_ctx(inp, n_layers=2)
        cache = binding.bf16_tensor(synth.make_cache(inp, 2))
        want = cache.clone()
        d, a = helpers.upload_accept(inp), helpers.upload_attn(inp)
        i32 = dict(dtype=torch.int32, device="cuda")
        out, path = torch.zeros_like(a["q"]), torch.zeros((B, N), **i32)
        n, bonus, new_len = (torch.zeros((B,), **i32) for _ in range(3))
        ctx.verify_step(cache, a["q"], a["tree_k"], a["tree_v"], d["parent"], a["prefix_len"], d["target_logits"], None, d["draft_tokens"],
                        d["temperature"], None, out, path, n, bonus, new_len)
        ctx.check()
        hard, near, msgs = helpers.compare_accept(inp, path.cpu().numpy(), n.cpu().numpy(), bonus.cpu().numpy())
        assert hard == 0, msgs
        ref_len = ctx.kv_compact(want, path, n, a["prefix_len"])
        assert torch.equal(new_len, ref_len) and torch.equal(cache.view(torch.int16), want.view(torch.int16))


@pytest.mark.parametrize("vocab,nodes,batch", [(8193, 2, 1), (8196, 3, 3), (32001, 4, 2), (128256, 9, 1)])
@pytest.mark.parametrize("temp", [0.0, 0.7])
def test_up_to_nine_rows(vocab, nodes, batch, temp):
    """Stars whose last child is certain to be accepted: the walk ends in a row that the scan has left out."""
    w = synth.scaled(W["tiny_greedy"], batch=batch, vocab=vocab, n_nodes=nodes, tree="star", temperatures=(temp,) * batch, prefix=(8, 8))
    for variant in range(3):
        inp = synth.generate(w, variant, with_attention=False)
        for b in range(batch):
            inp.target_logits[b, 0, inp.draft_tokens[b, nodes - 1]] = 60.0
        path, n_acc, _ = _parity(inp, allow_near=0)
        assert (n_acc == 2).all() and (path[:, 1] == nodes - 1).all()
