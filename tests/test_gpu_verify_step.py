"""The whole verify step in one call (`fspad_verify_step`: attention on the context's second
stream beside acceptance, then compaction) against the oracle: attention within the stated bound,
acceptance and the compacted cache bit-exact.  Both forms of the tree rows (explicit arrays, and
rows of the cache that the compaction then rewrites), eager and replayed from a CUDA graph."""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_15562_b200 import binding, synth
from tests import helpers

pytestmark = pytest.mark.gpu

W = synth.WORKLOADS


def _oracle_step(inp, cache_host, layer):
    ref_o = oracle.tree_attn(inp.q, inp.k_cache, inp.v_cache, inp.tree_k, inp.tree_v, inp.parent, inp.prefix_len)
    r = oracle.tree_accept(inp.target_logits, inp.draft_probs, inp.draft_tokens, inp.parent, inp.temperature,
                           inp.uniforms if inp.draft_probs is not None else None)
    want = cache_host.copy()
    want_len = oracle.kv_compact(want, r["accepted_path"], r["n_accepted"], inp.prefix_len)
    return ref_o, r, want, want_len


def _device_inputs(inp, cache_host):
    d = helpers.upload_accept(inp)
    a = helpers.upload_attn(inp)
    B, N = inp.parent.shape
    outs = dict(attn_out=torch.empty_like(a["q"]), path=torch.full((B, N), -7, dtype=torch.int32, device="cuda"),
                n_acc=torch.empty((B,), dtype=torch.int32, device="cuda"),
                bonus=torch.empty((B,), dtype=torch.int32, device="cuda"),
                new_len=torch.empty((B,), dtype=torch.int32, device="cuda"))
    return d, a, outs, binding.bf16_tensor(cache_host)


def _call(ctx, cache, a, d, outs, aliased, layer):
    ctx.verify_step(cache, a["q"], None if aliased else a["tree_k"], None if aliased else a["tree_v"], a["parent"],
                    a["prefix_len"], d["target_logits"], d["draft_probs"], d["draft_tokens"], d["temperature"],
                    d["uniforms"], outs["attn_out"], outs["path"], outs["n_acc"], outs["bonus"], outs["new_len"],
                    attn_layer=layer)


def _check(inp, outs, cache, ref_o, r, want, want_len):
    mx, mean = helpers.attn_errors(outs["attn_out"], ref_o)
    assert mx <= 1e-2 and mean <= 1e-3, (mx, mean)
    hard, near, msgs = helpers.compare_accept(inp, outs["path"].cpu().numpy(), outs["n_acc"].cpu().numpy(),
                                              outs["bonus"].cpu().numpy())
    assert hard == 0 and near == 0, msgs
    np.testing.assert_array_equal(outs["new_len"].cpu().numpy(), want_len)
    got = binding.bf16_bits(cache)
    for b in range(inp.parent.shape[0]):           # rows past the new length are dead
        rows = int(want_len[b])
        np.testing.assert_array_equal(got[:, :, b, :, :rows], want[:, :, b, :, :rows])


@pytest.mark.parametrize("n_layers", [3, 5])      # 48 and 80 (layer, K/V, head) slices per sequence: up to 64 the walk's
@pytest.mark.parametrize("aliased", [False, True])  # own CTAs compact the cache, above that the compaction kernel does
@pytest.mark.parametrize("mode", ["sample", "greedy", "mixed"])
def test_whole_step_against_oracle(mode, aliased, n_layers):
    temps = {"sample": (1.0, 0.8, 1.0), "greedy": (0.0, 0.0, 0.0), "mixed": (0.0, 1.0, 0.0)}[mode]
    w = synth.scaled(W["llama3_8b_2k"], batch=3, prefix=(40, 300), n_nodes=24, depth=4, branch=4, vocab=3000,
                     temperatures=temps)
    inp = synth.generate(w, 11)
    B, N = inp.parent.shape
    layer = 1
    cache_host = synth.make_cache(inp, n_layers)
    L = inp.prefix_len
    for b in range(B):          # the attention layer's planes are the workload's K/V; tree rows behind the prefix
        cache_host[layer, 0, b] = inp.k_cache[b]
        cache_host[layer, 1, b] = inp.v_cache[b]
        cache_host[layer, 0, b, :, L[b]:L[b] + N] = inp.tree_k[b]
        cache_host[layer, 1, b, :, L[b]:L[b] + N] = inp.tree_v[b]
    ref_o, r, want, want_len = _oracle_step(inp, cache_host, layer)
    ctx = helpers.make_ctx(inp, n_layers=n_layers)
    d, a, outs, cache = _device_inputs(inp, cache_host)
    _call(ctx, cache, a, d, outs, aliased, layer)
    ctx.check()
    _check(inp, outs, cache, ref_o, r, want, want_len)


def test_whole_step_headline_shape_in_a_graph():
    """Full llama3_8b_2k launch configuration, captured once and replayed: the fork and join of the
    second stream are part of the graph."""
    inp = synth.generate(W["llama3_8b_2k"], 0)
    cache_host = synth.make_cache(inp, 1)
    ref_o, r, want, want_len = _oracle_step(inp, cache_host, 0)
    ctx = helpers.make_ctx(inp, n_layers=1)
    d, a, outs, cache = _device_inputs(inp, cache_host)
    _call(ctx, cache, a, d, outs, False, 0)        # warm-up outside the capture (one-time attribute calls)
    torch.cuda.synchronize()
    cache.copy_(binding.bf16_tensor(cache_host))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        _call(ctx, cache, a, d, outs, False, 0)
    outs["attn_out"].zero_()
    outs["path"].fill_(-7)
    g.replay()
    torch.cuda.synchronize()
    ctx.check()
    _check(inp, outs, cache, ref_o, r, want, want_len)


@pytest.mark.parametrize("mode,heads,prefix,n_layers,aliased", [
    ("sample", 80, 300, 1, False),      # one key range a row; the walk's CTAs compact 160 slices
    ("sample", 80, 300, 2, False),      # 320 slices: the compaction kernel, behind the attention
    ("sample", 80, 300, 1, True),       # the compaction rewrites rows that the attention reads
    ("sample", 70, 3000, 1, False),     # two ranges of 12 chunks: the merge kernel follows
    ("greedy", 80, 300, 1, False),      # short scan, one-CTA walk
])
def test_step_in_one_stream(mode, heads, prefix, n_layers, aliased):
    """The attention launched beside the walk in the caller's stream: eager, and replayed twice back to back from a graph."""
    w = synth.scaled(W["llama3_8b_2k"], batch=1, n_q_heads=heads, n_kv_heads=heads, prefix=(prefix, prefix), n_nodes=24,
                     depth=4, branch=4, vocab=3000, temperatures=(1.0 if mode == "sample" else 0.0,))
    inp = synth.generate(w, 12)
    N, L = inp.parent.shape[1], int(inp.prefix_len[0])
    cache_host = synth.make_cache(inp, n_layers)
    cache_host[0, 0, 0], cache_host[0, 1, 0] = inp.k_cache[0], inp.v_cache[0]
    cache_host[0, 0, 0, :, L:L + N], cache_host[0, 1, 0, :, L:L + N] = inp.tree_k[0], inp.tree_v[0]
    ref = _oracle_step(inp, cache_host, 0)
    ctx = helpers.make_ctx(inp, n_layers=n_layers)
    d, a, outs, cache = _device_inputs(inp, cache_host)
    _call(ctx, cache, a, d, outs, aliased, 0)
    ctx.check()
    _check(inp, outs, cache, *ref)
    again = binding.bf16_tensor(cache_host)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(2):
            cache.copy_(again)
            _call(ctx, cache, a, d, outs, aliased, 0)
    outs["attn_out"].zero_()
    outs["path"].fill_(-7)
    g.replay()
    ctx.check()
    _check(inp, outs, cache, *ref)


@pytest.mark.parametrize("prefix,heads", [(60, 8), (300, 8), (2048, 8), (9000, 8), (1000, 40)])
def test_sequence_of_any_length_in_a_long_context(prefix, heads):
    """A context of 16384 rows cuts the keys into eight (three) ranges, some of them empty for a short sequence, and the step goes through
    one stream: the merge of the ranges reads them while the walk may still be under way.  Two different steps in turn, three times
    over, each checked against the oracle."""
    w = synth.scaled(W["llama3_8b_2k"], batch=1, n_q_heads=32 if heads == 8 else heads, n_kv_heads=heads,
                     prefix=(prefix, prefix), n_nodes=40, depth=5, branch=5, vocab=33000, temperatures=(1.0,))
    cap = 16384
    ctx, steps = None, []
    for seed in (1, 2):
        inp = synth.generate(w, seed)
        N, L = inp.parent.shape[1], int(inp.prefix_len[0])
        ctx = ctx or binding.Context(w.n_q_heads, heads, w.vocab, cap, max_nodes=N)
        ref_o, r, _, _ = _oracle_step(inp, synth.make_cache(inp, 1), 0)
        d, a, outs, _ = _device_inputs(inp, np.zeros((1, 2, 1, 1, 1, 1), np.uint16))
        cache = torch.zeros((1, 2, 1, heads, cap, 128), dtype=torch.bfloat16, device="cuda")
        cache[0, 0, :, :, :L], cache[0, 1, :, :, :L] = a["k_cache"][:, :, :L], a["v_cache"][:, :, :L]
        cache[0, 0, :, :, L:L + N], cache[0, 1, :, :, L:L + N] = a["tree_k"], a["tree_v"]
        steps.append((inp, d, a, outs, cache, cache.clone(), ref_o, r))
    for _ in range(3):
        for inp, d, a, outs, cache, fresh, _, _ in steps:
            outs["attn_out"].fill_(float("nan"))
            cache.copy_(fresh)
            _call(ctx, cache, a, d, outs, False, 0)
        ctx.check()
        for inp, d, a, outs, cache, fresh, ref_o, r in steps:
            mx, mean = helpers.attn_errors(outs["attn_out"], ref_o)
            assert mx <= 1e-2 and mean <= 1e-3, (mx, mean)
            hard, near, msgs = helpers.compare_accept(inp, outs["path"].cpu().numpy(), outs["n_acc"].cpu().numpy(),
                                                      outs["bonus"].cpu().numpy())
            assert hard == 0 and near == 0, msgs
            L, n = int(inp.prefix_len[0]), int(outs["n_acc"][0])
            rows = L + outs["path"][0, :n].long()
            assert torch.equal(cache[:, :, :, :, L:L + n], fresh[:, :, :, :, rows])
            assert int(outs["new_len"][0]) == L + n


@pytest.mark.parametrize("n_nodes,group", [(33, 4), (64, 4), (60, 5), (60, 8), (130, 3), (200, 2)])
@pytest.mark.parametrize("alias", [False, True])
def test_row_tiles_in_pairs_of_ctas(n_nodes, group, alias):
    """A batch whose row tiles fill the SMs goes on pairs of CTAs inside a step and on lone ones in a call of the attention alone
    (which is checked against the oracle at these shapes): the same bits, with 1 .. 12 chunks a sequence, an empty half of the last
    pair, the boundary between the tiles inside a node's heads, tree rows apart and in the cache."""
    B = 12
    L = np.array([0, 100, 128, 129, 383, 500, 640, 700, 900, 1151, 1280, 1400], np.int32)
    w = synth.scaled(W["batch16_ragged"], batch=B, n_q_heads=8 * group, n_kv_heads=8, n_nodes=n_nodes, depth=6, branch=12,
                     prefix=(int(L.max()), int(L.max())), temperatures=(0.0,) * B, vocab=64, n_layers=1)
    inp = synth.generate(w, n_nodes)
    N = inp.parent.shape[1]
    inp.prefix_len[:] = L
    ctx = helpers.make_ctx(inp, n_layers=1)
    cache_host = synth.make_cache(inp, 1)
    cache_host[0, 0], cache_host[0, 1] = inp.k_cache, inp.v_cache
    for b in range(B):
        cache_host[0, 0, b, :, L[b]:L[b] + N], cache_host[0, 1, b, :, L[b]:L[b] + N] = inp.tree_k[b], inp.tree_v[b]
    d, a, outs, cache = _device_inputs(inp, cache_host)
    tree = (None, None) if alias else (a["tree_k"], a["tree_v"])
    want = ctx.tree_attn(a["q"], cache[0, 0].clone(), cache[0, 1].clone(), *tree, a["parent"], a["prefix_len"])
    _call(ctx, cache, a, d, outs, alias, 0)
    ctx.check()
    assert torch.equal(outs["attn_out"], want)


@pytest.mark.parametrize("mode", ["sample", "mixed", "zero"])
@pytest.mark.parametrize("vocab,heads,n_layers", [
    (33000, 10, 4),        # clusters of 16 CTAs, 80 slices: half a slice a warp
    (33000, 32, 4),        # 256 slices
    (16500, 32, 2),        # clusters of eight, 128 slices
])
def test_step_in_one_stream_beside_clusters(mode, vocab, heads, n_layers):
    """Three sequences whose walks take a cluster each, the attention beside them, the cache compacted by the walk's CTAs (a sequence
    of temperature 0: by one of them).  Three launches and no more say that it went this way."""
    temps = {"sample": (1.0, 0.8, 1.0), "mixed": (0.0, 1.0, 0.0), "zero": (0.0, 0.0, 0.0)}[mode]
    w = synth.scaled(W["llama3_8b_2k"], batch=3, n_q_heads=heads, n_kv_heads=heads, prefix=(40, 500), n_nodes=24, depth=4, branch=4,
                     vocab=vocab, temperatures=temps if mode != "zero" else (1.0, 1.0, 1.0))
    inp = synth.generate(w, 21)
    inp.temperature[:] = temps
    B, N = inp.parent.shape
    cache_host = synth.make_cache(inp, n_layers)
    for b, L in enumerate(inp.prefix_len.tolist()):
        cache_host[0, 0, b, :, L:L + N], cache_host[0, 1, b, :, L:L + N] = inp.tree_k[b], inp.tree_v[b]
    ref = _oracle_step(inp, cache_host, 0)
    ctx = helpers.make_ctx(inp, n_layers=n_layers)
    d, a, outs, cache = _device_inputs(inp, cache_host)
    before = ctx.launch_count()
    _call(ctx, cache, a, d, outs, False, 0)
    assert ctx.launch_count() - before == 3              # scan, walk, attention
    ctx.check()
    _check(inp, outs, cache, *ref)


@pytest.mark.parametrize("mode,heads,prefix,max_len", [("sample", 32, 300, 400), ("sample", 8, 1000, 16384), ("greedy", 32, 300, 400),
                                                       ("sample", 8, 1000, 1100)])
def test_inputs_rewritten_between_steps(mode, heads, prefix, max_len):
    """Trees, lengths, queries and logits rewritten in place by kernels right before each step, with nothing waited for: every step
    sees its own, whichever stream its attention takes and however early that starts."""
    w = synth.scaled(W["llama3_8b_2k"], batch=1, n_q_heads=heads, n_kv_heads=heads, prefix=(prefix, prefix), n_nodes=24, depth=4, branch=4,
                     vocab=33000, temperatures=(1.0 if mode == "sample" else 0.0,))
    sets = []
    for k in range(3):
        inp = synth.generate(w, 30 + k)
        assert inp.parent.shape[1] == 24
        inp.prefix_len[:] = prefix - 37 * k
        d, a, outs, _ = _device_inputs(inp, np.zeros((1, 2, 1, 1, 1, 1), np.uint16))
        cache = torch.randn((1, 2, 1, heads, max_len, 128), device="cuda").to(torch.bfloat16)
        sets.append((d, a, cache))
    ctx = binding.Context(heads, heads, w.vocab, max_len, max_nodes=24)
    live = ({k: None if t is None else t.clone() for k, t in sets[0][0].items()}, {k: t.clone() for k, t in sets[0][1].items()}, sets[0][2].clone())

    def step(k, wait):
        for src, dst in ((sets[k][0], live[0]), (sets[k][1], live[1]), ({"c": sets[k][2]}, {"c": live[2]})):
            for name, t in src.items():
                if t is not None:
                    torch.add(t, 0, out=dst[name])       # (a kernel, not a copy)
        if wait:
            torch.cuda.synchronize()
        res = {key: torch.empty_like(t) for key, t in outs.items()}
        _call(ctx, live[2], live[1], live[0], res, False, 0)
        if wait:
            ctx.check()
        return [res[key] for key in ("attn_out", "path", "n_acc", "bonus", "new_len")] + [live[2].clone()]

    want = [step(k, True) for k in range(3)]
    assert not torch.equal(want[0][0], want[1][0]) and len({tuple(x[1][0].tolist()) for x in want}) > 1
    got = [step(k % 3, False) for k in range(12)]
    ctx.check()
    for k, res in enumerate(got):
        for g, r in zip(res, want[k % 3]):
            assert torch.equal(g, r), k


def test_argument_errors():
    w = synth.scaled(W["llama3_8b_2k"], batch=1, prefix=(40, 40), n_nodes=8, depth=3, branch=3, vocab=100,
                     temperatures=(0.0,))
    inp = synth.generate(w, 0)
    ctx = helpers.make_ctx(inp, n_layers=1)
    d, a, outs, cache = _device_inputs(inp, synth.make_cache(inp, 1))
    with pytest.raises(binding.FspadError) as e:
        _call(ctx, cache, a, d, outs, False, 1)    # layer out of range
    assert e.value.code == -3
    with pytest.raises(binding.FspadError) as e:
        ctx.verify_step(None, a["q"], None, None, a["parent"], a["prefix_len"], d["target_logits"], None,
                        d["draft_tokens"], d["temperature"], None, outs["attn_out"], outs["path"], outs["n_acc"],
                        outs["bonus"], outs["new_len"])
    assert e.value.code == -1
    _call(ctx, cache, a, d, outs, True, 0)         # and the context still works
    ctx.check()
