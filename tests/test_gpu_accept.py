"""CUDA acceptance (through the C ABI) against the oracle: bit-exact path, length
and bonus token; divergences are tolerated only inside the 1e-6 decision band and
are counted."""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_15562_b200 import binding, synth
from tests import helpers

pytestmark = pytest.mark.gpu

W = synth.WORKLOADS


def _run(inp, ctx=None):
    ctx = ctx or helpers.make_ctx(inp)
    d = helpers.upload_accept(inp)
    path, n_acc, bonus = ctx.tree_accept(d["target_logits"], d["draft_probs"], d["draft_tokens"], d["parent"],
                                         d["temperature"], d["uniforms"])
    ctx.check()
    return path.cpu().numpy(), n_acc.cpu().numpy(), bonus.cpu().numpy()


def _assert_parity(inp, allow_near=0):
    path, n_acc, bonus = _run(inp)
    hard, near, msgs = helpers.compare_accept(inp, path, n_acc, bonus)
    assert hard == 0, msgs
    assert near <= allow_near, msgs
    return near


@pytest.mark.parametrize("vocab", [8, 33, 1000, 4099, 32000])
@pytest.mark.parametrize("mode", ["greedy", "sample", "mixed"])
def test_small_trees_many_seeds(vocab, mode):
    temps = {"greedy": (0.0,) * 4, "sample": (1.0, 1.0, 0.7, 1.3), "mixed": (0.0, 1.0, 0.0, 0.5)}[mode]
    total_near = 0
    for variant in range(6):
        w = synth.scaled(W["llama3_8b_2k"], batch=4, vocab=vocab, n_nodes=min(20, vocab), depth=4, branch=3,
                         temperatures=temps, prefix=(8, 8))
        inp = synth.generate(w, variant, with_attention=False)
        total_near += _assert_parity(inp, allow_near=1)
    assert total_near <= 1


@pytest.mark.parametrize("tree", ["chain", "star", "bfs"])
def test_special_trees(tree):
    for temps in ((0.0, 0.0), (1.0, 1.0)):
        w = synth.scaled(W["tiny_greedy"], batch=2, vocab=2000, n_nodes=9, tree=tree, branch=2,
                         temperatures=temps, prefix=(8, 8))
        for variant in range(4):
            _assert_parity(synth.generate(w, variant, with_attention=False))


def test_root_only_tree_and_max_nodes():
    for n in (1, 64):
        w = synth.scaled(W["llama3_8b_2k"], batch=2, vocab=5000, n_nodes=n, depth=5 if n > 1 else 1, branch=4,
                         temperatures=(0.0, 1.0), prefix=(8, 8))
        _assert_parity(synth.generate(w, 0, with_attention=False))


def test_draft_far_from_target_forces_many_rejections():
    """A draft distribution unrelated to the target: most children are rejected,
    so the residual chain and the bonus draw from a deep residual are exercised."""
    w = synth.scaled(W["llama3_8b_2k"], batch=8, vocab=3000, n_nodes=24, depth=3, branch=8,
                     temperatures=(1.0,) * 8, prefix=(8, 8))
    rejected_somewhere = 0
    for variant in range(4):
        inp = synth.generate(w, variant, with_attention=False)
        rng = np.random.default_rng(variant)
        z = rng.standard_normal(inp.draft_probs.shape) * 3
        q = np.exp(z - z.max(-1, keepdims=True))
        inp.draft_probs[...] = (q / q.sum(-1, keepdims=True)).astype(np.float32)
        for b in range(w.batch):                    # children carry the draft's own favourite tokens
            for i, ch in enumerate(synth.children_lists(inp.parent[b])):
                if ch:
                    inp.draft_tokens[b, ch] = np.argsort(-inp.draft_probs[b, i], kind="stable")[:len(ch)]
        _assert_parity(inp)
        r = oracle.tree_accept(inp.target_logits, inp.draft_probs, inp.draft_tokens, inp.parent,
                               inp.temperature, inp.uniforms)
        rejected_somewhere += int((~np.isnan(r["trace_rq"])).sum() - (r["n_accepted"] - 1).sum())
    assert rejected_somewhere > 20


def test_draft_equal_to_target_up_to_fp32_rounding():
    """q = softmax(logits) up to a few fp32 ulps: every token sits inside the band where the scan's approximate
    denominator cannot fix the sign of p - q, so the one-sweep first rejection must hand over to the
    exact two-sweep path; the residual mass itself is of the order of fp32 rounding."""
    w = synth.scaled(W["llama3_8b_2k"], batch=6, vocab=5000, n_nodes=24, depth=3, branch=8,
                     temperatures=(1.0, 1.0, 0.7, 0.7, 1.3, 1.3), prefix=(8, 8))
    rejected = 0
    for variant in range(3):
        inp = synth.generate(w, variant, with_attention=False)
        z = inp.target_logits.astype(np.float64) / inp.temperature[:, None, None].astype(np.float64)
        p = np.exp(z - z.max(-1, keepdims=True))
        wobble = 1.0 + 3e-7 * np.random.default_rng(variant).choice([-1.0, 1.0], size=p.shape)
        inp.draft_probs[...] = (p / p.sum(-1, keepdims=True) * wobble).astype(np.float32)
        # uniforms just below one: r * q < p now fails wherever q lies above p, so rejections do occur
        keep = inp.uniforms[:, -1].copy()
        inp.uniforms[...] = np.nextafter(np.float32(1), np.float32(0))
        inp.uniforms[:, -1] = keep
        _assert_parity(inp, allow_near=w.batch)
        r = oracle.tree_accept(inp.target_logits, inp.draft_probs, inp.draft_tokens, inp.parent,
                               inp.temperature, inp.uniforms)
        rejected += int((~np.isnan(r["trace_rq"])).sum() - (r["n_accepted"] - 1).sum())
    assert rejected > 0


def test_zero_mass_and_minus_inf_logits():
    w = synth.scaled(W["llama3_8b_2k"], batch=4, vocab=512, n_nodes=16, depth=4, branch=3,
                     temperatures=(1.0,) * 4, prefix=(8, 8))
    inp = synth.generate(w, 3, with_attention=False)
    rng = np.random.default_rng(0)
    kill = rng.random(inp.target_logits.shape) < 0.3
    inp.target_logits[kill] = -np.inf
    dz = rng.random(inp.draft_probs.shape) < 0.3
    inp.draft_probs[dz] = 0.0
    _assert_parity(inp)


def test_stats_pass_matches_oracle_rows():
    w = synth.scaled(W["llama3_8b_2k"], batch=2, vocab=128256, n_nodes=7, depth=3, branch=3,
                     temperatures=(1.0, 0.6), prefix=(8, 8))
    inp = synth.generate(w, 0, with_attention=False)
    inp.target_logits[0, 3, 777] = inp.target_logits[0, 3].max()      # duplicate maxima: lowest index wins
    inp.target_logits[0, 3, 100000] = inp.target_logits[0, 3, 777]
    ctx = helpers.make_ctx(inp)
    lg = helpers.dev(inp.target_logits.reshape(-1, w.vocab))
    m, s, a = ctx.accept_stats(lg, helpers.dev(inp.temperature), 7)
    ctx.check()
    for b in range(2):
        om, os_, oa = oracle.row_stats(inp.target_logits[b], float(inp.temperature[b]))
        sl = slice(b * 7, b * 7 + 7)
        np.testing.assert_array_equal(m[sl].cpu().numpy().astype(np.float64), om)
        np.testing.assert_array_equal(a[sl].cpu().numpy(), oa)
        np.testing.assert_allclose(s[sl].cpu().numpy(), os_, rtol=2e-6)
    assert int(a[3]) == min(777, int(np.argmax(inp.target_logits[0, 3])))


@pytest.mark.parametrize("rows,vocab", [(1, 5), (3, 33), (7, 4097), (60, 32001), (130, 50257), (700, 2049), (1300, 1003), (64, 50258)])
def test_stats_rows_of_any_length(rows, vocab):
    """Vocabularies that are no multiple of four (rows start at every alignment), one piece per row and many, more rows than one
    wave of CTAs holds; the maximum sits at a random position, at the first and at the last.  Maximum and index exact; the sum is
    fp32 with ex2.approx: 2e-6 relative."""
    rng = np.random.default_rng(rows)
    x = (rng.standard_normal((rows, vocab)) * 3).astype(np.float32)
    x[::3, 0] = 20.0
    x[1::3, -1] = 20.0
    ctx = binding.Context(8, 2, vocab, 512, max_nodes=min(rows, 256), max_batch=(rows + 255) // 256)
    temp = torch.full(((rows + 9) // 10,), 0.8, device="cuda")
    m, s, a = ctx.accept_stats(helpers.dev(x), temp, 10)
    ctx.check()
    om, os_, oa = oracle.row_stats(x, 0.8)
    assert np.array_equal(m.cpu().numpy(), om.astype(np.float32))
    assert np.array_equal(a.cpu().numpy(), oa)
    np.testing.assert_allclose(s.cpu().numpy(), os_, rtol=2e-6)


@pytest.mark.parametrize("name", ["tiny_greedy", "llama3_8b_2k", "vicuna_33b_4k_greedy",
                                  "vicuna_33b_4k_sample", "llama3_70b_8k"])
def test_full_size_single_sequence_configs(name):
    for variant in range(2):
        inp = synth.generate(W[name], variant, with_attention=False)
        _assert_parity(inp, allow_near=1)


def test_full_size_batch16_mixed():
    inp = synth.generate(W["batch16_ragged"], 0, with_attention=False)
    _assert_parity(inp, allow_near=1)


@pytest.mark.parametrize("pattern", ["alternating", "greedy_last", "one_sampling", "all_sampling"])
def test_more_clusters_than_the_sms_hold(pattern):
    """20 sequences of 16 CTAs each: the sampling ones are taken first, wherever they stand in the batch, and a greedy one is one
    CTA's work; every sequence gets its own result."""
    B = 20
    temps = {"alternating": (0.0, 1.0) * 10, "greedy_last": (0.8,) * 13 + (0.0,) * 7, "one_sampling": (0.0,) * 11 + (1.0,) + (0.0,) * 8,
             "all_sampling": (1.0, 0.7, 1.3, 0.9) * 5}[pattern]
    w = synth.scaled(W["llama3_8b_2k"], batch=B, vocab=33000, n_nodes=12, depth=4, branch=4, temperatures=temps, prefix=(8, 8))
    _assert_parity(synth.generate(w, 1, with_attention=False), allow_near=1)


def test_device_detected_errors_are_reported_not_fatal():
    w = synth.scaled(W["tiny_greedy"], vocab=1000, n_nodes=8, prefix=(8, 8))
    inp = synth.generate(w, 0, with_attention=False)
    ctx = helpers.make_ctx(inp)
    bad = inp.parent.copy()
    bad[0, 3] = 5                                   # parent after child
    d = helpers.upload_accept(inp)
    ctx.tree_accept(d["target_logits"], None, d["draft_tokens"], helpers.dev(bad), d["temperature"], None)
    assert ctx.status() == -8
    assert ctx.status() == 0                        # cleared by the read
    toks = inp.draft_tokens.copy()
    toks[0, 2] = 1000                               # token id == V
    ctx.tree_accept(d["target_logits"], None, helpers.dev(toks), d["parent"], d["temperature"], None)
    assert ctx.status() == -5
    # the context still works
    path, n_acc, bonus = _run(inp, ctx)
    assert helpers.compare_accept(inp, path, n_acc, bonus)[0] == 0


@pytest.mark.parametrize("vocab", [4096, 128256, 151936])
@pytest.mark.parametrize("rest", ["zero", "denormal", "minus_zero"])
@pytest.mark.parametrize("temp", [1.0, 0.1])
def test_draft_rows_with_tiny_children(vocab, rest, temp):
    """A peaked draft row whose children run from 1 down to the smallest denormal, the other tokens exactly zero, negative zero or
    denormal: once the large ones are rejected the draft mass left is tiny and the coefficient of the draft row huge, so that even a
    draft probability of 1e-39 decides weights.  Rows that fit into a thread's registers (4096, 128256) and that do not (151936)."""
    B, N = 8, 9
    rng = np.random.default_rng(vocab)
    w = synth.scaled(W["llama3_8b_2k"], batch=B, vocab=vocab, n_nodes=N, tree="star", temperatures=(temp,) * B, prefix=(8, 8))
    inp = synth.generate(w, 0, with_attention=False)
    assert inp.parent.shape == (B, N)
    sizes = np.array([1.0, 1e-9, 3e-20, 1e-30, 2e-38, 9e-39, 5e-42, 1.5e-45], np.float32)
    for b in range(B):
        tok = rng.permutation(vocab)
        inp.target_logits[b] = -60.0 * temp
        heavy = tok[N:N + 40]
        inp.target_logits[b][:, heavy] = (rng.standard_normal(heavy.size) * temp).astype(np.float32)
        inp.draft_probs[b] = np.float32(-0.0) if rest == "minus_zero" else np.float32(0.0)
        if rest == "denormal":
            inp.draft_probs[b][:, heavy[::2]] = (rng.random(heavy[::2].size) * 1e-39).astype(np.float32)
        kids = tok[:N - 1]
        keep = N - 1 - b % 4                                     # how many of the tiny ones are listed; the rest repeat the first
        kids[keep:] = kids[0]
        inp.draft_probs[b][:, kids[:keep]] = sizes[:keep]
        inp.draft_tokens[b, 1:] = kids
        inp.uniforms[b] = rng.random(N + 1)
    _assert_parity(inp)
    r = oracle.tree_accept(inp.target_logits, inp.draft_probs, inp.draft_tokens, inp.parent, inp.temperature, inp.uniforms)
    assert int((r["n_accepted"] == 1).sum()) >= B - 2               # the children are rejected, the bonus token is drawn from what is left


def test_zero_draft_probabilities_keep_their_weight():
    """Two rejected children of 1 and 2e-38 leave two tokens of weight 1 and 0.497 that the draft gives nothing: neither loses any."""
    w = synth.scaled(W["llama3_8b_2k"], batch=1, vocab=4096, n_nodes=3, tree="star", temperatures=(1.0,), prefix=(8, 8))
    inp = synth.generate(w, 0, with_attention=False)
    inp.target_logits[...] = -60.0
    inp.target_logits[:, :, 100], inp.target_logits[:, :, 3000] = 0.0, -0.7
    inp.draft_probs[...] = 0.0
    inp.draft_probs[:, :, 200], inp.draft_probs[:, :, 300] = 1.0, 2e-38
    inp.draft_tokens[0] = [0, 200, 300]
    inp.uniforms[...] = [0.5, 0.5, 0.5, 0.8]
    path, n_acc, bonus = _run(inp)
    assert int(n_acc[0]) == 1 and int(bonus[0]) == 3000


@pytest.mark.parametrize("temp", [1e-3, 1e-8, 1e-10, 1e-12, 1e-14, 1e-16, 1e-20, 1e-30])
def test_temperatures_close_to_zero(temp):
    """Three tokens share the maximum, so p = 1/3 each however low the temperature; every first child is tested at r q = p (1 +- 3e-4),
    outside the margin inside which the scan's sum is replaced by an exact one."""
    B, N, V = 8, 7, 3000
    rng = np.random.default_rng(3)
    w = synth.scaled(W["llama3_8b_2k"], batch=B, vocab=V, n_nodes=N, tree="star", temperatures=(temp,) * B, prefix=(8, 8))
    inp = synth.generate(w, 0, with_attention=False)
    for b in range(B):
        top = np.float32(20.3 if b % 2 else 7.77)
        inp.target_logits[b] = top - np.float32(1.0) - rng.random((N, V)).astype(np.float32)
        tok = rng.permutation(V)[:N]
        inp.target_logits[b][:, tok[:3]] = top
        inp.draft_probs[b] = np.float32(0.1 / V)
        inp.draft_probs[b][:, tok[:N - 1]] = np.array([0.4, 0.5, 0.45, 0.02, 0.02, 0.01], np.float32)
        inp.draft_tokens[b, 1:] = tok[:N - 1]
        side = 3e-4 if b % 4 < 2 else -3e-4
        inp.uniforms[b] = rng.random(N + 1)
        inp.uniforms[b, 1] = (1.0 / 3.0) * (1.0 + side) / 0.4
    _assert_parity(inp)


def _check_stats(rows, vocab, noalloc):
    """Maximum and index exact, sum 2e-6 relative (fp32 with ex2.approx), every row start alignment among the rows."""
    x = (np.random.default_rng(vocab).standard_normal((rows, vocab)) * 3).astype(np.float32)
    temp = torch.full(((rows + 9) // 10,), 0.8, device="cuda")
    if noalloc:
        got = (torch.empty(rows, device="cuda"), torch.empty(rows, dtype=torch.float64, device="cuda"),
               torch.empty(rows, dtype=torch.int32, device="cuda"))
        assert binding.accept_stats_noalloc(helpers.dev(x), temp, 10, got) == 0
        torch.cuda.synchronize()
    else:
        ctx = binding.Context(8, 2, vocab, 512, max_nodes=min(rows, 256), max_batch=(rows + 255) // 256)
        got = ctx.accept_stats(helpers.dev(x), temp, 10)
        ctx.check()
    om, os_, oa = oracle.row_stats(x, 0.8)
    assert np.array_equal(got[0].cpu().numpy(), om.astype(np.float32))
    assert np.array_equal(got[2].cpu().numpy(), oa)
    np.testing.assert_allclose(got[1].cpu().numpy(), os_, rtol=2e-6)


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("rows,vocab", [(64, 46), (64, 47), (60, 166), (26, 79), (120, 22), (1000, 30), (512, 6), (300, 101), (60, 167)])
def test_stats_pieces_that_begin_past_the_end_of_a_row(rows, vocab, noalloc):
    """Sizes at which a row's last piece is one unit that only a row starting off a 16-byte boundary reaches into."""
    _check_stats(rows, vocab, noalloc)


@pytest.mark.parametrize("vocab", [22, 46, 47])
def test_sampling_walk_on_rows_of_many_short_pieces(vocab):
    for variant in range(4):
        w = synth.scaled(W["llama3_8b_2k"], batch=8, vocab=vocab, n_nodes=15, depth=4, branch=3, temperatures=(1.0, 0.7) * 4, prefix=(8, 8))
        _assert_parity(synth.generate(w, variant, with_attention=False), allow_near=1)


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("rows,vocab", [(8, 1), (9, 1), (64, 1), (8, 2), (33, 2), (8, 3), (50, 3), (1000, 1), (1024, 3)])
def test_stats_rows_shorter_than_one_load(rows, vocab, noalloc):
    """A row's first and last unit may be the same one: its tokens count once."""
    _check_stats(rows, vocab, noalloc)
